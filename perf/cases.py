"""The work that a user of this package has it do, as cases that can be timed.

A case is one call of the path (or, for a middle layer, the few calls that belong together) on a layer of a video diffusion
transformer: the shapes are those of the package's workload records (`paper_2609_32420_b200/workloads.py`), slices of them, and
generic grids between them.  Inputs follow the recipe of that module (standard normal tokens plus a rank-8 component per
frame), drawn on the GPU.  Masks are made here in plain torch from a second ("history") pair with the same structure, so that
an attention case gets the same mask whatever builder the library has.

    op      entry points                                                    who calls it
    attn    sparse_attn, or sparse_attn_compacted on lists made once        every self-attention layer of a cache hit
    region  build_regions, region_block_flags, sparse_attn_region,          a middle layer of a hit: attention for the active query
            fuse_latents                                                    blocks only, and the fused latent
    build   build_connectivity (top-k or cumulative mass)                   a cache write, once per layer and step
    exact   build_connectivity_exact                                        a cache write by true attention mass
    seed    seed_expansion                                                  the early probe of a request, once per layer used
"""
import math

import numpy as np
import torch

from paper_2609_32420_b200 import carnator as cn

# The fields a case may leave out.
DEFAULTS = dict(
    B=1,                 # 2: the conditional and the unconditional branch of guidance in one call
    n_text=0,            # text tokens in front (joint attention)
    block=128,
    layout="bhnd",       # "bnhd": token-major storage, as a fused QKV projection leaves it
    spare_rows=0,        # rows behind the N valid ones in a longer buffer
    mode="topk", ratio=0.25, mass=0.9, window=-1, text_dense=0, count_forced=1,
    recompute=0.0,       # share of the video-only query blocks that are recomputed densely
    lists="each",        # "kept": the mask was compacted once and its lists serve every call
    n_pos=0, n_neg=0,    # seed tokens
    channels=0, latent="f32",
    object_share=0.06,   # share of a frame that the evidence region covers
)


def _full(case):
    c = dict(DEFAULTS)
    c.update(case)
    c["N"] = c["n_text"] + c["T"] * c["Hg"] * c["Wg"]
    c["nb"] = -(-c["N"] // c["block"])
    return c


def listed():
    wan13b = dict(H=12, D=128, T=21, Hg=30, Wg=52, window=1, ratio=0.25)
    wan14b = dict(H=40, D=128, T=21, Hg=45, Wg=80, window=1, ratio=0.15)
    cog = dict(H=48, D=64, n_text=226, T=13, Hg=30, Wg=45, text_dense=1, count_forced=0, ratio=0.35)
    clip = dict(H=12, D=128, T=5, Hg=30, Wg=52, window=0, ratio=0.35)
    return [
        # the smallest layer of the workload records: 64-token blocks, a few hundred tiles; latency and launches
        dict(name="attn_tiny_b64", op="attn", H=2, D=64, T=4, Hg=16, Wg=16, block=64, ratio=0.30, recompute=3 / 16),
        # a clip of five latent frames, ragged last block, both guidance branches, Q/K/V as the projection leaves them
        dict(name="attn_clip", op="attn", B=2, layout="bnhd", recompute=0.15, **clip),
        # an ordinary layer: Wan-1.3B-shaped, 480p, in a buffer that is longer than the sequence
        dict(name="attn_wan13b", op="attn", recompute=0.15, spare_rows=8, **wan13b),
        # the same layer under a mask of the finer block size, its lists kept from call to call
        dict(name="attn_wan13b_b64", op="attn", recompute=0.15, block=64, lists="kept", **wan13b),
        # joint attention with text in front, head dimension 64: CogVideoX-5B-shaped
        dict(name="attn_cogvideox", op="attn", recompute=0.20, **cog),
        # the largest layer: Wan-14B-shaped, 720p
        dict(name="attn_wan14b", op="attn", recompute=0.10, **wan14b),
        # a middle layer of a hit: regions, region-restricted attention, latent fusion
        dict(name="middle_wan13b", op="region", channels=64, **wan13b),
        # cache writes: a clip, the largest layer, and the cumulative-mass rule on a joint-attention layer
        dict(name="build_clip", op="build", **clip),
        dict(name="build_wan14b", op="build", **wan14b),
        dict(name="build_cogvideox_mass", op="build", **dict(cog, mode="mass")),
        # cache write by true attention mass
        dict(name="exact_wan13b", op="exact", **dict(wan13b, mode="mass")),
        # seed tokens of one noun against the background, propagated through a whole layer
        dict(name="seed_wan14b", op="seed", n_pos=192, n_neg=320, **wan14b),
    ]


# Most matrix work of a drawn case, by op and block size: that of the largest listed case of the kind.
_MOST = {("attn", 128): 2.75e13, ("attn", 64): 6.0e12, ("region", 128): 4.0e12, ("build", 128): 1.55e9, ("build", 64): 3.0e8,
         ("exact", 128): 3.3e12, ("seed", 128): 4.0e11}


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    while True:
        op = rng.choice(["attn", "attn", "attn", "region", "build", "build", "exact", "seed"])
        D = rng.choice([64, 128, 128])
        c = dict(op=op, H=_log(rng, 1, 48), D=D, T=_log(rng, 1, 33), Hg=_log(rng, 8, 48), Wg=_log(rng, 8, 84))
        if op == "attn":
            c["block"] = rng.choice([64, 128, 128, 128])
            c["lists"] = rng.choice(["each", "kept"])
            c["recompute"] = rng.choice([0.0, round(rng.uniform(0.05, 0.25), 3)])
            c["B"] = rng.choice([1, 1, 2])
        elif op == "build":
            c["block"] = rng.choice([64, 128, 128])
            c["B"] = rng.choice([1, 1, 2])
        if op == "region":
            c["Wg"] = max(8, c["Wg"] // 8 * 8)           # latents are fused in rows of 16 bytes
            c["channels"] = rng.choice([16, 48, 64])
            c["latent"] = rng.choice(["f32", "bf16"])
            c["object_share"] = round(rng.uniform(0.02, 0.3), 3)
        elif rng.random() < 0.4:
            c["n_text"] = _log(rng, 7, 512)
            c["text_dense"], c["count_forced"] = 1, 0
        else:
            c["window"] = rng.choice([-1, 0, 1, 2])
        if op == "exact" or (op == "build" and rng.random() < 0.4):
            c["mode"], c["mass"] = "mass", rng.choice([0.5, 0.8, 0.9, 0.95])
        else:
            c["ratio"] = round(rng.uniform(0.05, 0.6), 3)
        c["layout"] = rng.choice(["bhnd", "bhnd", "bnhd"])
        if op == "seed":
            c["n_pos"], c["n_neg"] = _log(rng, 3, 256), _log(rng, 3, 320)
        n = _full(c)
        if n["N"] < 96 or n["N"] > 120000 or n["N"] * n["B"] * c["H"] * c["D"] > 390e6:
            continue
        if op in ("build", "exact"):                     # most of the mask has to be decided by the scores
            forced = _forced(n)
            free = n["mass"] / 2 - forced.mean() if n["mode"] == "mass" else (_kept_per_row(n, forced) - forced.sum(1)).mean() / n["nb"]
            if free < 0.03 or n["nb"] < 4:
                continue
        w = work(c)
        size = w["bytes"] if op == "build" else w["flops"]
        if op != "build" and size < 1e8:                 # below the smallest listed layer
            continue
        if size <= _MOST[(op, c.get("block", 128))]:
            return c


# ---- inputs ------------------------------------------------------------------------------------------------------------
def _tokens(c, gen, comp):
    """bf16 [B,H,N + spare,D] standard normal tokens plus the frame component on the video tokens; spare rows are zero."""
    B, H, N, D = c["B"], c["H"], c["N"], c["D"]
    rows = N + c["spare_rows"]
    if c["layout"] == "bnhd":
        x = torch.randn((B, rows, H, D), dtype=torch.bfloat16, device="cuda", generator=gen).permute(0, 2, 1, 3)
    else:
        x = torch.randn((B, H, rows, D), dtype=torch.bfloat16, device="cuda", generator=gen)
    hw = c["Hg"] * c["Wg"]
    for f in range(c["T"]):
        t0 = c["n_text"] + f * hw
        x[:, :, t0:t0 + hw] += comp[:, :, f:f + 1]
    if c["spare_rows"]:
        x[:, :, N:] = 0
    return x


def _component(c, gen):
    """[B,H,T,D]: rank 8, weight 0.5, as in the package's workload recipe."""
    a = torch.randn((c["B"], c["H"], c["T"], 8), device="cuda", generator=gen)
    w = torch.randn((c["B"], c["H"], 8, c["D"]), device="cuda", generator=gen)
    return ((0.5 / math.sqrt(8.0)) * (a @ w)).to(torch.bfloat16)


def _count(ratio, n):
    return np.where(n > 0, np.clip(np.ceil(float(np.float32(ratio)) * n - 1e-6), 1, np.maximum(n, 1)), 0).astype(np.int64)


def _forced(c):
    """bool [nb,nb]: block pairs that are always kept."""
    nb, bl, nt, hw = c["nb"], c["block"], c["n_text"], c["Hg"] * c["Wg"]
    lo, hi = np.arange(nb) * bl, np.minimum(c["N"], (np.arange(nb) + 1) * bl) - 1
    out = np.zeros((nb, nb), bool)
    if c["text_dense"] and nt > 0:
        text = lo < nt
        out |= text[:, None] | text[None, :]
    if c["window"] >= 0:
        video = hi >= nt
        f0, f1 = (np.maximum(lo, nt) - nt) // hw, (hi - nt) // hw
        near = (f0[None, :] <= (f1 + c["window"])[:, None]) & (f1[None, :] >= (f0 - c["window"])[:, None])
        out |= near & video[:, None] & video[None, :]
    return out


def _kept_per_row(c, forced):
    """Key blocks that the top-k rule keeps in each row."""
    nf = forced.sum(1)
    if c["count_forced"]:
        return np.maximum(nf, _count(c["ratio"], np.full_like(nf, c["nb"])))
    return nf + _count(c["ratio"], c["nb"] - nf)


def _block_means(c, x):
    nb, bl, N = c["nb"], c["block"], c["N"]
    out = torch.zeros((c["B"], c["H"], nb, c["D"]), device="cuda")
    whole = N // bl
    if whole:
        out[:, :, :whole] = x[:, :, :whole * bl].unflatten(2, (whole, bl)).mean(3, dtype=torch.float32)
    if whole < nb:
        out[:, :, whole] = x[:, :, whole * bl:N].mean(2, dtype=torch.float32)
    return out


def _mask(c, gen, comp):
    """uint8 [B,H,nb,nb]: the top-k rule on the block means of a history pair."""
    q, k = (_block_means(c, _tokens(c, gen, comp)).double() for _ in range(2))
    forced = _forced(c)
    keep = torch.from_numpy(_kept_per_row(c, forced)).cuda()
    s = (q @ k.transpose(2, 3)).masked_fill_(torch.from_numpy(forced).cuda(), math.inf)
    order = s.argsort(dim=3, descending=True, stable=True)
    rank = torch.empty_like(order).scatter_(3, order, torch.arange(c["nb"], device="cuda").expand_as(order).contiguous())
    return (rank < keep[None, None, :, None]).to(torch.uint8).contiguous()


def _recompute(c, gen):
    """uint8 [B,nb]: a random share of the blocks that hold no text."""
    first = -(-c["n_text"] // c["block"])
    n = int(round(c["recompute"] * (c["nb"] - first)))
    out = torch.zeros((c["B"], c["nb"]), dtype=torch.uint8, device="cuda")
    for b in range(c["B"]):
        out[b, first + torch.randperm(c["nb"] - first, device="cuda", generator=gen)[:n]] = 1
    return out


def _evidence(c, gen):
    """uint8 [T,Hg,Wg]: an ellipse that drifts through the frames."""
    T, Hg, Wg = c["T"], c["Hg"], c["Wg"]
    at = torch.rand(4, device="cuda", generator=gen) * 0.5 + 0.25
    t = torch.linspace(0, 1, T, device="cuda")[:, None, None]
    y = (torch.arange(Hg, device="cuda")[None, :, None] + 0.5) / Hg - (at[0] + (at[1] - at[0]) * t)
    x = (torch.arange(Wg, device="cuda")[None, None, :] + 0.5) / Wg - (at[2] + (at[3] - at[2]) * t)
    return ((x * x + y * y) * math.pi < c["object_share"]).to(torch.uint8).contiguous()


def _params(c):
    p = cn.BuildParams()
    p.mode = cn.MODE_CUMMASS if c["mode"] == "mass" else cn.MODE_TOPK
    p.keep_ratio, p.mass = c["ratio"], c["mass"]
    p.window_frames, p.text_dense, p.count_includes_forced = c["window"], c["text_dense"], c["count_forced"]
    return p


def _shape(c, *tensors):
    return cn.make_shape(c["B"], c["H"], c["N"], c["D"], c["n_text"], c["T"], c["Hg"], c["Wg"], c["block"], c["block"], *tensors)


def _dense_lse(c, Q, K):
    """What a dense run of the attention call leaves: fp32 [B,H,N]."""
    ones = torch.ones((c["B"], c["H"], c["nb"], c["nb"]), dtype=torch.uint8, device="cuda")
    return cn.sparse_attn(Q, K, K, ones, None, _shape(c, Q, K, K))[1]


def prepare(case, seed):
    c = _full(case)
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    comp = _component(c, gen)
    Q, K = _tokens(c, gen, comp), _tokens(c, gen, comp)
    s = dict(op=c["op"], Q=Q, K=K)
    if c["op"] in ("attn", "region"):
        s["V"] = V = _tokens(c, gen, _component(c, gen))
        s["mask"] = _mask(c, gen, comp)
        s["shape"] = _shape(c, Q, K, V)
        s["ws"] = torch.empty(cn.attn_workspace_bytes(s["shape"]), dtype=torch.uint8, device="cuda")
    if c["op"] == "attn":
        s["recompute"] = _recompute(c, gen) if c["recompute"] else None
        s["kept"] = c["lists"] == "kept"
        if s["kept"]:
            cn.compact_mask(s["mask"], s["recompute"], s["shape"], ws=s["ws"])
    elif c["op"] == "region":
        s["block"], s["evidence"] = c["block"], _evidence(c, gen)
        # what an earlier request left for this layer and step: outputs of the inactive blocks, and the latent
        s["O"] = torch.randn((c["B"], c["H"], c["N"], c["D"]), dtype=torch.bfloat16, device="cuda", generator=gen)
        s["LSE"] = torch.randn((c["B"], c["H"], c["N"]), device="cuda", generator=gen)
        dtype = torch.float32 if c["latent"] == "f32" else torch.bfloat16
        grid = (c["channels"], c["T"], c["Hg"], c["Wg"])
        s["z_target"], s["z_hist"] = (torch.randn(grid, device="cuda", generator=gen).to(dtype) for _ in range(2))
    else:
        s["shape"], s["params"] = _shape(c, Q, K), _params(c)
        if c["op"] == "build":
            s["ws"] = torch.empty(cn.build_workspace_bytes(s["shape"], s["params"]), dtype=torch.uint8, device="cuda")
        elif c["op"] == "exact":
            s["LSE"] = _dense_lse(c, Q, K)
            s["ws"] = torch.empty(cn.exact_workspace_bytes(s["shape"]), dtype=torch.uint8, device="cuda")
        else:
            s["LSE"] = _dense_lse(c, Q, K)
            s["n_pos"], s["n_neg"] = c["n_pos"], c["n_neg"]
            n = min(c["n_pos"] + c["n_neg"], c["N"])
            s["n_pos"] = min(s["n_pos"], n)
            s["n_neg"] = n - s["n_pos"]
            s["seeds"] = torch.randperm(c["N"], device="cuda", generator=gen)[:n].to(torch.int32)
            s["ws"] = torch.empty(cn.seed_workspace_bytes(s["shape"]), dtype=torch.uint8, device="cuda")
    return s


def run(s):
    op = s["op"]
    if op == "attn":
        if s["kept"]:
            return cn.sparse_attn_compacted(s["Q"], s["K"], s["V"], s["shape"], s["ws"])
        return cn.sparse_attn(s["Q"], s["K"], s["V"], s["mask"], s["recompute"], s["shape"], ws=s["ws"])[:2]
    if op == "region":
        active, context, W = cn.build_regions(s["evidence"], s["shape"])
        qf = cn.region_block_flags(active, s["shape"], s["block"])
        kf = cn.region_block_flags(context, s["shape"], s["block"])
        cn.sparse_attn_region(s["Q"], s["K"], s["V"], s["mask"], qf, kf, s["shape"], s["O"], s["LSE"], ws=s["ws"])
        z = cn.fuse_latents(s["z_target"], s["z_hist"], W)
        return active, context, W, s["O"], s["LSE"], z
    if op == "build":
        return cn.build_connectivity(s["Q"], s["K"], s["shape"], s["params"], ws=s["ws"])[0]
    if op == "exact":
        return cn.build_connectivity_exact(s["Q"], s["K"], s["LSE"], s["shape"], s["params"], ws=s["ws"])[0]
    return cn.seed_expansion(s["Q"], s["K"], s["LSE"], s["seeds"], s["n_pos"], s["n_neg"], s["shape"], ws=s["ws"])


# ---- what a pass cannot do without ---------------------------------------------------------------------------------------
def work(case):
    """Listed tiles count in full blocks' keys and queries (ragged ends by their tokens); each input read once, each output
    written once."""
    c = _full(case)
    B, H, N, D, nb = c["B"], c["H"], c["N"], c["D"], c["nb"]
    tensor = 2.0 * B * H * N * D
    pairs = B * H * nb * nb
    if c["op"] == "attn":
        kept = _kept_per_row(c, _forced(c)).astype(float)
        first = -(-c["n_text"] // c["block"])
        n = int(round(c["recompute"] * (nb - first)))
        kept[first:] += (nb - kept[first:]) * (n / max(1, nb - first))
        return {"bytes": 4 * tensor + 4.0 * B * H * N + pairs, "flops": 4.0 * D * B * H * c["block"] * N * kept.mean()}
    if c["op"] == "region":
        # the object and the rings around it, taken as a square of the same share
        side_q, side_k = (min(1.0, (math.sqrt(c["object_share"] * c["Hg"] * c["Wg"]) + 2 * r) / math.sqrt(c["Hg"] * c["Wg"])) for r in (2, 5))
        rows, keys = min(1.0, side_q * 1.1), min(1.0, side_k * 1.1)      # blocks are runs along the rows of a frame
        kept = _kept_per_row(c, _forced(c)).mean()
        tokens, e = c["T"] * c["Hg"] * c["Wg"], 4 if c["latent"] == "f32" else 2
        return {"bytes": tensor * 2 * (rows + keys) + rows * keys * pairs + tokens * (3.0 + 4) + 3.0 * e * c["channels"] * tokens,
                "flops": 4.0 * D * B * H * c["block"] * N * rows * keys * kept}
    if c["op"] == "build":
        return {"bytes": 2 * tensor + pairs, "flops": 2.0 * tensor + 2.0 * D * pairs}
    if c["op"] == "exact":
        return {"bytes": 2 * tensor + 4.0 * B * H * N + pairs, "flops": 2.0 * D * B * H * float(N) * N}
    n = min(c["n_pos"] + c["n_neg"], N)
    return {"bytes": tensor + 2.0 * B * H * n * D + 4.0 * B * H * N + 4.0 * B * N, "flops": 2.0 * D * B * H * float(N) * n}


def tolerance(case):
    """About four times what was measured: the two attention executors against each other (O in bf16: 9.6e-4, largest 7.8e-3), the
    seed contrasts against the same in 64 bits (8.5e-7, 6.5e-6).  Masks came out alike by different builder paths and against
    the cumulative-mass rule in 64 bits; the share that may differ is for scores that tie to the last bits of a 32-bit sum."""
    op = case["op"]
    if op in ("attn", "region"):
        return {"rel": 4e-3, "max": 3e-2}
    if op in ("build", "exact"):
        return {"rel": 0.0, "differ": 1e-4}
    return {"rel": 1e-5, "max": 1e-4}
