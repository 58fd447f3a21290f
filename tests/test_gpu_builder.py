"""GPU parity of carnator_build_connectivity against the builder oracle, through the C ABI.

Bar: the block mask is bit-exact except for blocks whose fp32 pooled score (the oracle's) lies
within 1e-4 of the row's selection threshold; always-kept blocks must match; in top-k mode the
per-row count must match.  Pooled scores themselves are compared to 2e-5 absolute.
"""
import dataclasses
import os

import numpy as np
import pytest
import torch

from oracle import carnator_oracle as orc
from paper_2609_32420_b200 import carnator as cn
from paper_2609_32420_b200 import workloads as wl
from tests.gpu_util import to_dev
from tests.helpers import check_mask

pytestmark = pytest.mark.gpu


def _oracle(w, Qb, Kb, heads=None):
    bp = w.build
    return orc.build_connectivity(Qb, Kb, w.N, w.n_text, w.T, w.Hg, w.Wg, w.block, w.block, w.scale,
                                  bp.mode, bp.keep_ratio, bp.mass, bp.window_frames, bp.text_dense,
                                  bp.count_includes_forced, heads=heads)


def _gpu(w, Qb, Kb):
    Q, K = to_dev(Qb), to_dev(Kb)
    shape = cn.shape_of(w, Q, K)
    scores = torch.empty((w.B, w.H, w.nqb, w.nkb), dtype=torch.float32, device="cuda")
    mask, ws = cn.build_connectivity(Q, K, shape, cn.params_of(w.build), pooled_scores=scores)
    assert cn.query_status(ws) == cn.OK
    return mask.cpu().numpy(), scores.cpu().numpy()


def _compare(w, Qb, Kb, heads=None, what=""):
    mask_g, scores_g = _gpu(w, Qb, Kb)
    mask_r, scores_r, theta, F = _oracle(w, Qb, Kb, heads)
    if heads is not None:
        sel = np.zeros((w.B, w.H), dtype=bool)
        for (b, h) in heads:
            sel[b, h] = True
        mask_g = np.where(sel[:, :, None, None], mask_g, 0)
        scores_g = np.where(sel[:, :, None, None], scores_g, 0)
    assert np.abs(scores_g - scores_r).max() <= 2e-5, f"{what}: pooled scores differ by {np.abs(scores_g - scores_r).max()}"
    return check_mask(mask_g, mask_r, scores_r, theta, F, topk_mode=(w.build.mode == wl.MODE_TOPK), what=what)


PATHS = [cn.BUILDER_THREE_KERNELS, cn.BUILDER_FUSED]
PATH_IDS = ["three_kernels", "fused"]


@pytest.fixture
def builder_path(request):
    """Small layers would take the three kernels by size; the parity cases below run on both paths."""
    cn.debug_set_builder_path(request.param)
    yield request.param
    cn.debug_set_builder_path(cn.BUILDER_AUTO)


@pytest.mark.parametrize("builder_path", PATHS, ids=PATH_IDS, indirect=True)
def test_tiny_topk(builder_path):
    w = wl.get("tiny")
    Qb, Kb, _ = wl.gen_qkv(w)
    _compare(w, Qb, Kb, what="tiny")


@pytest.mark.parametrize("builder_path", PATHS, ids=PATH_IDS, indirect=True)
@pytest.mark.parametrize("name,kw", [
    ("wan1p3b_480p", dict(H=2, T=3)),
    ("cogvideox5b", dict(H=3, T=2)),
    ("hunyuan_720p", dict(H=2, T=1)),
    ("hunyuan_720p", dict(H=2, T=28)),         # nkb = 790: four score tiles per row, 32 keys per lane
])
def test_midsize_window_text_rules(name, kw, builder_path):
    w = wl.shrunk(wl.get(name), **kw)
    Qb, Kb, _ = wl.gen_qkv(w, "history")
    _compare(w, Qb, Kb, what=name)


@pytest.mark.parametrize("mass", [0.5, 0.9, 0.95])
@pytest.mark.parametrize("name,kw", [("tiny", {}), ("wan1p3b_480p", dict(H=2, T=4))])
def test_cumulative_mass_mode(name, kw, mass):
    w = wl.get(name)
    if kw:
        w = wl.shrunk(w, **kw)
    w = w.replace(build=dataclasses.replace(w.build, mode=wl.MODE_CUMMASS, mass=mass))
    Qb, Kb, _ = wl.gen_qkv(w, "history")
    _compare(w, Qb, Kb, what=f"{name} cummass {mass}")


@pytest.mark.parametrize("builder_path", PATHS, ids=PATH_IDS, indirect=True)
def test_ties_are_broken_by_lower_block_index(builder_path):
    """Identical key blocks give identical pooled scores: the lower index must win, exactly as the oracle does."""
    w = wl.shrunk(wl.get("wan1p3b_480p"), H=1, T=2).replace(
        build=wl.BuildParams(keep_ratio=0.3, window_frames=-1))
    Qb, Kb, _ = wl.gen_qkv(w, "history")
    blk = Kb[:, :, :128].copy()
    for J in range(w.N // 128):
        Kb[:, :, J * 128:(J + 1) * 128] = blk
    mask_g, _ = _gpu(w, Qb, Kb)
    mask_r, _, _, _ = _oracle(w, Qb, Kb)
    full = w.N // 128
    np.testing.assert_array_equal(mask_g[..., :full], mask_r[..., :full])


@pytest.mark.parametrize("builder_path", PATHS, ids=PATH_IDS, indirect=True)
def test_keep_ratio_one_is_all_ones(builder_path):
    w = wl.shrunk(wl.get("hunyuan_720p"), H=1, T=1).replace()
    w = w.replace(build=dataclasses.replace(w.build, keep_ratio=1.0))
    Qb, Kb, _ = wl.gen_qkv(w, "history")
    mask_g, _ = _gpu(w, Qb, Kb)
    assert (mask_g == 1).all()


@pytest.mark.parametrize("name,kw", [("tiny", {}), ("wan1p3b_480p", dict(H=3, T=5)), ("cogvideox5b", dict(H=5, T=3)),
                                     ("hunyuan_720p", dict(H=2, T=2)), ("wan14b_720p", dict(H=3)), ("hunyuan_720p", dict(H=2))])
def test_fused_kernel_and_three_kernel_path_agree(name, kw):
    """Large top-k layers run as one persistent kernel that pools and scores on the tensor cores (block means as three
    bf16 terms, six products per score, fp32 accumulate); the three separate kernels use CUDA-core fp32 sums and FFMA
    chains.  Both carry rounding errors of a few 1e-6 on scores of magnitude 3 to 4 (each is checked against the fp64
    oracle to 2e-5 elsewhere); masks may differ only where a score sits that close to the row's threshold."""
    w = wl.shrunk(wl.get(name), **kw) if kw else wl.get(name)
    nthreads = min(16, os.cpu_count() or 1)
    Q = to_dev(wl.gen_tensor(w, "Q", "history", threads=nthreads))
    K = to_dev(wl.gen_tensor(w, "K", "history", threads=nthreads))
    shape = cn.shape_of(w, Q, K)
    out = []
    try:
        for path in (cn.BUILDER_FUSED, cn.BUILDER_THREE_KERNELS):
            cn.debug_set_builder_path(path)
            scores = torch.full((w.B, w.H, w.nqb, w.nkb), float("nan"), dtype=torch.float32, device="cuda")
            mask, ws = cn.build_connectivity(Q, K, shape, cn.params_of(w.build), pooled_scores=scores)
            assert cn.query_status(ws) == cn.OK, cn.last_cuda_error()
            mask2, ws = cn.build_connectivity(Q, K, shape, cn.params_of(w.build), ws=ws)       # without the score output
            assert cn.query_status(ws) == cn.OK
            assert torch.equal(mask, mask2)
            out.append((mask, scores))
    finally:
        cn.debug_set_builder_path(cn.BUILDER_AUTO)
    (m0, s0), (m1, s1) = out
    assert float((s0 - s1).abs().max()) <= 1e-5
    assert bool((m0.sum(-1) == m1.sum(-1)).all())                       # top-k: same number of blocks per row
    assert int((m0 != m1).sum()) <= 1e-5 * m0.numel() + 2


# the HunyuanVideo-shaped layer also at the ends of its density sweep
FULL = [("wan1p3b_480p", None), ("cogvideox5b", None), ("wan14b_720p", None), ("hunyuan_720p", None),
        ("hunyuan_720p", 0.05), ("hunyuan_720p", 0.50)]


@pytest.mark.parametrize("name,keep", FULL, ids=[f[0] + ("" if f[1] is None else f"_{f[1]}") for f in FULL])
def test_full_size_masks_on_sampled_heads(name, keep):
    """Full-size launch; the oracle checks two heads in full (every row, every block)."""
    w = wl.get(name)
    if keep is not None:
        w = w.replace(build=dataclasses.replace(w.build, keep_ratio=keep))
    heads = [(0, 1), (0, w.H - 2)]
    nthreads = min(16, os.cpu_count() or 1)
    Qb = wl.gen_tensor(w, "Q", "history", threads=nthreads)
    Kb = wl.gen_tensor(w, "K", "history", threads=nthreads)
    n_excused = _compare(w, Qb, Kb, heads=heads, what=f"{name} keep={w.build.keep_ratio}")
    assert n_excused <= 8


# One kernel scores and selects for up to 1024 key blocks (a warp holds 5, 8, 20 or 32 keys a lane), two take more: the edges of those
# ranges, ragged last blocks and query tiles, both CTA sizes (8 and 16 rows), unequal block sizes.
@pytest.mark.parametrize("mode", [wl.MODE_TOPK, wl.MODE_CUMMASS], ids=["topk", "mass"])
@pytest.mark.parametrize("B,H,N,n_text,D,bq,bk,window", [
    (1, 1, 50, 0, 128, 64, 64, -1), (1, 1, 64 * 31 + 1, 7, 64, 128, 64, -1), (2, 3, 64 * 33, 0, 128, 64, 64, 0),
    (1, 48, 64 * 129 - 1, 100, 64, 64, 64, 1), (1, 2, 64 * 256, 0, 64, 128, 64, -1), (1, 2, 64 * 160, 0, 64, 128, 64, -1), (1, 1, 64 * 161, 9, 64, 128, 64, 0),
    (1, 1, 64 * 640 - 3, 0, 128, 128, 64, 1), (1, 1, 64 * 257, 0, 128, 128, 64, 1),
    (1, 1, 64 * 1024, 0, 64, 128, 64, -1), (1, 1, 64 * 1024 + 1, 0, 64, 128, 64, 0), (1, 2, 128 * 40 + 5, 0, 128, 128, 128, 2)])
def test_score_and_selection_at_the_edges_of_their_ranges(B, H, N, n_text, D, bq, bk, window, mode):
    rng = np.random.default_rng(N + D + mode)
    T = 4 if (N - n_text) % 4 == 0 else 1
    hw = (N - n_text) // T
    Qb, Kb = (rng.standard_normal((B, H, N, D)).astype(np.float32) for _ in range(2))
    Qb, Kb = ((x.view(np.uint32) >> 16).astype(np.uint16) for x in (Qb, Kb))
    if N >= 4 * bk:
        Kb[:, :, 2 * bk:3 * bk] = Kb[:, :, :bk]                 # equal scores: the lower index comes first
    Q, K = to_dev(Qb), to_dev(Kb)
    shape = cn.make_shape(B, H, N, D, n_text, T, 1, hw, bq, bk, Q, K)
    p = cn.BuildParams()
    p.mode, p.keep_ratio, p.mass, p.window_frames, p.text_dense, p.count_includes_forced = mode, 0.3, 0.8, window, 1, 0
    nqb, nkb = -(-N // bq), -(-N // bk)
    scores = torch.empty((B, H, nqb, nkb), dtype=torch.float32, device="cuda")
    cn.debug_set_builder_path(cn.BUILDER_THREE_KERNELS)
    try:
        ws = torch.full((cn.build_workspace_bytes(shape, p),), 0xFF, dtype=torch.uint8, device="cuda")   # a workspace that was something else
        mask, ws = cn.build_connectivity(Q, K, shape, p, pooled_scores=scores, ws=ws)
        assert cn.query_status(ws) == cn.OK
        mask2, _ = cn.build_connectivity(Q, K, shape, p)
    finally:
        cn.debug_set_builder_path(cn.BUILDER_AUTO)
    assert torch.equal(mask, mask2)
    ref = orc.build_connectivity(Qb, Kb, N, n_text, T, 1, hw, bq, bk, 1.0 / np.sqrt(D), mode, 0.3, 0.8, window, 1, 0)
    s = scores.cpu().numpy()
    assert np.abs(s - ref[1]).max() <= 2e-5
    check_mask(mask.cpu().numpy(), ref[0], ref[1], ref[2], ref[3], topk_mode=(mode == wl.MODE_TOPK), what=f"N={N}")


def check_prefix(p, mask, forced, target, what):
    """The rule on given masses p (64 bits, sum 1): always-kept blocks, and of the others the shortest prefix in descending order
    (ties: lower index first) with which the kept mass reaches the target.  Sums of up to 1024 terms in 64 bits, in whatever
    order, are good to 1024 * 2^-53, 1.2e-13."""
    eps = 1.2e-13
    free = np.flatnonzero(~forced)
    ranked = free[np.lexsort((free, -p[free]))]
    n = int(mask[ranked].sum())
    assert mask[forced].all() and mask[ranked[:n]].all(), f"{what}: not a prefix"
    kept = p[forced].sum() + p[ranked[:n]].sum()
    assert kept >= target - eps or n == len(ranked), f"{what}: {kept} of {target}"
    assert n == 0 or kept - p[ranked[n - 1]] < target + eps, f"{what}: longer than needed"
    return n


@pytest.mark.parametrize("mass", [1.0 - 2.0 ** -24, 1.0, 0.999], ids=["one_minus_2^-24", "one", "0.999"])
@pytest.mark.parametrize("H,nb,D,spread", [(3, 61, 128, 9.0), (2, 200, 64, 9.0), (1, 500, 64, 12.0), (1, 1000, 128, 9.0), (2, 130, 64, 0.0), (1, 520, 64, -1.0),
                                             (2, 1000, 128, -1.0)])
def test_cumulative_mass_where_the_tail_decides(H, nb, D, spread, mass):
    """Rows whose last admitted blocks weigh less than 2^-31, far below the units of 2^-20 to 2^-24 that the search counts in (spread
    -1: one block with nearly all of the mass, hundreds of 2^-32 each), targets that all blocks together may miss, and blocks with equal
    scores at the threshold (every third is a copy of its neighbour; with a spread of 0 all are equal)."""
    block, rng = 64, np.random.default_rng(nb)
    u, v = (rng.standard_normal((1, H, nb, D)).astype(np.float32) for _ in range(2))
    v[:, :, 2::3] = v[:, :, 1::3][:, :, :v[:, :, 2::3].shape[2]]
    if spread < 0:
        u[:] = u[:, :, :1]
        v *= 0.3
        v[:, :, 0] = u[:, :, 0] * 22.5 * np.sqrt(D) / (u[:, :, 0] ** 2).sum(-1, keepdims=True)
    else:
        u *= spread
    tokens = lambda x: torch.from_numpy(np.repeat(x, block, axis=2)).cuda().to(torch.bfloat16)
    Q, K = tokens(u), tokens(v)
    N = nb * block
    shape = cn.make_shape(1, H, N, D, 0, 1, 1, N, block, block, Q, K)
    p = cn.BuildParams()
    p.mode, p.mass, p.keep_ratio, p.window_frames, p.text_dense, p.count_includes_forced = cn.MODE_CUMMASS, mass, 0.5, -1, 0, 1
    scores = torch.empty((1, H, nb, nb), dtype=torch.float32, device="cuda")
    mask, ws = cn.build_connectivity(Q, K, shape, p, pooled_scores=scores)
    assert cn.query_status(ws) == cn.OK
    mask, scores = mask.cpu().numpy() != 0, scores.cpu().numpy().astype(np.float64)
    target, beyond = float(np.float32(mass)), 0
    for h in range(H):
        for I in range(nb):
            e = np.exp(scores[0, h, I] - scores[0, h, I].max())
            e /= e.sum()
            n = check_prefix(e, mask[0, h, I], np.zeros(nb, bool), target, f"head {h} row {I}")
            beyond += n > 0 and np.sort(e)[::-1][n - 1] < 2.0 ** -31
    assert beyond > 0 or spread == 0.0 or mass < 0.9999 or (mass < 1.0 and spread > 0)


@pytest.mark.parametrize("H,nb,D", [(48, 139, 64), (31, 266, 64), (16, 1000, 64)])
def test_a_high_mass_target_takes_no_longer(H, nb, D):
    """A target of 0.999 lies among blocks that weigh about as much as the search's units, so its first outcome is often a few keys
    off.  Putting that right must not cost a search of its own: with one, these layers took 22 to 31 % longer than at 0.5,
    without 2 to 4 %.  The same rows checked against the rule."""
    block, rng = 64, np.random.default_rng(nb)
    tokens = lambda x: torch.from_numpy(np.repeat(x.astype(np.float32), block, axis=2)).cuda().to(torch.bfloat16)
    Q, K = tokens(3 * rng.standard_normal((1, H, nb, D))), tokens(rng.standard_normal((1, H, nb, D)))
    shape = cn.make_shape(1, H, nb * block, D, 0, 1, 1, nb * block, block, block, Q, K)
    scores, took = torch.empty((1, H, nb, nb), dtype=torch.float32, device="cuda"), {}
    start, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    for mass in (0.5, 0.999) * 5:
        p = cn.BuildParams()
        p.mode, p.mass, p.keep_ratio, p.window_frames, p.text_dense, p.count_includes_forced = cn.MODE_CUMMASS, mass, 0.5, -1, 0, 1
        mask, ws = cn.build_connectivity(Q, K, shape, p, pooled_scores=scores)
        assert cn.query_status(ws) == cn.OK
        start.record()
        for _ in range(50):
            cn.build_connectivity(Q, K, shape, p, ws=ws)
        end.record()
        end.synchronize()
        took[mass] = min(took.get(mass, 1e9), start.elapsed_time(end))
    mask, scores = mask.cpu().numpy() != 0, scores.cpu().numpy().astype(np.float64)
    for h in range(0, H, 5):
        for I in range(nb):
            e = np.exp(scores[0, h, I] - scores[0, h, I].max())
            check_prefix(e / e.sum(), mask[0, h, I], np.zeros(nb, bool), float(np.float32(0.999)), f"head {h} row {I}")
    assert took[0.999] < 1.12 * took[0.5], took
