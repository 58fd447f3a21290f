"""The library in a process with more than one CUDA context, and from several threads at once."""
import os
import subprocess
import sys

import pytest

from tests.conftest import ROOT

pytestmark = pytest.mark.gpu

# A mask from the builder and an attention call over it in the primary context, in a second context on the same device, and in
# the primary context again, through the C ABI and the driver alone; the three outputs have to be the same bytes.
TWO_CONTEXTS = r"""
import ctypes, sys
import numpy as np
from paper_2609_32420_b200 import carnator as cn

cu = ctypes.CDLL("libcuda.so.1")
def ok(r, what):
    if r != 0:
        sys.exit(f"{what}: CUDA driver error {r}")
ok(cu.cuInit(0), "cuInit")
dev, first, second = ctypes.c_int(), ctypes.c_void_p(), ctypes.c_void_p()
ok(cu.cuDeviceGet(ctypes.byref(dev), 0), "cuDeviceGet")
ok(cu.cuDevicePrimaryCtxRetain(ctypes.byref(first), dev), "cuDevicePrimaryCtxRetain")
lib, B, H, N = cn.lib(), 1, 2, 700

def layer(D, block):
    rng, held = np.random.default_rng(D + block), []
    def buf(host):
        p = ctypes.c_uint64()
        host = np.ascontiguousarray(host)
        ok(cu.cuMemAlloc_v2(ctypes.byref(p), ctypes.c_size_t(host.nbytes + 256)), "cuMemAlloc")
        ok(cu.cuMemcpyHtoD_v2(p, host.ctypes.data_as(ctypes.c_void_p), ctypes.c_size_t(host.nbytes)), "cuMemcpyHtoD")
        held.append(p)
        return ctypes.c_void_p(p.value)
    def tokens():
        x = rng.standard_normal((B, H, N, D)).astype(np.float32)
        return buf((x.view(np.uint32) >> 16).astype(np.uint16))
    Q, K, V = tokens(), tokens(), tokens()
    s = cn.make_shape(B, H, N, D, 0, 1, 1, N, block, block)
    p = cn.BuildParams()
    p.mode, p.mass, p.keep_ratio, p.window_frames, p.count_includes_forced = cn.MODE_CUMMASS, 0.8, 0.5, -1, 1
    nb = s.nqb
    mask, O, L = buf(np.zeros(B * H * nb * nb, np.uint8)), buf(np.zeros(B * H * N * D, np.uint16)), buf(np.zeros(B * H * N, np.float32))
    wb, wa = cn.build_workspace_bytes(s, p), cn.attn_workspace_bytes(s)
    ws_b, ws_a = buf(np.zeros(wb, np.uint8)), buf(np.zeros(wa, np.uint8))
    st = lib.carnator_build_connectivity(Q, K, ctypes.byref(s), ctypes.byref(p), mask, None, ws_b, wb, None)
    if st == 0:
        st = lib.carnator_sparse_attn(Q, K, V, mask, None, ctypes.byref(s), O, L, ws_a, wa, None)
    if st != 0:
        sys.exit(f"D {D}, blocks of {block}: status {st}, {cn.last_cuda_error()}")
    ok(cu.cuCtxSynchronize(), "cuCtxSynchronize")
    out = np.empty(B * H * N * D, np.uint16)
    ok(cu.cuMemcpyDtoH_v2(out.ctypes.data_as(ctypes.c_void_p), ctypes.c_uint64(O.value), ctypes.c_size_t(out.nbytes)), "cuMemcpyDtoH")
    for q in held:
        ok(cu.cuMemFree_v2(q), "cuMemFree")
    return out

def layers():
    return [layer(D, b).tobytes() for D in (64, 128) for b in (64, 128)]

ok(cu.cuCtxSetCurrent(first), "cuCtxSetCurrent")
a = layers()
ok(cu.cuCtxCreate_v2(ctypes.byref(second), 0, dev), "cuCtxCreate")
b = layers()
ok(cu.cuCtxSetCurrent(first), "cuCtxSetCurrent")
assert layers() == a and b == a and len(set(a)) == 4
print("same outputs")
"""


def test_a_second_context_on_the_device():
    """What a kernel was allowed in one context (dynamic shared memory) it has not been allowed in another."""
    r = subprocess.run([sys.executable, "-c", TWO_CONTEXTS], cwd=ROOT, capture_output=True, text=True, timeout=300, env=dict(os.environ, PYTHONPATH=ROOT))
    assert r.returncode == 0 and "same outputs" in r.stdout, r.stdout + r.stderr


# n calls in a row without coming back to Python, whose lock would keep the two threads apart
LOOPS = r"""
#include "carnator.h"
extern "C" int compaction(decltype(&carnator_compact_mask) f, const uint8_t* mask, const carnator_shape* s, void* ws, size_t bytes, void* stream, int n) {
    for (int i = 0; i < n; ++i) if (int st = f(mask, nullptr, s, ws, bytes, stream)) return st;
    return 0;
}
extern "C" int builder(decltype(&carnator_build_connectivity) f, const void* Q, const void* K, const carnator_shape* s, const carnator_build_params* p,
                       uint8_t* mask, void* ws, size_t bytes, void* stream, int n) {
    for (int i = 0; i < n; ++i) if (int st = f(Q, K, s, p, mask, nullptr, ws, bytes, stream)) return st;
    return 0;
}
"""


@pytest.mark.parametrize("call", ["compaction", "builder"])
def test_two_threads_with_layers_of_different_size(call, tmp_path):
    """Kernels whose shared memory grows with the layer: one thread's smaller layer must not take back what another thread's
    larger one is about to be launched with."""
    import ctypes
    import threading

    import torch

    from paper_2609_32420_b200 import build
    from paper_2609_32420_b200 import carnator as cn
    src, lib = tmp_path / "loops.cpp", tmp_path / "loops.so"
    src.write_text(LOOPS)
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I", build.INCLUDE, "-o", str(lib), str(src)], check=True)
    loops = ctypes.CDLL(str(lib))
    vp, n = ctypes.c_void_p, 400
    entry = lambda f: ctypes.cast(f, vp)

    def compaction(nqb, stream):        # 64-token query blocks: 10 bytes of shared memory a row, above the 48 KB that need no leave
        shape = cn.make_shape(1, 1, nqb * 64, 64, 0, 1, 1, nqb * 64, 64, 128)
        mask = torch.ones((1, 1, shape.nqb, shape.nkb), dtype=torch.uint8, device="cuda")
        ws = torch.empty(cn.attn_workspace_bytes(shape), dtype=torch.uint8, device="cuda")
        held = (mask, ws, shape)
        return held, lambda: loops.compaction(entry(cn.lib().carnator_compact_mask), vp(mask.data_ptr()), ctypes.byref(shape), vp(ws.data_ptr()),
                                              ctypes.c_size_t(ws.numel()), vp(stream.cuda_stream), n)

    def builder(nb, stream):            # the persistent builder: a row of scores per query block of an item
        N = nb * 128
        Q, K = (torch.randn((1, 16, N, 64), device="cuda").to(torch.bfloat16) for _ in range(2))
        shape = cn.make_shape(1, 16, N, 64, 0, 1, 1, N, 128, 128, Q, K)
        p = cn.BuildParams()
        p.mode, p.keep_ratio, p.mass, p.window_frames, p.count_includes_forced = cn.MODE_TOPK, 0.2, 0.5, -1, 1
        mask = torch.empty((1, 16, nb, nb), dtype=torch.uint8, device="cuda")
        ws = torch.empty(cn.build_workspace_bytes(shape, p), dtype=torch.uint8, device="cuda")
        held = (Q, K, mask, ws, shape, p)
        return held, lambda: loops.builder(entry(cn.lib().carnator_build_connectivity), vp(Q.data_ptr()), vp(K.data_ptr()), ctypes.byref(shape),
                                           ctypes.byref(p), vp(mask.data_ptr()), vp(ws.data_ptr()), ctypes.c_size_t(ws.numel()), vp(stream.cuda_stream), n)
    make, sizes = (compaction, (5200, 4950)) if call == "compaction" else (builder, (320, 260))
    streams = [torch.cuda.Stream() for _ in sizes]
    jobs = [make(nb, s) for nb, s in zip(sizes, streams)]
    torch.cuda.synchronize()
    status = [None, None]

    def work(i):
        torch.cuda.set_device(0)
        status[i] = jobs[i][1]()
    threads = [threading.Thread(target=work, args=(i,)) for i in (0, 1)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert status == [0, 0], (status, cn.last_cuda_error())


def test_a_refused_launch_does_not_fail_the_next_call():
    """More heads than a grid has rows: the runtime refuses the launch and the call says so.  The next call, a good one, must
    not report that error again."""
    import torch

    from paper_2609_32420_b200 import carnator as cn
    H, N, D = 70000, 64, 64             # heads that share their tokens, one row of 64 apart
    x = torch.randn((N + H, D), device="cuda").to(torch.bfloat16)
    t = x.as_strided((1, H, N, D), (D * (N + H), D, D, 1))
    shape = cn.make_shape(1, H, N, D, 0, 1, 1, N, 64, 64, t, t, t, t)
    mask = torch.ones((1, H, 1, 1), dtype=torch.uint8, device="cuda")
    L = torch.empty((1, H, N), device="cuda")
    O = torch.empty_like(x).as_strided((1, H, N, D), t.stride())
    with pytest.raises(cn.CarnatorError) as e:
        cn.sparse_attn(t, t, t, mask, None, shape, O=O, LSE=L)
    assert e.value.status == cn.ERR_CUDA
    Q = torch.randn((1, 2, 512, D), device="cuda").to(torch.bfloat16)
    shape = cn.make_shape(1, 2, 512, D, 0, 1, 1, 512, 128, 128, Q, Q)
    p = cn.BuildParams()
    p.mode, p.keep_ratio, p.mass, p.window_frames, p.count_includes_forced = cn.MODE_TOPK, 0.5, 0.5, -1, 1
    m, _ = cn.build_connectivity(Q, Q, shape, p)
    assert int(m.sum()) == 2 * 4 * 2


FIRST_CALL = r"""
import threading, torch
from paper_2609_32420_b200 import carnator as cn
n, N, D = 16, 512, 64
x = torch.randn((1, 1, N, D), device="cuda").to(torch.bfloat16)
shapes = [cn.make_shape(1, 1, N, D, 0, 1, 1, N, 128, 128, x, x, x) for _ in range(n)]
spaces = [cn.compact_mask(torch.ones((1, 1, 4, 4), dtype=torch.uint8, device="cuda"), None, s) for s in shapes]
out = [(torch.empty_like(x), torch.empty((1, 1, N), device="cuda")) for _ in range(n)]
torch.cuda.synchronize()
gate, failed = threading.Barrier(n), []
def work(i):
    torch.cuda.set_device(0)
    gate.wait()
    try:
        cn.sparse_attn_compacted(x, x, x, shapes[i], spaces[i], O=out[i][0], LSE=out[i][1])
    except Exception as e:
        failed.append(str(e))
threads = [threading.Thread(target=work, args=(i,)) for i in range(n)]
[t.start() for t in threads]
[t.join() for t in threads]
torch.cuda.synchronize()
assert not failed, failed
assert all(torch.equal(o, out[0][0]) for o, _ in out)
print("all alike")
"""


def test_first_calls_of_many_threads():
    """The driver's tensor-map function is looked up by the first call that needs it; a call that comes during the look-up waits
    for it.  A process of its own: the look-up happens once."""
    r = subprocess.run([sys.executable, "-c", FIRST_CALL], cwd=ROOT, capture_output=True, text=True, timeout=300, env=dict(os.environ, PYTHONPATH=ROOT))
    assert r.returncode == 0 and "all alike" in r.stdout, r.stdout + r.stderr
