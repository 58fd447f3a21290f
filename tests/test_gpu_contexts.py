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
