"""The error word that a call reports: on both paths it is this call's own, whatever the
memory held before.  The server's buffers come from the device's default memory pool, so
the pool is left full of another value first."""
import ctypes

import pytest

import fmc_synth as fs
from gpu_common import need_gpu

pytestmark = pytest.mark.gpu


def _fill_pool(value):
    """Allocates most of 64 MB of the default pool, fills it and gives it back."""
    cu = ctypes.CDLL("libcuda.so.1")
    pool, keep = ctypes.c_void_p(), ctypes.c_uint64(1 << 30)
    assert cu.cuDeviceGetDefaultMemPool(ctypes.byref(pool), 0) == 0
    assert cu.cuMemPoolSetAttribute(pool, 4, ctypes.byref(keep)) == 0  # the release threshold
    held = []
    for size in [64 << 20] + [1 << 16] * 64 + [512] * 256:
        p = ctypes.c_uint64()
        assert cu.cuMemAllocFromPoolAsync(ctypes.byref(p), ctypes.c_size_t(size), pool, None) == 0
        assert cu.cuMemsetD8Async(p, ctypes.c_ubyte(value), ctypes.c_size_t(size), None) == 0
        held.append(p)
    for p in held:
        assert cu.cuMemFreeAsync(p, None) == 0
    assert cu.cuStreamSynchronize(None) == 0


@pytest.mark.parametrize("path,precision", [("plain", "f32"), ("fused", "bf16x3")])
def test_memory_of_a_new_server_holds_other_values(path, precision):
    fmc = need_gpu()
    fmc.default_context()
    sc = fs.multimachine_case(n=4, d=2, K=10, T=0.2, dt=0.005, N=100, seed=3)
    _fill_pool(0x55)
    srv = fmc.Server(slots=1, mem_budget_bytes=1 << 30)
    try:
        for _ in range(2):
            res, _, _ = srv.wait(srv.submit(sc, path=path, precision=precision))
            assert res["status"] == 0, res["message"]
    finally:
        srv.close()
