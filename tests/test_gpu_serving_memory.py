"""What a served request holds on the device against what it was charged: the high-water
mark of the device's default memory pool, which the server's workspaces come from.  Shapes
where the cosine table and the team kernel's partials are a large part: few samples and few
KL terms over a long horizon, with and without the table, and a target-error request."""
import ctypes

import pytest

import fmc_synth as fs
from gpu_common import need_gpu

pytestmark = pytest.mark.gpu

USED, USED_HIGH = 7, 8  # CU_MEMPOOL_ATTR_USED_MEM_CURRENT, _HIGH


@pytest.fixture(scope="module")
def pool():
    fmc = need_gpu()
    fmc.default_context()
    cu = ctypes.CDLL("libcuda.so.1")
    p = ctypes.c_void_p()
    assert cu.cuDeviceGetDefaultMemPool(ctypes.byref(p), 0) == 0

    def value(attr, reset=False):
        v = ctypes.c_uint64(0)
        f = cu.cuMemPoolSetAttribute if reset else cu.cuMemPoolGetAttribute
        assert f(p, attr, ctypes.byref(v)) == 0
        return v.value
    return fmc, value


@pytest.mark.parametrize("n,N,K,Nt,precision,path,tol,budget", [
    (2, 64, 6, 100000, "bf16x3", "fused", 0.0, 1 << 30),      # table and partials
    (2, 64, 32, 100000, "bf16", "fused", 0.0, 1 << 30),
    (2, 64, 6, 100000, "bf16x3", "fused", 0.0, 15_000_000),   # neither fits
    (20, 64, 6, 20000, "bf16x3", "fused", 0.0, 1 << 30),      # no team
    (10, 4800, 10, 4000, "bf16x3", "fused", 0.0, 1 << 30),    # mostly partials
    (4, 100, 6, 50000, "f32", "plain", 0.0, 1 << 30),
    (2, 128, 6, 50000, "bf16x3", "fused", 1e-9, 2 << 30),     # replicates in one launch
    (2, 100, 6, 50000, "bf16x3", "fused", 1e-9, 2 << 30)])    # ... and in four
def test_charge_covers_the_workspace(pool, n, N, K, Nt, precision, path, tol, budget):
    import torch
    fmc, value = pool
    sc = fs.multimachine_case(n=n, d=1, K=K, T=Nt * 1e-4, dt=1e-4, N=N, seed=n)
    srv = fmc.Server(slots=1, mem_budget_bytes=budget)
    try:
        torch.cuda.synchronize()
        before = value(USED)
        value(USED_HIGH, reset=True)
        more = dict(tol_E=tol, max_N=4 * N) if tol else {}
        res, mean, var = srv.wait(srv.submit(sc, path=path, precision=precision, **more))
        assert res["status"] == 0, res["message"]
        assert res["device_bytes"] <= budget
        # a target's replicate moments (FP64, 2 x 4 designs) are outside the charge, and small buffers
        # of every context (equilibrium, status) are rounded up by the pool
        outside = (8 * 2 * (Nt + 1) * 2 * n * 4 if tol else 0) + (1 << 18)
        assert value(USED_HIGH) - before <= res["device_bytes"] + outside
    finally:
        srv.close()
