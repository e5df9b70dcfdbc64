"""The sliced form of the per-sample kernel (tiles handed on between CTAs slice by slice)
against the unsliced launch, which a context with a memory budget takes: the same
samples, tiles and operations, so the moments are equal bit for bit.  Sizes: two and
three CTAs per SM, whole tiles before the sliced ones, a partly empty last tile, a last
slice shorter than the others, per-step normals, an event and the response function."""
import numpy as np
import pytest

import fmc_synth as fs
from gpu_common import need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pair():
    fmc = need_gpu()
    plain = fmc.Context(0, mem_budget_bytes=64 << 30)
    yield fmc, plain
    plain.close()


@pytest.mark.parametrize("n,d,N,Nt,opt", [
    (10, 3, 60000, 150, ""), (10, 3, 65536, 333, "heun"), (5, 8, 39500, 100, ""), (4, 5, 40000, 129, "srs_em"),
    (10, 4, 130001, 90, ""), (16, 2, 62000, 300, ""), (9, 3, 45000, 200, "trip")])
def test_sliced_equals_unsliced(pair, n, d, N, Nt, opt):
    import torch
    fmc, plain = pair
    sc = fs.multimachine_case(n=n, d=d, K=24, T=Nt * 0.005, dt=0.005, N=N, seed=n + d)
    if opt == "srs_em":
        sc = sc.replace(sampling=fs.SRS_EM)
    if opt == "heun":
        sc = sc.replace(integrator=fs.HEUN)
    if opt == "trip":
        sc = sc.replace(event_machine=1, event_time=0.3, event_dpm=-1.0)
        (r, m, v), (r1, m1, v1) = (fmc.simulate_rrf(sc, ctx=c) for c in (None, plain))
        # FP64 atomics of the same FP32 values
        assert np.allclose(r.cpu().numpy(), r1.cpu().numpy(), rtol=1e-9)
    else:
        (m, v), (m1, v1) = (fmc.simulate(sc, path="fused", ctx=c) for c in (None, plain))
    fmc.device_status()
    fmc.device_status(ctx=plain)
    assert torch.equal(m, m1) and torch.equal(v, v1)
