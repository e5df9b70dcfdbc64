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


# Launches of a batch that share the GPU: more tiles than two CTAs per SM hold, so each
# launch gets a share of the CTAs and hands its tiles on slice by slice (the smooth one
# does not).  Against a batch of each scenario by itself in the context with a budget: the
# same FP32 sums of a tile, added in FP64 in another order (at most a few hundred terms of
# 2^-53 each).
@pytest.mark.parametrize("shapes", [
    [(9, 2, 10007, 97, ""), (9, 2, 10007, 97, "srs"), (9, 2, 10007, 97, "srs_em"), (9, 2, 10007, 97, "smooth")],
    [(4, 3, 60000, 50, ""), (10, 3, 5000, 333, ""), (16, 1, 20001, 129, "heun")],
    [(2, 1, 100000, 40, ""), (5, 2, 130, 64, ""), (12, 8, 6000, 65, "")]])
@pytest.mark.parametrize("use_graph", [False, True])
def test_batch_shares(pair, shapes, use_graph):
    fmc, plain = pair
    scs = []
    for k, (n, d, N, Nt, opt) in enumerate(shapes):
        sc = fs.multimachine_case(n=n, d=d, K=24, T=Nt * 0.005, dt=0.005, N=N, seed=n + d + k)
        scs.append(sc.replace(**{"": {}, "srs": dict(sampling=fs.SRS), "srs_em": dict(sampling=fs.SRS_EM),
                                 "smooth": dict(forcing=fs.FORCING_SMOOTH), "heun": dict(integrator=fs.HEUN)}[opt]))
    ctx = fmc.Context(0)  # (13 to 16 machines: the per-sample kernel, not a measured rule's)
    fmc.set_launch_rules([], ctx=ctx)
    fmc.set_launch_rules([], ctx=plain)
    alone = []
    for sc in scs:
        a = fmc.Batch([sc], use_graph=False, ctx=plain)
        alone.append([t.cpu().numpy() for ts in a.launch() for t in ts])
        a.close()
    b = fmc.Batch(scs, use_graph=use_graph, ctx=ctx)
    for _ in range(2):
        b.launch()
        fmc.device_status(ctx=ctx)
        for m, v, (m1, v1) in zip(b.mean, b.var, alone):
            for x, y in ((m.cpu().numpy(), m1), (v.cpu().numpy(), v1)):
                assert np.max(np.abs(x - y)) <= 1e-9 * np.max(np.abs(y))
    b.close()
    ctx.close()
