"""Batches whose per-sample launches share the GPU by the plan (``batch_plan``): tiles that
divide evenly among a launch's CTAs, a launch with one CTA for all its tiles, three CTAs per
SM, fewer tiles than CTAs, and one CTA per SM.  Against each scenario in a batch of its own:
the same FP32 sums of a tile, added in FP64 in another order."""
import numpy as np
import pytest

import fmc_synth as fs
from gpu_common import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shapes", [
    [(10, 3, 2, 0, 40), (10, 3, 2, 0, 40), (10, 3, 2, 0, 40)],            # 2 SMs of tiles each: even
    [(16, 2, 3, 17, 200), (2, 1, 0, 5000, 8)],                            # one CTA for 40 tiles
    [(8, 2, 1, 100, 70), (9, 1, 1, 40, 70), (5, 8, 1, 0, 70)],            # three CTAs per SM
    [(10, 2, 0, 6000, 300), (4, 2, 2, 5, 40), (12, 4, 1, 77, 40)],        # fewer tiles than CTAs
    [(10, 2, 0, 4900, 50), (3, 1, 0, 5500, 70)]])                         # an SM each
def test_planned_batches(shapes):
    import torch
    fmc = need_gpu()
    ctx, alone = fmc.Context(0), fmc.Context(0, mem_budget_bytes=64 << 30)
    fmc.set_launch_rules([], ctx=ctx)
    fmc.set_launch_rules([], ctx=alone)
    sms = ctx.info()[0]
    scs = [fs.multimachine_case(n=n, d=d, K=24, T=Nt * 0.005, dt=0.005, N=m * sms * 128 + N, seed=n + k)
           for k, (n, d, m, N, Nt) in enumerate(shapes)]
    plan = fmc.batch_plan(scs, sms=sms)
    assert not any(p["team"] for p in plan) and all(p["per_sm"] > 0 for p in plan)
    b = fmc.Batch(scs, ctx=ctx)
    for _ in range(2):
        b.launch()
        fmc.device_status(ctx=ctx)
    for i, sc in enumerate(scs):
        a = fmc.Batch([sc], use_graph=False, ctx=alone)
        a.launch()
        torch.cuda.synchronize()
        for x, y in ((b.mean[i], a.mean[0]), (b.var[i], a.var[0])):
            x, y = x.cpu().numpy(), y.cpu().numpy()
            assert np.max(np.abs(x - y)) <= 1e-9 * np.max(np.abs(y))
        a.close()
    b.close()
    ctx.close()
    alone.close()


@pytest.mark.parametrize("shapes,teams", [
    ([(10, 3, 1000, 400), (10, 3, 4800, 60), (9, 2, 4800, 60), (10, 1, 4500, 60), (10, 2, 4800, 60)], 1),
    ([(12, 2, 1000, 100)] * 8, 8), ([(10, 2, 700, 100)] * 17, 1), ([(8, 2, 4800, 70), (8, 1, 4700, 70)], 0),
    ([(4, 1, 4800, 90), (2, 1, 33, 900), (12, 3, 2000, 90)], 1)])
@pytest.mark.parametrize("use_graph", [False, True])
def test_batches_with_teams(shapes, teams, use_graph):
    import torch
    fmc = need_gpu()
    ctx, alone = fmc.Context(0), fmc.Context(0, mem_budget_bytes=64 << 30)  # (no teams with a budget)
    fmc.set_launch_rules([], ctx=ctx)
    fmc.set_launch_rules([], ctx=alone)
    scs = [fs.multimachine_case(n=n, d=d, K=24, T=Nt * 0.005, dt=0.005, N=N, seed=n + k)
           for k, (n, d, N, Nt) in enumerate(shapes)]
    if ctx.info()[0] == 152:
        assert sum(p["team"] for p in fmc.batch_plan(scs)) == teams
    b = fmc.Batch(scs, use_graph=use_graph, ctx=ctx)
    for _ in range(2):
        b.launch()
        fmc.device_status(ctx=ctx)
    for i, sc in enumerate(scs):
        a = fmc.Batch([sc], use_graph=False, ctx=alone)
        a.launch()
        torch.cuda.synchronize()
        for x, y in ((b.mean[i], a.mean[0]), (b.var[i], a.var[0])):
            x, y = x.cpu().numpy(), y.cpu().numpy()
            assert np.max(np.abs(x - y)) <= 1e-9 * np.max(np.abs(y))
        a.close()
    b.close()
    ctx.close()
    alone.close()
