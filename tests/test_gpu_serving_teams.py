"""Requests of a server that would take the team kernel alone, more of them at once than the
SMs have room for: some run by teams, others by the per-sample kernel, as they come.  The
same moments as each scenario alone in a batch without teams (FP64 sums in another order),
and every charge is given back."""
import numpy as np
import pytest

import fmc_synth as fs
from gpu_common import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,N,slots,count", [(10, 4800, 8, 12), (4, 3000, 4, 9), (16, 500, 8, 10)])
def test_more_teams_than_room(n, N, slots, count):
    import torch
    fmc = need_gpu()
    alone = fmc.Context(0, mem_budget_bytes=64 << 30)
    fmc.set_launch_rules([], ctx=alone)
    scs = [fs.multimachine_case(n=n, d=2, K=24, T=0.5, dt=0.005, N=N - 7 * k, seed=n + k) for k in range(count)]
    srv = fmc.Server(slots=slots, mem_budget_bytes=8 << 30)
    try:
        for _ in range(2):
            handles = [srv.submit(sc) for sc in scs]
            done = [srv.wait(h) for h in handles]
            assert all(res["status"] == 0 for res, _, _ in done), [res["message"] for res, _, _ in done]
        assert srv.stats() == {"queued": 0, "running": 0, "bytes_in_use": 0}
    finally:
        srv.close()
    for sc, (_, mean, var) in zip(scs, done, strict=True):
        b = fmc.Batch([sc], use_graph=False, ctx=alone)
        b.launch()
        torch.cuda.synchronize()
        for x, y in ((mean, b.mean[0]), (var, b.var[0])):
            x, y = x.cpu().numpy(), y.cpu().numpy()
            assert np.max(np.abs(x - y)) <= 1e-9 * np.max(np.abs(y))
        b.close()
    alone.close()
