"""A launch rule that names a split kernel and a scenario with smooth forcing, which only the
per-sample kernel takes: the rule's kernel is ignored, as it is for other systems that it
cannot take, in single calls and in batches.  The same kernel as without rules, so the
moments are equal (a batch adds them with FP64 atomics: to rounding)."""
import numpy as np
import pytest

import fmc_synth as fs
from gpu_common import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,N", [(8, 300), (13, 300), (16, 6000)])
@pytest.mark.parametrize("kernel", [2, 3])
def test_smooth_forcing_passes_a_split_rule_by(n, N, kernel):
    import torch
    fmc = need_gpu()
    sc = fs.multimachine_case(n=n, d=2, K=20, T=0.2, dt=0.005, N=N, seed=n).replace(forcing=fs.FORCING_SMOOTH)
    ctx = fmc.Context(0)
    try:
        fmc.set_launch_rules([], ctx=ctx)
        m0, v0 = fmc.simulate(sc, ctx=ctx)
        fmc.set_launch_rules([dict(kernel=kernel)], ctx=ctx)
        m1, v1 = fmc.simulate(sc, ctx=ctx)
        assert torch.equal(m0, m1) and torch.equal(v0, v1)
        b = fmc.Batch([sc], ctx=ctx)
        bm, bv = b.launch()
        fmc.device_status(ctx)
        for x, y in ((bm[0], m0), (bv[0], v0)):
            # FP32 partials merged by tiles, or tile by tile: 2^-24 of the spread at most
            assert np.max(np.abs((x - y).cpu().numpy())) <= 1e-5 * np.max(np.abs(y.cpu().numpy()))
        b.close()
    finally:
        ctx.close()
