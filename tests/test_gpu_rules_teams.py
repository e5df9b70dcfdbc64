"""Launch rules and teams: a rule that names the per-sample kernel keeps teams off, in single
calls and in batches; a rule that leaves the kernel to the library does not; and the
measured table of this GPU leaves it for up to 10 machines.  The same moments either way."""
import json
import os

import pytest

import fmc_synth as fs
from gpu_common import need_gpu


@pytest.mark.gpu
@pytest.mark.parametrize("kernel,form", [(1, "per_sample"), (0, "team"), (2, "split")])
def test_a_rules_kernel(kernel, form):
    import torch
    fmc = need_gpu()
    ctx = fmc.Context(0)
    try:
        fmc.set_launch_rules([], ctx=ctx)
        sc = fs.multimachine_case(n=9, d=3, K=12, T=0.3, dt=0.005, N=500, seed=4)
        m, v = fmc.simulate(sc, ctx=ctx)
        assert fmc.last_form(ctx)[0] == "team"
        fmc.set_launch_rules([dict(n_min=5, n_max=10, kernel=kernel, max_ctas=1, TC=32)], ctx=ctx)
        m1, v1 = fmc.simulate(sc, ctx=ctx)
        assert fmc.last_form(ctx)[0] == form
        b = fmc.Batch([sc], use_graph=False, ctx=ctx)
        b.launch()
        fmc.device_status(ctx)
        assert fmc.last_form(ctx)[0] == form
        b.close()
        if kernel != 2:
            assert torch.equal(m, m1) and torch.equal(v, v1)
    finally:
        ctx.close()


def test_the_measured_table_names_no_per_sample_kernel():
    from paper_2007_03847_gb300 import autotune
    with open(os.path.join(autotune.TUNING_DIR, "NVIDIA_GB300_152sm.json")) as f:
        rules = json.load(f)["rules"]
    # (what it measured for up to 16 machines besides the split kernels is the library's own choice)
    assert rules and all(r["kernel"] != 1 for r in rules)
    assert all(r["kernel"] == 0 for r in rules if r["n_max"] <= 10)
    assert all(c[0] != 1 for n in (4, 10, 16, 20) for c in autotune.candidates(n))
