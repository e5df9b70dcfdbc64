"""Which form a single fused launch takes at the lines of the rules, with sample counts from
the device's SM count, and that the forms give the same moments where each of them did run:
teams of warps against the per-sample kernel, tiles dealt to a fixed grid against a CTA per
tile (which a context with a memory budget takes)."""
import pytest

import fmc_synth as fs
from gpu_common import need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def two():
    fmc = need_gpu()
    free, bounded = fmc.Context(0), fmc.Context(0, mem_budget_bytes=64 << 30)
    for c in (free, bounded):
        fmc.set_launch_rules([], ctx=c)
    yield fmc, free, bounded, free.info()[0]
    free.close()
    bounded.close()


def _sc(n, N, Nt=60, **kw):
    return fs.multimachine_case(n=n, d=2, K=12, T=Nt * 0.005, dt=0.005, N=N, seed=n).replace(**kw)


@pytest.mark.parametrize("n", [4, 9, 13, 16])
def test_teams_up_to_an_sm_each(two, n):
    import torch
    fmc, free, bounded, sms = two
    sc = _sc(n, 32 * sms)
    m, v = fmc.simulate(sc, ctx=free)
    assert fmc.last_form(free) == ("team", sms)
    assert fmc.fused_occupancy(free) >= 1
    m1, v1 = fmc.simulate(sc, ctx=bounded)
    assert fmc.last_form(bounded) == ("per_sample", (32 * sms + 127) // 128)
    fmc.device_status(free)
    fmc.device_status(bounded)
    assert torch.equal(m, m1) and torch.equal(v, v1)
    fmc.simulate(_sc(n, 32 * sms + 1), ctx=free)
    assert fmc.last_form(free)[0] == "per_sample"
    assert fmc.fused_occupancy(free) >= 1


@pytest.mark.parametrize("tiles,grid", [
    (lambda s: 2 * s, 0), (lambda s: 2 * s + 1, 2), (lambda s: 14 * s // 5 - 1, 2), (lambda s: 3 * s, 0),
    (lambda s: 3 * s + 1, 3), (lambda s: 7 * s // 2, 3), (lambda s: 4 * s, 0)])
def test_tiles_dealt_to_a_grid(two, tiles, grid):
    import torch
    fmc, free, bounded, sms = two
    t = tiles(sms)
    sc = _sc(10, 128 * t - 5, Nt=100)
    m, v = fmc.simulate(sc, ctx=free)
    assert fmc.last_form(free) == (("sliced", grid * sms) if grid else ("per_sample", t))
    m1, v1 = fmc.simulate(sc, ctx=bounded)
    assert fmc.last_form(bounded) == ("per_sample", t)
    fmc.device_status(free)
    fmc.device_status(bounded)
    assert torch.equal(m, m1) and torch.equal(v, v1)


def test_other_forms(two):
    fmc, free, _, _ = two
    for sc, form in ((_sc(20, 200), "split_tc"), (_sc(16, 200), "team"),
                     (_sc(10, 200, forcing=fs.FORCING_SMOOTH), "team")):
        fmc.simulate(sc, ctx=free)
        assert fmc.last_form(free)[0] == form
    fmc.simulate(_sc(5, 100), path="plain", precision="f32", ctx=free)
    assert fmc.last_form(free) == ("none", 0)
    for policy, form in (("split", "split"), ("per_sample", "per_sample")):
        fmc.set_kernel_policy(policy, ctx=free)
        fmc.simulate(_sc(14, 100), ctx=free)
        assert fmc.last_form(free)[0] == form
    fmc.set_kernel_policy("auto", ctx=free)
