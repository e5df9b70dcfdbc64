"""How a batch's launches share the GPU (host logic, no GPU; 152 SMs): the CTAs that each
per-sample launch's tiles are dealt to, and the resident CTAs per SM."""
import math

import pytest

import fmc_synth as fs

SMS = 152


@pytest.fixture(scope="module")
def fmc():
    import paper_2007_03847_gb300 as m
    m.build()
    return m


def _sc(n, N, Nt=1000, d=2, **kw):
    return fs.multimachine_case(n=n, d=d, K=20, T=Nt * 0.005, dt=0.005, N=N, seed=n).replace(**kw)


def _arms(n, N):
    return [_sc(n, N), _sc(n, N, sampling=fs.SRS), _sc(n, N, sampling=fs.SRS_EM), _sc(n, N, forcing=fs.FORCING_SMOOTH)]


@pytest.mark.parametrize("N", [10007, 16000, 20000, 24000, 28000])
def test_a_smooth_arm_takes_its_part_only(fmc, N):
    # its tiles are no CTAs of the others': each arm keeps its part of the 304 by its work
    tiles = math.ceil(N / 128)
    plan = fmc.batch_plan(_arms(9, N), sms=SMS)
    assert [p["per_sm"] for p in plan] == [2] * 4
    assert plan[3]["ctas"] == 0  # one CTA per tile
    part = 2 * SMS / 4.4  # the smooth arm's work is 1.4 of another's
    for p in plan[:3]:
        assert int(part) <= p["ctas"] <= min(tiles, math.ceil(2 * SMS - min(tiles, 1.4 * part)) / 3 + 1)


@pytest.mark.parametrize("N", [31000, 38000, 100000])
def test_large_arms_beside_a_smooth_one_keep_a_cta_per_tile(fmc, N):
    plan = fmc.batch_plan(_arms(9, N), sms=SMS)
    assert all(p["ctas"] == 0 and p["per_sm"] == 2 for p in plan)


def test_equal_launches_get_equal_shares(fmc):
    # an SM's tiles each: three CTAs per SM; fewer: two
    assert fmc.batch_plan([_sc(10, 20000)] * 4, sms=SMS) == [{"team": False, "per_sm": 3, "ctas": 3 * SMS // 4}] * 4
    plan = fmc.batch_plan([_sc(10, 6000)] * 12, sms=SMS)
    assert plan == [{"team": False, "per_sm": 2, "ctas": 2 * SMS // 12}] * 12


def test_a_share_may_divide_the_tiles(fmc):
    # 304 tiles on 152 CTAs, and a launch so small beside the other that one CTA is its part:
    # dealt out all the same, not a CTA per tile
    plan = fmc.batch_plan([_sc(10, 304 * 128)] * 3, sms=SMS)
    assert [p["ctas"] for p in plan] == [SMS] * 3
    plan = fmc.batch_plan([_sc(16, 200000, Nt=4000), _sc(1, 6000, Nt=40, d=1)], sms=SMS)
    assert plan[1]["ctas"] == 1


def test_fewer_tiles_than_a_share(fmc):
    # the small launch runs all its tiles at once, the others share what it leaves
    plan = fmc.batch_plan([_sc(10, 6000, Nt=4000), _sc(10, 20000, Nt=500), _sc(10, 20000, Nt=500)], sms=SMS)
    assert plan[0]["ctas"] == 0 and plan[0]["per_sm"] == 2
    assert plan[1]["ctas"] == plan[2]["ctas"] == (2 * SMS - 47) // 2


def test_few_tiles_take_an_sm_each(fmc):
    # 4 x 38 tiles fit the SMs; 5 x 38 take two CTAs per SM
    assert [p["per_sm"] for p in fmc.batch_plan([_sc(10, 4864 + 1)] * 3, sms=SMS)] == [1] * 3
    assert [p["per_sm"] for p in fmc.batch_plan([_sc(10, 4864 + 1)] * 5, sms=SMS)] == [2] * 5
    # a split kernel's CTAs count
    assert [p["per_sm"] for p in fmc.batch_plan([_sc(10, 9000), _sc(30, 12000)], sms=SMS)] == [2, 0]
    # and many launches share, whatever their streams
    plan = fmc.batch_plan([_sc(10, 6000)] * 18, sms=SMS)
    assert all(p["ctas"] == 0 for p in plan)


def test_no_refusal_is_lost(fmc):
    with pytest.raises(fmc.FastMCError):
        fmc.batch_plan([_sc(20, 100, forcing=fs.FORCING_SMOOTH)])
    assert fmc.batch_plan([_sc(5, 100)], path="plain")[0]["ctas"] == 0


def _teams(fmc, scs):
    return [p["team"] for p in fmc.batch_plan(scs, sms=SMS)]


@pytest.mark.parametrize("n,N,count,team", [
    (10, 1000, 1, True), (10, 4864, 1, True), (10, 4865, 1, False),
    (10, 2400, 2, True),      # 150 groups: an SM each
    (12, 1000, 8, True),      # two rounds of teams are still shorter than one of tiles
    (10, 1000, 8, False), (10, 1000, 16, False), (10, 4800, 4, False), (12, 4800, 8, False), (16, 4800, 16, False),
    (8, 1000, 8, True), (8, 2400, 4, True),   # two teams to an SM
    (8, 4800, 2, False), (4, 4800, 2, True), (8, 2400, 8, False), (4, 2400, 8, False), (1, 4800, 16, False)])
def test_teams_while_the_batch_has_room(fmc, n, N, count, team):
    assert _teams(fmc, [_sc(n, N, d=1)] * count) == [team] * count


def test_the_launch_that_the_batch_waits_for(fmc):
    # a long horizon beside short ones; not beside a split kernel's longer chain, nor where
    # the SMs are full for longer than its chain
    assert _teams(fmc, [_sc(10, 1000, Nt=4000)] + [_sc(10, 4800)] * 4) == [True] + [False] * 4
    assert _teams(fmc, [_sc(10, 1000), _sc(50, 1000)]) == [False, False]
    assert _teams(fmc, [_sc(10, 1000), _sc(10, 60000)]) == [False, False]
    # launches of a stream follow one another
    assert sum(_teams(fmc, [_sc(10, 100)] * 33)) > 0


def test_a_smooth_launch_is_the_longest(fmc):
    # 13 to 16 machines: its step alone is twice a split kernel's
    rules = [_sc(14, 2000, forcing=fs.FORCING_SMOOTH), _sc(20, 2000), _sc(20, 2000)]
    assert _teams(fmc, rules) == [True, False, False]
    assert _teams(fmc, [_sc(10, 2000, forcing=fs.FORCING_SMOOTH), _sc(50, 2000)]) == [False, False]


def test_what_is_no_team_alone_is_none_in_a_batch(fmc):
    # (four groups' partials, 240 bytes a time: past 512 MiB from 559241 steps on)
    assert _teams(fmc, [_sc(20, 100), _sc(10, 100, Nt=560000)]) == [False, False]
    assert [p["team"] for p in fmc.batch_plan([_sc(5, 100)], path="plain")] == [False]
