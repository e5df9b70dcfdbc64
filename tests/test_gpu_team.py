"""The team kernel (few samples, up to 12 machines) against the per-sample kernel it
stands in for: the same FP32 operations in the same order, so trajectories and
moments are equal bit for bit.  Sizes at its edges: partial groups of 32 and tiles
of 128, every machine-slot bucket with and without padding, one step, partial time
chunks and moment buffers, every option that changes the paths or the step."""
import numpy as np
import pytest

import fmc_synth as fs
from gpu_common import need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fmc():
    return need_gpu()


def _both(fmc, call):
    out = []
    for policy in ("auto", "per_sample"):
        fmc.set_kernel_policy(policy)
        try:
            out.append(call())
            fmc.device_status()
        finally:
            fmc.set_kernel_policy("auto")
    return out


def _equal(fmc, sc, **kw):
    import torch
    team, one = _both(fmc, lambda: fmc.simulate(sc, path="fused", want_traj=True, **kw))
    for a, b in zip(team, one):
        assert torch.equal(torch.nan_to_num(a), torch.nan_to_num(b))
        assert torch.equal(a.isnan(), b.isnan())


@pytest.mark.parametrize("n,d,N,T", [
    (2, 1, 1, 0.005), (3, 2, 31, 0.03), (4, 4, 32, 0.165), (5, 3, 33, 0.3), (8, 5, 127, 0.2), (9, 2, 128, 0.7),
    (10, 3, 129, 0.5), (10, 8, 1000, 0.1), (11, 1, 257, 0.4), (12, 8, 100, 0.2), (7, 3, 5000, 0.05)])
@pytest.mark.parametrize("precision", ["bf16x3", "bf16"])
def test_team_equals_per_sample(fmc, n, d, N, T, precision):
    _equal(fmc, fs.multimachine_case(n=n, d=d, K=37, T=T, dt=0.005, N=N, seed=n * 100 + d), precision=precision)


@pytest.mark.parametrize("opt", ["smib", "smib_strong", "heun", "srs_em", "cosine", "trip", "ito", "smooth", "smooth_heun",
                                 "smooth_trip"])
def test_team_options(fmc, opt):
    sc = fs.multimachine_case(n=6, d=3, K=20, T=0.6, dt=0.005, N=300, seed=5)
    sc = {"smib": lambda: fs.smib_case(N=300, K=20, T=1.0),
          # angle deviations through all series tiers
          "smib_strong": lambda: fs.smib_case(N=300, K=20, T=2.0, sigma=1.0),
          "heun": lambda: sc.replace(integrator=fs.HEUN),
          "srs_em": lambda: sc.replace(sampling=fs.SRS_EM),
          "cosine": lambda: sc.replace(basis=fs.BASIS_COSINE),
          "trip": lambda: sc.replace(event_machine=2, event_time=0.2, event_dpm=-2.0),
          "ito": lambda: sc.replace(ito=[None, fs.ito_gamma(2.0, 20.0), fs.ito_wind()]),
          "smooth": lambda: sc.replace(forcing=fs.FORCING_SMOOTH),
          "smooth_heun": lambda: sc.replace(forcing=fs.FORCING_SMOOTH, integrator=fs.HEUN),
          "smooth_trip": lambda: sc.replace(forcing=fs.FORCING_SMOOTH, event_machine=0, event_time=0.1,
                                            event_dpm=-0.5)}[opt]()
    _equal(fmc, sc)


def test_team_response_function_and_blocks(fmc):
    import torch
    sc = fs.multimachine_case(n=9, d=2, K=10, T=0.5, dt=0.005, N=333, seed=8).replace(
        event_machine=1, event_time=0.1, event_dpm=-0.4)
    (r, m, v), (r1, m1, v1) = _both(fmc, lambda: fmc.simulate_rrf(sc))
    assert torch.equal(m, m1) and torch.equal(v, v1)
    # the response function's sums are FP64 atomics of the same FP32 values
    assert np.allclose(r.cpu().numpy(), r1.cpu().numpy(), rtol=1e-9)
    s, s1 = _both(fmc, lambda: fmc.simulate_sums(sc, 100, 130))
    assert all(torch.equal(a, b) for a, b in zip(s, s1))


@pytest.mark.parametrize("n,d,N,T", [(13, 3, 70, 0.2), (14, 1, 33, 0.165), (16, 8, 300, 0.1)])
@pytest.mark.parametrize("precision", ["bf16x3", "bf16"])
def test_team_of_sixteen_equals_per_sample(fmc, n, d, N, T, precision):
    # without launch rules (a measured one may take the split kernel for these systems)
    from paper_2007_03847_gb300 import autotune
    fmc.set_launch_rules([])
    try:
        _equal(fmc, fs.multimachine_case(n=n, d=d, K=37, T=T, dt=0.005, N=N, seed=n * 100 + d), precision=precision)
    finally:
        autotune.apply_cached(fmc.default_context())
