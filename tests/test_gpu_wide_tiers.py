"""The split kernel's tensor-core form where its warps leave the shortest series: strong
disturbances drive the angles through the tiers, in the two-warp layout, the layouts
that keep the next stage input in shared memory (ten and thirteen slots), and those
with an infinite bus.  Against the oracle, with the trajectory tolerance of the parity
tests (normwise 1e-4 on angles and speeds)."""
import numpy as np
import pytest

import fmc_synth as fs
from gpu_common import need_gpu, traj_errors

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,bus", [(18, False), (27, False), (30, False), (40, False), (45, False), (52, False),
                                   (30, True), (45, True)])
def test_series_tiers(orc, n, bus):
    fmc = need_gpu()
    sc = fs.multimachine_case(n=n, d=3, K=12, T=0.6, dt=0.005, N=140, seed=60 + n)
    sc = sc.replace(sigma=np.array([40.0, 15.0, 6.0]) * np.sqrt(n / 20.0))
    if bus:
        rng = np.random.default_rng(n)
        sc = sc.replace(has_inf_bus=True, Ginf=np.zeros(n), Binf=rng.uniform(1.0, 3.0, n), Vinf=1.0)
    fmc.set_kernel_policy("split_tc")
    try:
        _, _, traj = fmc.simulate(sc, path="fused", precision="bf16x3", want_traj=True)
    finally:
        fmc.set_kernel_policy("auto")
    fmc.device_status()
    ref = orc.simulate(sc, orc.lhs_sample(sc.seed, sc.N, sc.M), want_traj=True, nthreads=8)
    dev = ref["traj"][..., :n] - ref["traj"][:, :1, :n]
    rel = np.abs(dev - dev.mean(axis=2, keepdims=True)).max()
    assert 0.25 < rel < 3.0, rel  # past two tiers at least
    ed, ew = traj_errors(traj.cpu().numpy(), ref["traj"], n)
    assert ed <= 1e-4 and ew <= 1e-4, (ed, ew)
