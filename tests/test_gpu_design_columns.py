"""The design kernel's split into column blocks: fewer than four columns (a block each), and
block widths with one to three columns left over, over every form of the permutation
(8-bit and 16-bit tables, rounds by definition, none, given strata).  Strata are whole
numbers and bit-exact against the oracle; values equal those of the whole design's first
columns, whatever the width it is computed in."""
import numpy as np
import pytest

from gpu_common import need_gpu

pytestmark = pytest.mark.gpu

SIZES = [(3, 3), (1000, 1000), (4096, 4096), (65536, 700), (65537, 2100), ((1 << 22) + 5, 300)]


@pytest.mark.parametrize("N,count", SIZES)
@pytest.mark.parametrize("mode", [0, 1, 2])
def test_few_columns(orc, N, count, mode):
    import torch
    fmc = need_gpu()
    k0 = N - count
    wide = torch.empty((16, count), dtype=torch.int32, device="cuda")
    zw, _ = fmc.lhs_sample(5, N, 16, mode=mode, k0=k0, count=count, strata=wide)
    if mode == 0:
        _, ref = orc.lhs_sample(5, N, 16, mode=orc.LHS, k0=k0, count=count, with_strata=True)
        assert np.array_equal(wide.cpu().numpy().view(np.uint32), ref)
    for M in (1, 2, 3, 4, 5, 6, 7, 9):
        st = torch.full((M + 1, count), -1, dtype=torch.int32, device="cuda")
        z = torch.full((count * M + 64,), 7.0, device="cuda")
        fmc.lhs_sample(5, N, M, mode=mode, k0=k0, count=count, zeta=z[:count * M].view(count, M), strata=st[:M])
        assert torch.equal(z[:count * M].view(count, M), zw[:, :M]) and torch.all(z[count * M:] == 7.0)
        assert torch.equal(st[:M], wide[:M]) and torch.all(st[M] == -1)


@pytest.mark.parametrize("M", [1, 2, 3, 5])
def test_given_strata(M):
    import torch
    fmc = need_gpu()
    N = 3001
    zeta = torch.empty((N, M), device="cuda")
    strata = torch.empty((M, N), dtype=torch.int32, device="cuda")
    fmc.lhs_decorrelate(8, N, M, zeta=zeta, strata=strata)
    s = strata.cpu().numpy().view(np.uint32)
    assert all(np.array_equal(np.sort(row), np.arange(N)) for row in s)
    # every value lies in its own stratum
    p = torch.special.ndtr(zeta.double()).cpu().numpy().T * N
    assert np.all(np.abs(p - (s + 0.5)) <= 0.5 + 1e-6 * N)


@pytest.mark.parametrize("N,M,k0,count", [
    (1 << 22, 20, 70001, 30000), (1 << 22, 2, 5, 9000), (65536, 4, 0, 65536), (65536, 5, 65000, 536),
    (262144, 4, 100000, 3000), (100000, 9, 0, 100000)])
def test_where_tables_and_rounds_meet(orc, N, M, k0, count):
    # blocks whose CTAs with tables would leave SMs idle take the rounds by definition
    import torch
    fmc = need_gpu()
    st = torch.empty((M, count), dtype=torch.int32, device="cuda")
    fmc.lhs_sample(11, N, M, k0=k0, count=count, strata=st)
    _, ref = orc.lhs_sample(11, N, M, mode=orc.LHS, k0=k0, count=count, with_strata=True)
    assert np.array_equal(st.cpu().numpy().view(np.uint32), ref)
