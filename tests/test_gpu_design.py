"""The tabulated permutation of the design kernel at the edges of its ranges: exact
powers of four and their neighbours (no cycle walking, much of it), the last
sizes of the 8-bit and 16-bit tables, the rounds by definition beyond them and for
short blocks, ragged rows and columns.  Strata are whole numbers: bit-exact
against the oracle; a block of rows equals the same rows of the whole design."""
import numpy as np
import pytest

from gpu_common import need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fmc():
    return need_gpu()


def _sample(fmc, N, M, k0, count, mode=0):
    import torch
    strata = torch.empty((M, count), dtype=torch.int32, device="cuda")
    zeta, _ = fmc.lhs_sample(23, N, M, mode=mode, k0=k0, count=count, strata=strata)
    return zeta, strata


@pytest.mark.parametrize("N,M,k0,count", [
    (4, 17, 0, 4), (5, 16, 0, 5), (256, 15, 0, 256), (257, 33, 0, 257), (4097, 16, 1, 3000),
    (16384, 3, 0, 16384), (65536, 2, 60000, 511), (65536, 2, 60000, 512),
    (65537, 9, 64000, 1024), (262144, 3, 5, 2047), (262145, 8, 260000, 2048),
    (1 << 22, 2, 7, 4096), ((1 << 22) + 1, 2, 7, 9000), ((1 << 24) + 1, 1, 3, 40)])
def test_strata_at_the_edges(fmc, orc, N, M, k0, count):
    _, strata = _sample(fmc, N, M, k0, count)
    _, sr = orc.lhs_sample(23, N, M, mode=orc.LHS, k0=k0, count=count, with_strata=True)
    assert np.array_equal(strata.cpu().numpy().view(np.uint32), sr)


@pytest.mark.parametrize("N,M", [(65536, 19), (65537, 19), (100000, 7)])
@pytest.mark.parametrize("mode", [0, 1, 2])
def test_blocks_equal_the_whole_design(fmc, N, M, mode):
    import torch
    whole, ws = _sample(fmc, N, M, 0, N, mode)
    for k0, count in ((0, 31), (511, 1), (40000, 5000)):
        part, ps = _sample(fmc, N, M, k0, count, mode)
        assert torch.equal(part, whole[k0:k0 + count])
        assert torch.equal(ps, ws[:, k0:k0 + count])


@pytest.mark.parametrize("N,d,K", [(1000, 1, 1), (65536, 3, 13), (5000, 2, 50), (70001, 2, 8)])
@pytest.mark.parametrize("mode", [0, 1, 2])
def test_split_rows_are_the_values(fmc, N, d, K, mode):
    import torch
    zeta, _ = fmc.lhs_sample(9, N, d * K, mode=mode)
    hi, lo = fmc.lhs_sample_split(9, N, d, K, mode=mode)
    z = zeta.view(N, d, K)
    h = z.to(torch.bfloat16)
    assert torch.equal(hi[:, :, :K], h)
    assert torch.equal(lo[:, :, :K], (z - h.float()).to(torch.bfloat16))
    assert not hi[:, :, K:].any() and not lo[:, :, K:].any()
