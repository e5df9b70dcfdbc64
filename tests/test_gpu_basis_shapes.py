"""The increment basis at the edges of its launch shapes: one entry per thread or several,
blocks of 64 or 256 threads, with the cosine table and without (the same operations either
way, so equal bits).  FP32 against the oracle's FP64 (rounded once: 2 ulps of the largest
entry); the split form through reconstructions with the table (from 32768 entries on) and
without (the allocation-free form)."""
import numpy as np
import pytest

from gpu_common import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K,Nt", [(1, 1), (3, 65), (6, 400), (50, 500), (6, 12000), (31, 1057), (97, 1603), (9, 70001)])
@pytest.mark.parametrize("basis", [0, 1])
def test_f32_rows(orc, K, Nt, basis):
    fmc = need_gpu()
    phi = fmc.kl_basis(K, 7.5, Nt, basis).cpu().numpy()
    ref = orc.kl_increment_basis(K, 7.5, Nt, basis)
    assert np.max(np.abs(phi - ref)) <= 2 * 2.0**-23 * np.max(np.abs(ref))


@pytest.mark.parametrize("K,Nt", [(1, 8), (20, 300), (32, 1023), (32, 1024), (33, 993), (100, 1000), (70, 4001)])
@pytest.mark.parametrize("precision", ["bf16x3", "bf16", "f32"])
def test_table_and_direct_cosines_agree(K, Nt, precision):
    import torch
    fmc = need_gpu()
    z, _ = fmc.lhs_sample(9, 70, 2 * K)
    a = fmc.kle_reconstruct(z, 2, K, Nt * 0.005, 0.005, precision=precision)
    b = fmc.kle_reconstruct_noalloc(z, 2, K, Nt * 0.005, 0.005, precision=precision)
    fmc.device_status()
    assert torch.equal(a, b)
