"""The contraction's bulk stores where a warp holds a few rows only and a block spans two
store passes (256 steps): the lanes without a row skip the copy and its wait, and meet the
others again before the warp's next loads from TMEM.  Against plain stores (a result buffer
that starts 4 bytes on): the same accumulators, bit for bit.  Sizes: one row, all but one,
and one warp's worth and a row in the last tile of 128; a last block of 232 steps."""
import pytest

from gpu_common import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rest", [1, 31, 33, 127])
@pytest.mark.parametrize("precision", ["bf16x3", "bf16"])
def test_partial_warps_in_blocks_of_256_steps(rest, precision):
    import torch
    fmc = need_gpu()
    count, d, K, Nt, dt = 16384 + rest, 2, 24, 1000, 0.01
    zeta, _ = fmc.lhs_sample(6, count, d * K)
    size = count * d * Nt
    out = []
    for first in (4, 5):
        buf = torch.full((size + 16,), -7.0, dtype=torch.float32, device="cuda")
        fmc.kle_reconstruct(zeta, d, K, Nt * dt, dt, precision=precision, dW=buf[first:first + size])
        fmc.device_status()
        assert torch.all(buf[:first] == -7.0) and torch.all(buf[first + size:] == -7.0)
        out.append(buf[first:first + size])
    assert torch.equal(*out)
