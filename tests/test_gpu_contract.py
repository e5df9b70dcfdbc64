"""The contraction's two ways of storing its rows: bulk copies where every row of the result
starts on 16 bytes, else transposes and plain stores (here by a result buffer that starts
4 bytes on).  The same accumulators, so the increments are equal bit for bit, and nothing
outside the result is written.  Sizes: partial row tiles and column blocks, one sample, four
steps, one K block and several."""
import pytest

from gpu_common import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("count,d,K,Nt", [(1, 1, 1, 4), (129, 3, 200, 1300), (4100, 2, 33, 128), (257, 8, 7, 132),
                                          (640, 1, 288, 2000), (31, 2, 40, 1001)])
@pytest.mark.parametrize("precision", ["bf16x3", "bf16"])
def test_bulk_stores_equal_plain_stores(count, d, K, Nt, precision):
    import torch
    fmc = need_gpu()
    dt = 0.01
    zeta, _ = fmc.lhs_sample(5, count, d * K)
    size = count * d * Nt
    out = []
    for first in (4, 5):  # floats before the result: 16-byte aligned, and not
        buf = torch.full((size + 16,), -7.0, dtype=torch.float32, device="cuda")
        fmc.kle_reconstruct(zeta, d, K, Nt * dt, dt, precision=precision, dW=buf[first:first + size])
        fmc.device_status()
        assert torch.all(buf[:first] == -7.0) and torch.all(buf[first + size:] == -7.0)
        out.append(buf[first:first + size].clone())
    assert torch.equal(out[0], out[1])


@pytest.mark.parametrize("count,d,K,Nt", [(8200, 2, 40, 1001), (16500, 2, 7, 132), (8192, 2, 288, 1000)])
@pytest.mark.parametrize("precision", ["bf16x3", "bf16"])
def test_blocks_of_256_steps_equal_blocks_of_128(count, d, K, Nt, precision):
    # the whole takes blocks of 256 steps, 640 rows at a time take blocks of 128
    import torch
    fmc = need_gpu()
    dt = 0.01
    zeta, _ = fmc.lhs_sample(5, count, d * K)
    whole = fmc.kle_reconstruct(zeta, d, K, Nt * dt, dt, precision=precision)
    fmc.device_status()
    for r in range(0, count, 640):
        part = fmc.kle_reconstruct(zeta[r:r + 640].contiguous(), d, K, Nt * dt, dt, precision=precision)
        assert torch.equal(whole[r:r + 640], part)
