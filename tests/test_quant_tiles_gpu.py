"""The codec's kernels at the edges of their groups (16 values per lane, a warp or a CTA per block, remainders of n) and of the
scale range in which codes are divided by a reciprocal and an exact remainder: bit for bit against the CPU oracle."""
import numpy as np
import pytest
import torch

from oracle import quant_oracle as qo

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,block", [(15, 16), (16 * 33 + 1, 16), (512 * 3 - 1, 32), (64 * 70 + 17, 64), (512 * 5 + 511, 512),      # sixteen per lane
                                     (100 * 37 + 3, 100), (1000 * 3 + 998, 1000), (4 * 9 + 1, 4), (1020 * 2 + 2, 1020),              # a warp per block
                                     (1024 * 3 + 1, 1024), (4096 * 2 + 4095, 4096), (48 * 11 + 7, 48), (33 * 20 + 5, 33)])
@pytest.mark.parametrize("scale", [1.0, 1e-31, 1e32])
def test_bit_exact(n, block, scale):
    import paper_2408_10746_b200 as pac
    x = torch.randn(n, generator=torch.Generator().manual_seed(n)) * scale
    x[:: max(2, n // 5)] = 0.0
    q, c = pac.quantize_absmax(x.cuda(), block)
    out = pac.dequantize_absmax(q, c, block)
    torch.cuda.synchronize()
    rq, rc = qo.quantize_absmax(x.numpy(), block)
    assert np.array_equal(q.cpu().numpy(), rq)
    assert np.array_equal(c.cpu().numpy().view(np.uint32), rc.view(np.uint32))
    assert np.array_equal(out.cpu().numpy().view(np.uint32), qo.dequantize_absmax(rq, rc, block).view(np.uint32))
