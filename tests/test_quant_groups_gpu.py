"""Blocks of a multiple of four: several of them per warp when quantised, sixteen codes across two of them when dequantised.  Bit for bit against the CPU oracle."""
import numpy as np
import pytest
import torch

from oracle import quant_oracle as qo

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("block", [20, 36, 100, 124, 128 + 4, 256, 256 + 4, 512 + 4, 1000, 1020, 1024])
@pytest.mark.parametrize("blocks,rest", [(1, -1), (1, 0), (7, 3), (8, 0), (9, 5), (1200, 1), (20000, 2)])
def test_bit_exact(block, blocks, rest):
    import paper_2408_10746_b200 as pac
    n = blocks * block + rest
    x = torch.randn(n, generator=torch.Generator().manual_seed(n))
    x[block // 2::997] *= 50.0
    q, c = pac.quantize_absmax(x.cuda(), block)
    out = pac.dequantize_absmax(q, c, block)
    torch.cuda.synchronize()
    rq, rc = qo.quantize_absmax(x.numpy(), block)
    assert np.array_equal(q.cpu().numpy(), rq)
    assert np.array_equal(c.cpu().numpy().view(np.uint32), rc.view(np.uint32))
    assert np.array_equal(out.cpu().numpy().view(np.uint32), qo.dequantize_absmax(rq, rc, block).view(np.uint32))
