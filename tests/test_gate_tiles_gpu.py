"""The second pass on the tensor path builds du from gate bytes and da_L, and lambda's gradient comes from <D, W_down>: at the edges of
its tiles, term counts, row splits and of both finalisations, against the oracle.

Tolerance 2e-2 per gradient block as for the other bf16 tests; what two bf16 terms of da give without flipped gates is bounded in
test_gradient_precision_gpu.py."""
import numpy as np
import pytest

import pac_inputs as pi
from oracle import pac_oracle as po
from tests.common import Case, block_slices, rel_l2

pytestmark = pytest.mark.gpu


def spec(name, **kw):
    base = dict(N=10, L=3, S=40, d=128, dtype="bf16", r=32, n_out=3, B=4)
    return pi.CacheSpec(name, **{**base, **kw})


SPECS = [
    spec("one_token", S=1, r=16, d=64, B=3),
    spec("r_64_two_terms", r=64, S=65, d=264),              # widest adapter of the two-term tiles, two chunks of d and a remainder
    spec("r_80", r=80, S=129, d=136),
    spec("r_128", r=128, S=63, d=256),
    spec("r_144_wide", r=144, S=64, d=128),                 # four column blocks, the third partly filled, the fourth empty
    spec("r_256", r=256, S=33, d=128, L=2),
    spec("many_splits", L=1, d=64, S=100, B=9, N=20),       # eight row splits; a batch of one leaves all but two without rows
    spec("long_sample", S=300, r=48, d=192, L=4, B=2),      # several row tiles per sample
    spec("many_classes", n_out=40, S=37),                   # head outside the fused kernels: gradients from gated_grads_kernel
    spec("many_layers", L=34, S=20, d=64, r=16),
    spec("lm_token_da", head="lm", n_out=96, r=64, S=30, L=3, d=64),
    spec("lm_wide_two_terms", head="lm", n_out=64, r=144, S=65, L=2, d=128, B=2),
]


@pytest.mark.parametrize("act", [0, 1], ids=["relu", "identity"])
@pytest.mark.parametrize("sp", SPECS, ids=lambda s: s.name)
def test_gradients_match_oracle(sp, act):
    case = Case(sp)
    ctx = case.context(max_batch=sp.B, act=act)
    assert ctx.kernel_path().startswith("tensor")
    flat = pi.random_params(sp, 3)
    for edge in (False, True):
        if edge:                                            # lambda exactly 1 cuts off the layers below, exactly 0 the layer itself
            lam = block_slices(sp)["lam"]
            flat[lam.start + sp.L // 2] = 1.0
            flat[lam.stop - 1] = 0.0
        ctx.set_params(flat)
        for B in (sp.B, 1):
            ids = [(3 * i + 1) % sp.N for i in range(B)]
            loss = ctx.train_step(ids)
            g = ctx.get_grads()
            ref_loss, ref_g, _ = case.oracle_loss_grads(flat, ids, act)
            ref = po.flatten(ref_g)
            assert abs(loss - ref_loss) <= 1e-3 * abs(ref_loss)
            for name, sl in block_slices(sp).items():
                assert rel_l2(g[sl], ref[sl]) < 2e-2, (name, B, edge, rel_l2(g[sl], ref[sl]))
    ctx.close()
