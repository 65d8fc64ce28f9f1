"""The fp32-precision products of the plain path (u = h W_down, dW_down = h^T du, dW_up of the LM head) at the edges
of their tiles, against the oracle.

Tolerance 1e-4 as for every fp32 path: sums of up to 903 fp32 products in another order differ by about
903^0.5 * 2^-24 = 1.8e-6 relative to the sum's size."""
import numpy as np
import pytest

import pac_inputs as pi
from oracle import pac_oracle as po
from tests.common import Case, block_slices, rel_l2

pytestmark = pytest.mark.gpu


def spec(name, **kw):
    base = dict(N=12, L=3, S=40, d=128, dtype="f32", r=32, n_out=3, B=4)
    return pi.CacheSpec(name, **{**base, **kw})


SPECS = [
    spec("r_below_16", r=7, d=97),                                  # one narrow tile, rows that start off a vector boundary
    spec("r_16", r=16, S=33),
    spec("r_17", r=17, d=130, dtype="bf16"),                        # first width of the next tile
    spec("r_65", r=65, S=65, d=100),
    spec("r_96", r=96, d=68, S=31),
    spec("r_97", r=97, d=192, dtype="bf16"),
    spec("r_129", r=129, d=72, S=34),                               # first width of two tiles
    spec("r_256", r=256, d=136, S=20, L=2),                         # two full tiles
    spec("one_row", r=20, S=1, B=1, d=64),
    spec("row_slices", r=16, S=160, B=6, d=80, L=2),                # the reduction over rows cut into slices
    spec("row_slices_odd", r=24, S=171, B=6, d=132, L=2, dtype="bf16"),
    spec("few_shared_tiles", d=450, r=20, S=37),                    # every tile shared by several CTAs, the last slice of the reduction short
    spec("last_wave_shared", d=330, r=72, L=24, S=129, B=7),        # more tiles than SMs: only those of the last wave are shared
    spec("last_wave_shared_bf16", d=401, r=130, L=11, S=129, B=7, dtype="bf16"),
    # LM head: dW_up in row slices, its gradient block off a 16-byte boundary (L = 3)
    spec("lm_slices", L=3, S=160, d=64, r=16, n_out=96, B=4, N=6, dtype="bf16", head="lm"),
]


@pytest.mark.parametrize("sp", SPECS, ids=lambda s: s.name)
def test_loss_and_gradients_match_oracle(sp):
    case = Case(sp)
    ctx = case.context(force_simt=True)
    flat = pi.random_params(sp, 3)
    ctx.set_params(flat)
    ids = [(5 * i + 1) % sp.N for i in range(sp.B)]
    loss = ctx.train_step(ids)
    g = ctx.get_grads()
    ref_loss, ref_g, _ = case.oracle_loss_grads(flat, ids)
    ref = po.flatten(ref_g)
    assert abs(loss - ref_loss) <= 1e-4 * abs(ref_loss)
    for name, sl in block_slices(sp).items():
        assert np.linalg.norm(ref[sl]) > 0 and rel_l2(g[sl], ref[sl]) < 1e-4, (name, rel_l2(g[sl], ref[sl]))
    ctx.close()
