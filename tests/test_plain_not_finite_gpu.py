"""The plain path's products on operands that bf16 terms cannot carry: an infinity in the cache stays one, and finite values beyond the largest
bf16 (3.39e38) multiply like any other.  The oracle says what fp32 arithmetic gives; tolerance 1e-4 as for every fp32 path."""
import numpy as np
import pytest
import torch

import pac_inputs as pi
from oracle import pac_oracle as po
from tests.common import Case, block_slices, rel_l2

pytestmark = pytest.mark.gpu


def spec(name, **kw):
    return pi.CacheSpec(name, **{**dict(N=6, L=3, S=20, d=128, dtype="f32", r=16, n_out=3, B=3), **kw})


SPECS = [spec("whole_tiles"), spec("shared_tiles", d=450, r=20), spec("row_slices", S=160, d=80, L=2, B=6, N=8, r=72)]
AT = (1, 0, 3, 5)                           # sample, layer, token and column of the value


def make(sp, value):
    case = Case(sp)
    case.cache[AT] = value
    case.cache_np[AT] = value
    return case, case.context()


@pytest.mark.parametrize("sp", SPECS, ids=lambda s: s.name)
def test_large_finite_value(sp):
    case, ctx = make(sp, 3.4e38)
    flat = pi.random_params(sp, 3)
    w = flat[:sp.L * sp.d * sp.r].reshape(sp.L, sp.d, sp.r)
    w[AT[1], AT[3]] *= 1e-37                # |u| stays around one
    ctx.set_params(flat)
    ids = [1, 4, 0, 2, 3, 5][:sp.B]
    loss = ctx.train_step(ids)
    g = ctx.get_grads().astype(np.float64)
    ref_loss, ref_g, _ = case.oracle_loss_grads(flat, ids)
    ref = po.flatten(ref_g).astype(np.float64)
    assert abs(loss - ref_loss) <= 1e-4 * abs(ref_loss)
    assert np.isfinite(ref).all() and np.isfinite(g).all()
    big = np.abs(ref) > 1e30                # the row of dW_down that belongs to the value; the rest by itself
    assert big.any() and rel_l2(g[big], ref[big]) < 1e-4
    g[big] = ref[big] = 0
    for name, sl in block_slices(sp).items():
        assert rel_l2(g[sl], ref[sl]) < 1e-4, name
    ctx.close()


@pytest.mark.parametrize("sp", SPECS[:2], ids=lambda s: s.name)
def test_infinity_reaches_the_logits(sp):
    case, ctx = make(sp, np.inf)
    flat = pi.random_params(sp, 3)
    sl = block_slices(sp)
    flat[:sp.L * sp.d * sp.r].reshape(sp.L, sp.d, sp.r)[AT[1], AT[3]] = 0.5
    for name in ("W_up", "W_head"):
        flat[sl[name]] = np.abs(flat[sl[name]])
    flat[sl["lam"]] = 0.5
    ctx.set_params(flat)
    ids = [4, 1, 0]
    out = torch.zeros((3, sp.n_out), device="cuda")
    ctx.eval_logits(ids, out)
    ctx.sync()
    got = out.cpu().numpy()
    ref = po.eval_logits(case.oracle_params(flat), case.H(ids))
    assert np.isposinf(ref[1]).all() and np.isposinf(got[1]).all()
    assert rel_l2(got[[0, 2]], ref[[0, 2]]) < 1e-4
    ctx.close()
