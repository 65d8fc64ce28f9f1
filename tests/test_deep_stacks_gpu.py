"""Stacks of more layers than seven bits count, on the tensor-core path up to 255 of them (gate bytes hold a layer number): every layer's
gradient against the oracle, 2e-2 per block as for the other bf16 tests."""
import numpy as np
import pytest

import pac_inputs as pi
from oracle import pac_oracle as po
from tests.common import Case, block_slices, rel_l2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("act", [0, 1], ids=["relu", "identity"])
@pytest.mark.parametrize("L,r,head", [(127, 16, "cls"), (128, 16, "cls"), (200, 96, "cls"), (255, 16, "cls"), (255, 32, "lm"), (256, 16, "cls")])
def test_every_layer_matches_oracle(L, r, head, act):
    sp = pi.CacheSpec(f"deep_{L}_{r}_{head}", N=4, L=L, S=35, d=64, dtype="bf16", r=r, n_out=3 if head == "cls" else 64, B=2, head=head)
    case = Case(sp)
    ctx = case.context(act=act)
    assert ctx.kernel_path() == ("tensor" if L < 256 else "simt")
    flat = pi.random_params(sp, 3)
    sl = block_slices(sp)
    flat[sl["lam"]] = np.linspace(0.01, 0.04, L)        # the lowest layer's share is still one in a few hundred, and gates close at every depth
    ctx.set_params(flat)
    loss = ctx.train_step([2, 1])
    g = ctx.get_grads()
    ref_loss, ref_g, _ = case.oracle_loss_grads(flat, [2, 1], act)
    ref = po.flatten(ref_g)
    assert abs(loss - ref_loss) <= 1e-3 * abs(ref_loss)
    for name, s in sl.items():
        assert rel_l2(g[s], ref[s]) < 2e-2, (name, rel_l2(g[s], ref[s]))
    W, R = (x[sl["W_down"]].reshape(L, -1) for x in (g, ref))
    size = np.linalg.norm(R, axis=1)                    # (few gates are open all the way down: layers below a thousandth of the largest count as that)
    off = np.linalg.norm(W - R, axis=1) / np.maximum(size, 1e-3 * size.max())
    assert off.max() < 2e-2, off.argmax()
    ctx.close()
