"""AdamW updates where a layer of W_down is not a multiple of four elements but all layers together are (the finalisation then takes them as one),
and where neither is: ten steps through the fused and the separate update against the oracle's, fp32 tolerances."""
import numpy as np
import pytest

import pac_inputs as pi
from oracle import pac_oracle as po
from tests.common import Case, rel_l2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fused", [True, False], ids=["epoch", "separate"])
@pytest.mark.parametrize("L", [4, 3])
def test_ten_steps(L, fused):
    import paper_2408_10746_b200 as pac
    sp = pi.CacheSpec(f"ragged_{L}", N=10, L=L, S=9, d=97, dtype="f32", r=7, n_out=3, B=4)
    case = Case(sp)
    ctx = case.context()
    flat = pi.random_params(sp, 3)
    ctx.set_params(flat)
    hp = po.AdamW()
    dev_hp = pac.AdamW(hp.lr, hp.beta1, hp.beta2, hp.eps, hp.weight_decay)
    perm = np.concatenate([pi.epoch_permutation(sp.N, 2, epoch=e) for e in range(4)])[:40]
    batches = perm.reshape(10, 4)
    if fused:
        losses = list(ctx.train_epoch(perm, 4, dev_hp))
    else:
        losses = []
        for b in batches:
            losses.append(ctx.train_step(b))
            ctx.adam_step(dev_hp)
    tr, _ = case.oracle_trainer(flat, 0, hp)
    for b, loss in zip(batches, losses):
        ref = tr.train_step(b)
        tr.adam_step()
        assert abs(loss - ref) <= 1e-4 * abs(ref)
    p, ref_p = ctx.get_params(), po.flatten(tr.P)
    assert rel_l2(p, ref_p) < 1e-4 and rel_l2(p - flat, ref_p - flat) < 1e-2
    ctx.close()
