"""Transformer-body adapters on bf16 caches, whose passes over the cache run at fp32 precision whatever the body's width: loss, every
gradient block and evaluation at the widths and row counts where those products' tiles end, and a trajectory through both forms of the update.

Tolerance 1e-4 as in test_tbody_tiles_gpu.py."""
import numpy as np
import pytest

import pac_inputs as pi
from oracle import pac_oracle as po
from oracle import tbody_oracle as tb
from tests.common import rel_l2
from tests.test_tbody_gpu import make_ctx, random_flat
from tests.test_tbody_tiles_gpu import test_loss_gradients_and_eval_match_oracle as check

pytestmark = pytest.mark.gpu


def spec(name, **kw):
    base = dict(N=6, L=2, S=16, d=64, dtype="bf16", r=16, n_out=3, B=3)
    return pi.CacheSpec(name, **{**base, **kw})


CASES = [                                                            # spec, heads, ffn width
    (spec("r_16"), 2, 64), (spec("r_64", r=64, S=65, d=264), 4, 128), (spec("r_80", r=80, S=129, d=200, B=2), 4, 96),
    (spec("r_128", r=128, S=65, d=1024, B=2), 8, 128), (spec("r_192", r=192, S=33, d=136, B=2), 3, 64), (spec("d_off_8", r=24, S=37, d=100), 4, 48),
]


@pytest.mark.parametrize("sp,heads,f", CASES, ids=[c[0].name for c in CASES])
def test_loss_gradients_and_eval(sp, heads, f):
    check(sp, heads, f)


@pytest.mark.parametrize("fused", [True, False], ids=["epoch", "separate"])
def test_ten_steps_follow_the_oracle(fused):
    """Batches smaller than max_batch at the end; parameters after every kind of update feed the next step's products."""
    import paper_2408_10746_b200 as pac
    sp, heads, f = spec("steps", S=20, d=72, r=32, N=10, B=4), 4, 64
    ctx = make_ctx(sp, heads, f)
    flat = random_flat(sp, f, 4)
    ctx.set_params(flat)
    hp = po.AdamW()
    dev_hp = pac.AdamW(hp.lr, hp.beta1, hp.beta2, hp.eps, hp.weight_decay)
    perm = np.concatenate([pi.epoch_permutation(sp.N, 2, epoch=e) for e in range(4)])
    batches = [perm[4 * s:4 * s + 4] for s in range(8)] + [perm[32:35], perm[35:37]]
    if fused:
        losses = list(ctx.train_epoch(perm[:32], 4, dev_hp)) + [ctx.train_epoch(b, len(b), dev_hp)[0] for b in batches[8:]]
    else:
        losses = []
        for b in batches:
            losses.append(ctx.train_step(b))
            ctx.adam_step(dev_hp)
    cache = pi.cache_full(sp, 0, "cpu").float().numpy()
    labels = pi.labels(sp, 0, "cpu").numpy().astype(np.int64)
    theta, m, v = flat.copy(), np.zeros_like(flat), np.zeros_like(flat)
    for s, ids in enumerate(batches):
        P, T = tb.unflatten(theta, sp.L, sp.d, sp.r, sp.n_out, f)
        loss, (rg, rG), _ = tb.loss_and_grads_cls(P, T, po.gather(cache, ids), labels[ids], heads)
        assert abs(losses[s] - loss) <= 1e-4 * abs(loss), s
        theta, m, v = po.adamw_step(theta, tb.flatten(rg, rG), m, v, s + 1, hp, tb.decay_mask(P, T).astype(np.float32))
    p = ctx.get_params()
    assert rel_l2(p, theta) < 1e-4 and rel_l2(p - flat, theta - flat) < 1e-2
    assert ctx.get_opt_state()[2] == 10
    ctx.close()
