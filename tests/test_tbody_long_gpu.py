"""Transformer-body adapters whose sequences take several rounds of keys per warp, and widths at the edges of the kernels' variants, against the oracle.
Tolerance 1e-4 as in test_tbody_tiles_gpu.py."""
import numpy as np
import pytest

import pac_inputs as pi
from oracle import tbody_oracle as tb
from tests.common import rel_l2
from tests.test_tbody_gpu import block_names, make_ctx, random_flat

pytestmark = pytest.mark.gpu


def spec(name, **kw):
    return pi.CacheSpec(name, **{**dict(N=3, L=2, S=40, d=64, dtype="f32", r=16, n_out=3, B=2), **kw})


CASES = [
    (spec("sixteen_warps_of_keys", S=512, B=1, L=1), 2, 32),
    (spec("two_rounds", S=530, B=1, L=1), 2, 32),
    (spec("three_rounds", S=1100, B=1, L=1, N=2), 1, 32),
    (spec("first_key_of_a_second_round", S=513, B=1, L=2, r=18), 3, 40),      # two heads at a time, the last one alone
    (spec("last_two_heads_at_a_time", S=768, B=1, L=1, r=32), 4, 64),
    (spec("first_one_head_at_a_time", S=769, B=1, L=1, r=12), 3, 24),
    (spec("two_rounds_three_columns", S=521, B=1, L=2, r=70), 2, 140),
    (spec("two_rounds_six_columns", S=600, B=1, L=1, r=98), 2, 98),
    (spec("two_rounds_short_ring", S=530, B=1, L=1, r=8), 1, 1100),           # a wide feed-forward layer leaves room for fewer weight units
    (spec("r_64", r=64), 4, 256),                          # widest of two columns per lane
    (spec("r_66", r=66), 2, 130),                          # three columns per lane; more than eight tiles: sums not cut along K
    (spec("r_96_seven_heads_of_keys", r=96, S=70), 8, 384),
    (spec("r_98", r=98, S=17), 7, 98),
    (spec("ffn_beyond_eight_tiles_per_warp", r=8, S=20), 2, 1100),
]


@pytest.mark.parametrize("sp,heads,f", CASES, ids=[c[0].name for c in CASES])
def test_loss_and_gradients_match_oracle(sp, heads, f):
    ctx = make_ctx(sp, heads, f)
    flat = random_flat(sp, f, 3)
    ctx.set_params(flat)
    ids = [sp.N - 1, 0][:sp.B]
    H = pi.cache_samples(sp, 0, ids, "cpu").float().numpy()
    lab = pi.labels(sp, 0, "cpu").numpy().astype(np.int64)[ids]
    P, T = tb.unflatten(flat, sp.L, sp.d, sp.r, sp.n_out, f)
    loss = ctx.train_step(ids)
    g = ctx.get_grads()
    ref_loss, (rg, rG), _ = tb.loss_and_grads_cls(P, T, H, lab, heads)
    ref = tb.flatten(rg, rG)
    assert abs(loss - ref_loss) <= 1e-4 * abs(ref_loss)
    o = 0
    for name, size in block_names(sp, f):
        assert rel_l2(g[o:o + size], ref[o:o + size]) < 1e-4, (name, rel_l2(g[o:o + size], ref[o:o + size]))
        o += size
    assert o == g.size
    ctx.close()
