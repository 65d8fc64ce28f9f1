"""Transformer-body adapters at the edges of the tiles their kernels work in (16 tokens, 16 x 8 weight tiles, heads of any
width) against the oracle: loss, every gradient block, evaluation.

Tolerance 1e-4 as in test_tbody_gpu.py: products are formed at fp32 precision (operands as exact sums of three bf16 terms,
dropped terms below 2^-25), sums of at most 512 of them differ by about 512^0.5 * 2^-24 = 1.3e-6."""
import numpy as np
import pytest
import torch

import pac_inputs as pi
from oracle import tbody_oracle as tb
from tests.common import rel_l2
from tests.test_tbody_gpu import block_names, make_ctx, random_flat

pytestmark = pytest.mark.gpu


def spec(name, **kw):
    base = dict(N=6, L=2, S=16, d=64, dtype="f32", r=16, n_out=3, B=3)
    return pi.CacheSpec(name, **{**base, **kw})


CASES = [                                                            # spec, heads, ffn width
    (spec("tile", d=96), 1, 64),                                     # exactly one tile of tokens, keys and head width
    (spec("head_6_of_18", S=37, r=18, d=72), 3, 50),                 # heads narrower than a tile, last tile of five tokens
    (spec("odd_widths", S=33, r=21, d=80, dtype="bf16"), 3, 45),     # odd head and ffn widths: no paired loads
    (spec("head_40", S=129, r=80, B=2), 2, 320),                     # a head of two and a half k steps, keys one past eight tiles
    (spec("wide", S=20, r=130, B=2), 1, 512),                        # r beyond four columns per lane, one head
    (spec("many_heads", S=70, r=64, B=2), 16, 256),                  # more head tiles than warps
    (spec("long", S=300, r=32, B=1, N=2), 8, 128),                   # head groups: not all score rows fit at once
    (spec("beyond", S=9, r=200, B=2, L=1), 4, 40),                   # wider than the fused kernels take
]


@pytest.mark.parametrize("sp,heads,f", CASES, ids=[c[0].name for c in CASES])
def test_loss_gradients_and_eval_match_oracle(sp, heads, f):
    ctx = make_ctx(sp, heads, f)
    L, d, r, C = sp.L, sp.d, sp.r, sp.n_out
    flat = random_flat(sp, f, 3)
    ctx.set_params(flat)
    ids = [sp.N - 1, 0, 0][:sp.B]
    H = pi.cache_samples(sp, 0, ids, "cpu").float().numpy()
    lab = pi.labels(sp, 0, "cpu").numpy().astype(np.int64)[ids]
    P, T = tb.unflatten(flat, L, d, r, C, f)
    out = torch.zeros((len(ids), C), dtype=torch.float32, device="cuda")
    ctx.eval_logits(ids, out)
    ctx.sync()
    assert rel_l2(out.cpu().numpy(), tb.eval_logits(P, T, H, heads)) < 1e-4
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
