"""Gradients against the oracle in 64 bits, at sizes where a shortened operand or a drifting accumulation shows.

bf16 caches (identity bodies, so that no gate flips): da_L and W_down enter the tensor-core products as two bf16 terms each, 2^-17 of a value at
worst and 2^-18 on average; dlambda is a sum of B S r products of either sign, a few times smaller than its terms: 1e-4.  One term is 2^-9.
fp32 caches: sums of at most 1024 products rounded to 24 bits one by one differ by about 1024^0.5 * 2^-25 = 1e-6; a chain of
288 additions cut instead of rounded is off by 3e-6 to 5e-6."""
import numpy as np
import pytest

import pac_inputs as pi
from oracle import pac_oracle as po
from oracle import tbody_oracle as tb
from tests.common import Case, block_slices, rel_l2
from tests.test_tbody_gpu import make_ctx, random_flat

pytestmark = pytest.mark.gpu


def errors(sp, act, force_simt=False, seeds=(3, 4, 5)):
    case = Case(sp)
    ctx = case.context(act=act, force_simt=force_simt)
    worst = {}
    for seed in seeds:
        flat = pi.random_params(sp, seed)
        ctx.set_params(flat)
        ids = [(3 * i + seed) % sp.N for i in range(sp.B)]
        ctx.train_step(ids)
        g = ctx.get_grads()
        ref = po.flatten(case.oracle_loss_grads(flat, ids, act, dtype=np.float64)[1])
        for name, sl in block_slices(sp).items():
            worst[name] = max(worst.get(name, 0.0), rel_l2(g[sl], ref[sl]))
    path = ctx.kernel_path()
    ctx.close()
    return worst, path


def bf16(name, **kw):
    return pi.CacheSpec(name, **{**dict(N=16, L=4, S=64, d=256, dtype="bf16", r=64, n_out=3, B=4), **kw})


@pytest.mark.parametrize("sp", [
    bf16("r_64"), bf16("r_80_one_sample", r=80, B=1, S=40, d=128), bf16("r_96_short", r=96, S=30), bf16("r_128", r=128), bf16("r_128_many", r=128, B=16),
    bf16("r_128_chain", r=128, S=256, B=8, L=3), bf16("r_192", r=192), bf16("r_256_one_sample", r=256, B=1, S=32),
], ids=lambda s: s.name)
def test_tensor_path_keeps_the_bits_of_da(sp):
    worst, path = errors(sp, act=1)
    assert path.startswith("tensor")
    assert worst["lam"] < 1e-4 and worst["W_down"] < 2e-5, worst


def f32(name, **kw):
    return bf16(name, **{**dict(dtype="f32", L=4, S=128, d=768, B=8, N=12), **kw})


@pytest.mark.parametrize("sp", [
    f32("d_768"), f32("r_128_wide", d=1024, r=128), f32("r_16", r=16, d=512, S=64), f32("two_tiles_d_2048", d=2048, r=144, S=64, B=4, L=2),
    f32("bf16_cache", dtype="bf16", r=24),
], ids=lambda s: s.name)
def test_plain_products_round_like_fp32(sp):
    worst, _ = errors(sp, act=1, force_simt=True)
    for name in ("W_down", "W_up", "lam"):
        assert worst[name] < (1e-6 if name != "lam" else 4e-6), worst            # (lam: a sum of both signs, see above)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_transformer_body_rounds_like_fp32(dtype):
    """1024 rows and d = 1024: long reductions in both passes over the cache (those of the layers between them are shorter)."""
    sp, heads, f = bf16("tb", dtype=dtype, L=2, S=256, d=1024, r=16, B=4, N=6), 2, 32
    ctx = make_ctx(sp, heads, f)
    ids = [5, 0, 3, 3]
    H = pi.cache_samples(sp, 0, ids, "cpu").double().numpy()
    lab = pi.labels(sp, 0, "cpu").numpy().astype(np.int64)[ids]
    for seed in (3, 4):
        flat = random_flat(sp, f, seed)
        ctx.set_params(flat)
        ctx.train_step(ids)
        g = ctx.get_grads()
        P, T = tb.unflatten(flat.astype(np.float64), sp.L, sp.d, sp.r, sp.n_out, f)
        ref = tb.flatten(*tb.loss_and_grads_cls(P, T, H, lab, heads)[1])
        body = sum(s.stop - s.start for s in block_slices(sp).values())
        assert rel_l2(g[body:], ref[body:]) < 1.5e-6
        for name, sl in block_slices(sp).items():
            assert rel_l2(g[sl], ref[sl]) < (4e-6 if name == "lam" else 1.5e-6), (name, seed, rel_l2(g[sl], ref[sl]))
    ctx.close()


def test_wide_transformer_body_forward_rounds_like_fp32():
    """r = 128 on a bf16 cache: W_up's gradient is a_L^T dy, with nothing of the reverse pass in it (a gate that flips there moves other
    blocks by single elements)."""
    sp, heads, f = bf16("tb_wide", L=3, S=128, d=1024, r=128, B=4, N=6), 8, 256
    ctx = make_ctx(sp, heads, f)
    ids = [5, 0, 3, 1]
    H = pi.cache_samples(sp, 0, ids, "cpu").double().numpy()
    lab = pi.labels(sp, 0, "cpu").numpy().astype(np.int64)[ids]
    flat = random_flat(sp, f, 3)
    ctx.set_params(flat)
    ctx.train_step(ids)
    g = ctx.get_grads()
    P, T = tb.unflatten(flat.astype(np.float64), sp.L, sp.d, sp.r, sp.n_out, f)
    ref = tb.flatten(*tb.loss_and_grads_cls(P, T, H, lab, heads)[1])
    sl = block_slices(sp)["W_up"]
    assert rel_l2(g[sl], ref[sl]) < 1e-6, rel_l2(g[sl], ref[sl])
    ctx.close()
