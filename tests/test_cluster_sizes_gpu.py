"""The one-launch forward at every cluster size its rule can choose (by batch and sequence length), against the oracle: loss, every
gradient block, evaluation.  Tolerances as for the other bf16 tests (a gate whose argument is within 1e-6 of zero may
open on one side only)."""
import numpy as np
import pytest
import torch

import pac_inputs as pi
from oracle import pac_oracle as po
from tests.common import Case, block_slices, rel_l2

pytestmark = pytest.mark.gpu


def spec(name, **kw):
    base = dict(N=80, L=12, S=30, d=192, dtype="bf16", r=64, n_out=3, B=4)
    return pi.CacheSpec(name, **{**base, **kw})


SPECS = [
    spec("one_layer_per_cta", B=1),                     # clusters beyond eight CTAs
    spec("more_ctas_than_tokens", B=2, S=5, L=16, r=16),
    spec("odd_cluster", B=20, L=11, S=33),              # cluster size not a power of two, layers not a multiple of it
    spec("two_per_sample", B=60, L=12, S=20, r=32),
    spec("single_cta", B=70, L=7, S=19, r=48),
    spec("one_layer", B=9, L=1, S=40),
    spec("full_tile", B=3, L=24, S=128, d=136),
]


@pytest.mark.parametrize("sp", SPECS, ids=lambda s: s.name)
def test_loss_gradients_and_eval_match_oracle(sp):
    case = Case(sp)
    ctx = case.context(max_batch=sp.B)
    assert ctx.kernel_path() == "tensor+fused_forward"
    flat = pi.random_params(sp, 3)
    ctx.set_params(flat)
    for B in {sp.B, max(1, sp.B // 3)}:                 # a smaller batch may take another cluster size
        ids = [(7 * i + 1) % sp.N for i in range(B)]
        loss = ctx.train_step(ids)
        g = ctx.get_grads()
        ref_loss, ref_g, _ = case.oracle_loss_grads(flat, ids)
        ref = po.flatten(ref_g)
        assert abs(loss - ref_loss) <= 1e-3 * abs(ref_loss)
        for name, sl in block_slices(sp).items():
            assert rel_l2(g[sl], ref[sl]) < 2e-2, (name, B, rel_l2(g[sl], ref[sl]))
        out = torch.zeros((B, sp.n_out), dtype=torch.float32, device="cuda")
        ctx.eval_logits(ids, out)
        ctx.sync()
        assert rel_l2(out.cpu().numpy(), po.eval_logits(case.oracle_params(flat), case.H(ids), 0, None)) < 1e-3
    ctx.close()
