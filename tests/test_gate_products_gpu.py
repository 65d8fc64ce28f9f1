"""dW_down of wide classifier adapters on long samples, formed from the gates alone, sample by sample, at the edges of its tiles and of its row splits.

Against 64 bits, identity bodies and ReLU: bounds of test_gradient_precision_gpu.py (W_down in two bf16 terms, 2^-17; ReLU gates within that of zero may
open on one side only, so there the fp32 oracle with the tensor path's own bound of 2e-2 stands in)."""
import numpy as np
import pytest
import torch

import pac_inputs as pi
from paper_2408_10746_b200.binding import second_pass_plan
from oracle import pac_oracle as po
from tests.common import Case, block_slices, rel_l2
from tests.test_gradient_precision_gpu import bf16, errors

pytestmark = pytest.mark.gpu

SPECS = [
    bf16("third_tile_of_one_token", S=129, r=128, L=2),
    bf16("two_full_tiles_keep_two_terms", S=128, r=128, L=2),
    bf16("one_column_block", S=200, r=80, d=136, L=3),              # d below two blocks, ragged; the second half of the columns 16 wide
    bf16("one_sample", S=192, r=96, B=1),
    bf16("splits_cut_samples", S=300, r=112, B=7, L=5, d=520),
    bf16("deep", S=140, r=128, L=130, d=64, B=2, N=4),              # layer numbers of eight bits
]
# Sizes of which the launch takes the gates kernel (three row tiles to a CTA and more)
LONG = [
    bf16("third_tile_of_one_token_long", S=129, r=128, L=2, B=8),
    bf16("one_column_block_long", S=200, r=80, d=136, L=3, B=6),
    bf16("one_sample_long", S=1540, r=96, B=1, N=3),
    bf16("splits_cut_samples_long", S=300, r=112, B=8, L=5, d=520),
    bf16("deep_long", S=140, r=128, L=130, d=64, B=4, N=4),
    bf16("several_waves", S=129, r=80, L=24, d=1024, B=24, N=24),
]


def gates_of(sp, sms):
    return second_pass_plan(sp.L, sp.S, sp.d, sp.r, sp.B, sp.B, sms, 232448)[2]


def test_long_sizes_take_the_gates():
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for sp in LONG:
        assert gates_of(sp, sms), sp.name
    assert not gates_of(bf16("several_waves_short", S=129, r=80, L=24, d=1024, B=23), sms)


@pytest.mark.parametrize("sp", SPECS + LONG, ids=lambda s: s.name)
def test_gradients_against_64_bits(sp):
    worst, path = errors(sp, act=1, seeds=(3,))
    assert path.startswith("tensor")
    assert worst["lam"] < 1e-4 and worst["W_down"] < 2e-5, worst


@pytest.mark.parametrize("sp", SPECS[:5] + LONG[:4], ids=lambda s: s.name)
def test_relu_gates(sp):
    case = Case(sp)
    ctx = case.context()
    flat = pi.random_params(sp, 5)
    ctx.set_params(flat)
    ids = [(3 * i + 2) % sp.N for i in range(sp.B)]
    loss = ctx.train_step(ids)
    g = ctx.get_grads()
    ref_loss, ref, _ = case.oracle_loss_grads(flat, ids)
    ref = po.flatten(ref)
    assert abs(loss - ref_loss) <= 2e-2 * abs(ref_loss)
    for name, sl in block_slices(sp).items():
        assert rel_l2(g[sl], ref[sl]) < 2e-2, (name, rel_l2(g[sl], ref[sl]))
    ctx.close()
