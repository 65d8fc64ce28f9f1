"""The fp32-precision products of the plain path (u = h W_down, dW_down = h^T du, dW_up of the LM head) at the edges
of their tiles, against the oracle.

Tolerance 1e-4 as for every fp32 path: sums of up to 903 fp32 products in another order differ by about
903^0.5 * 2^-24 = 1.8e-6 relative to the sum's size."""
import numpy as np
import pytest
import torch

import pac_inputs as pi
from paper_2408_10746_b200.binding import rows_plan
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

# u = h W_down in each form of its plan (producer teams per CTA; whether whole tiles and shared ones of the last wave occur together)
PLANS = [
    (spec("one_team_unshared", d=330, r=72, L=24, S=129, B=7), 1, False),
    (spec("one_team_last_wave_shared", d=330, r=72, L=40, S=129, B=7), 1, True),
    (spec("one_team_last_wave_shared_bf16", d=328, r=130, L=20, S=129, B=7, dtype="bf16"), 1, True),
    (spec("accumulators_of_two_ctas_do_not_fit", d=450, r=128, L=22, S=129, B=7), 2, True),
    (spec("long_reductions_just_over_a_wave", d=800, r=16, L=19, S=129, B=7), 2, True),
    (spec("bf16_off_a_boundary", d=515, r=24, L=20, S=129, B=7, dtype="bf16"), 2, True),
    (spec("bf16_off_a_boundary_short", d=255, r=24, L=20, S=129, B=7, dtype="bf16"), 1, False),
]


def plan_of(sp, sms):
    bf = sp.dtype == "bf16"
    tiles = sp.L * -(-sp.B * sp.S // 128) * -(-sp.r // 128)
    return rows_plan(tiles, sp.d, sp.r, not bf, sp.d * (2 if bf else 4) % 16 == 0, sms)


def check(sp, act=0):
    case = Case(sp)
    ctx = case.context(act=act, force_simt=True)
    flat = pi.random_params(sp, 3)
    ctx.set_params(flat)
    ids = [(5 * i + 1) % sp.N for i in range(sp.B)]
    loss = ctx.train_step(ids)
    g = ctx.get_grads()
    ref_loss, ref_g, _ = case.oracle_loss_grads(flat, ids, act)
    ref = po.flatten(ref_g)
    assert abs(loss - ref_loss) <= 1e-4 * abs(ref_loss)
    for name, sl in block_slices(sp).items():
        assert np.linalg.norm(ref[sl]) > 0 and rel_l2(g[sl], ref[sl]) < 1e-4, (name, rel_l2(g[sl], ref[sl]))
    ctx.close()


@pytest.mark.parametrize("sp,teams,mixed", PLANS, ids=[p[0].name for p in PLANS])
def test_every_form_of_the_plan(sp, teams, mixed):
    got, whole, parts, _ = plan_of(sp, torch.cuda.get_device_properties(0).multi_processor_count)
    assert got == teams and (whole > 0 and parts > 1) == mixed
    check(sp, act=1)                # identity bodies: no gate of two million decides differently for a sum in another order


@pytest.mark.parametrize("sp", SPECS, ids=lambda s: s.name)
def test_loss_and_gradients_match_oracle(sp):
    check(sp)
