"""How the tiles of the fp32-precision u = h W_down are dealt to CTAs: every stage of every tile is taken exactly once and the workspace suffices; and the sizes
of the numeric tests of both cache passes reach the forms that they are about."""
import pytest

from paper_2408_10746_b200.binding import rows_plan, second_pass_plan
from tests.test_gate_products_gpu import LONG, gates_of
from tests.test_plain_products_gpu import PLANS, plan_of

SMS = 148


def tile_columns(r):
    tiles = -(-r // 128)
    return -(-(-(-r // tiles)) // 16) * 16


@pytest.mark.parametrize("f32,aligned", [(True, True), (True, False), (False, True), (False, False)])
def test_plans_cover_every_stage_once(f32, aligned):
    shared = 0
    for sms in (148, 132, 20):
        for d in (1, 64, 65, 255, 320, 450, 768, 800, 1024, 2048, 4096):
            stages = -(-d // 64)
            for r in (8, 16, 40, 64, 80, 128, 200):
                for tiles in list(range(1, 40)) + list(range(sms - 3, sms + 60)) + list(range(2 * sms - 3, 2 * sms + 40)) + [3 * sms, 4 * sms + 7]:
                    teams, whole, parts, per = rows_plan(tiles, d, r, f32, aligned, sms)
                    slots = sms * (2 if teams == 1 else 1)
                    assert teams in (1, 2) and 0 <= whole <= tiles
                    if teams == 1:                                       # accumulators of two CTAs in 512 columns
                        accs = max(1, -(-4 * stages // 24))
                        assert (accs + 1) * tile_columns(r) <= 256 and tiles > sms
                    if whole < tiles:
                        shared += 1
                        assert whole % slots == 0 and parts > 1 and per * parts >= stages > per * (parts - 1)
                        assert (tiles - whole) * parts <= slots and stages - per >= 4      # ws: 2 sms tiles
                    else:
                        assert parts == 1
    assert shared > 1000


@pytest.mark.parametrize("sp,teams,mixed", PLANS, ids=[p[0].name for p in PLANS])
def test_sizes_reach_their_forms(sp, teams, mixed):
    got, whole, parts, _ = plan_of(sp, SMS)
    assert got == teams and (whole > 0 and parts > 1) == mixed


def test_gates_alone_only_where_streams_are_long():
    assert all(gates_of(sp, SMS) for sp in LONG)
    for r, S, B, L, d, want in [(128, 256, 64, 24, 1024, True), (64, 256, 64, 24, 1024, False), (144, 256, 64, 24, 1024, False), (128, 128, 64, 24, 1024, False),
                                (96, 129, 2, 7, 768, False), (96, 160, 4, 12, 768, True), (96, 160, 8, 24, 1024, False), (112, 160, 8, 24, 1024, True), (80, 129, 23, 24, 1024, False)]:
        assert second_pass_plan(L, S, d, r, B, B, SMS, 232448)[2] == want, (r, S, B, L, d)
    # the plan is made for the largest batch, the form chosen for the one that runs
    assert second_pass_plan(12, 160, 768, 96, 16, 16, SMS, 232448)[2] and not second_pass_plan(12, 160, 768, 96, 16, 1, SMS, 232448)[2]
