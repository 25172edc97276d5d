"""How the tensor-core scoring lays a problem out on the SMs, asked of the library without a GPU: the lines between the kernel's
forms, and what every layout has to keep."""
import random

import pytest

import paper_2509_05165_b200 as kvc

SMS = 148


def _desc(q_heads, kv_heads, d, n_ctx, w, layers, batch=1, after=False, **options):
    desc = kvc.kvc_desc_init(layers, batch, q_heads, kv_heads, d, n_ctx, w, kvc.BF16)
    if after:
        desc.q_pos0 = n_ctx
    for key, val in options.items():
        setattr(desc, key, val)
    return desc


@pytest.mark.parametrize("q_heads,kv_heads,d,n_ctx,w,layers,after,pairs", [
    # the window's mask, or a partial last tile, in one of few tiles: one row tile at a time whatever the window's length
    (64, 8, 128, 1787, 128, 36, False, 1),
    (128, 8, 128, 811, 128, 28, False, 1),
    (72, 8, 128, 1155, 500, 16, True, 1),
    (32, 8, 128, 3000, 500, 32, True, 1),
    (16, 8, 64, 3000, 150, 32, True, 1),
    (32, 8, 128, 6016, 64, 32, False, 1),        # one of 47 tiles ...
    (32, 8, 128, 6400, 64, 32, False, 2),        # ... and one of 50
    # whole tiles
    (32, 8, 128, 4096, 500, 32, True, 2),
    (32, 8, 128, 8192, 64, 32, False, 2),
    (28, 4, 128, 131072, 64, 28, False, 2),
    (32, 8, 64, 8192, 300, 16, True, 2),
    (56, 8, 128, 32768, 128, 16, False, 1),      # seven row tiles
    (36, 4, 128, 32768, 128, 16, False, 1),      # nine ...
    (12, 4, 64, 8192, 300, 16, True, 2),         # ... of heads of 64
    (28, 4, 128, 32768, 300, 4, True, 2),        # twenty-one
    (32, 8, 128, 32768, 49, 32, False, 1),       # a run-time window
])
def test_row_tiles_go_in_pairs_where_few_tiles_are_masked(q_heads, kv_heads, d, n_ctx, w, layers, after, pairs):
    assert kvc.kvc_debug_score_plan(_desc(q_heads, kv_heads, d, n_ctx, w, layers, after=after), SMS)["row_tiles"] == pairs


def test_value_norms_take_fewer_sms_from_dearer_scorings():
    """Of 148 SMs, at 16K tokens of the 8B shape: a scoring that takes k times as long per logit can spare about 1 / k as many."""
    def share(w, **options):
        return kvc.kvc_debug_score_plan(_desc(32, 8, 128, 16384, w, 32, value_norm=1, **options), SMS)["norm_ctas"]

    assert 40 <= share(32) <= 56
    assert 32 <= share(24) <= 44                                     # column blocks of a run-time window
    assert 28 <= share(32, agg_task=kvc.AGG_MEAN) <= 38              # a second exponential per logit
    assert 10 <= share(24, agg_task=kvc.AGG_MEAN) <= 18              # column by column
    assert share(32, agg_task=kvc.AGG_MEAN) < share(24) < share(32)
    # none where the norms are a small part and V would go through the L2 that the K tiles wait in
    assert kvc.kvc_debug_score_plan(_desc(32, 8, 128, 65536, 300, 3, after=True, value_norm=1), SMS)["norm_ctas"] == 0


def test_value_norms_leave_the_scoring_no_grid_that_meets_masked_tiles_all_the_time():
    """500 rows at the end of 4096 tokens: the last two of a unit's eight runs are masked; an odd grid meets all eight in turn."""
    plan = kvc.kvc_debug_score_plan(_desc(32, 8, 128, 4096, 500, 16, value_norm=1), SMS)
    assert plan["norm_ctas"] > 0 and plan["ctas"] % 2 == 1


def test_every_layout_fits_the_device():
    """All CTAs are resident at once (they wait for one another), no scoring CTA is without a run, and pass 1 may run ahead as far as
    the statistics of a unit are spread over the CTAs."""
    rng = random.Random(1)
    for _ in range(3000):
        kv_heads = rng.choice((1, 2, 8))
        group = rng.choice((1, 2, 4, 7, 9, 11))
        n_ctx, w = int(2 ** rng.uniform(0, 20)), rng.choice((1, 8, 24, 32, 64, 128, 130, 500, 3000))
        desc = _desc(group * kv_heads, kv_heads, rng.choice((64, 128)), n_ctx, w, rng.randint(1, 64), rng.choice((1, 3)),
                     after=rng.random() < 0.5, value_norm=rng.randrange(2), agg_task=rng.choice((kvc.AGG_MAX, kvc.AGG_MEAN)))
        sms = rng.choice((1, 2, 7, 132, 148))
        plan = kvc.kvc_debug_score_plan(desc, sms)
        assert 1 <= plan["ctas"] <= plan["runs"] and plan["norm_ctas"] >= 0
        assert plan["ctas"] + plan["norm_ctas"] <= sms
        tiles = -(-n_ctx // 128)
        run_tiles = max(4, -(-tiles // 255))
        runs_per_unit = -(-tiles // run_tiles)
        assert plan["lead"] >= (1 + (plan["ctas"] + runs_per_unit - 2) // plan["ctas"]) * run_tiles


def test_problems_of_the_cuda_core_kernels_have_no_such_layout():
    with pytest.raises(kvc.KvcError):
        kvc.kvc_debug_score_plan(kvc.kvc_desc_init(2, 1, 4, 2, 64, 512, 16, kvc.F32), SMS)
    with pytest.raises(kvc.KvcError):
        kvc.kvc_debug_score_plan(kvc.kvc_desc_init(2, 1, 4, 2, 64, 0, 16, kvc.BF16), SMS)
