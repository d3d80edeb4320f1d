"""The choice between the ways of a step's attention at the places where both sides were timed (8B shape: eight kv heads, 148 CTAs)."""
import shutil

import pytest

import att_plan

pytestmark = pytest.mark.skipif(shutil.which("g++") is None, reason="no host compiler")


@pytest.mark.parametrize("prompts, on_pairs", [
    ([256], 0), ([257], 1), ([300], 1), ([512], 1),
    # two prompts of a little more than 256 rows: 80 units on 74 pairs, 144 on 148 CTAs
    ([257, 257], 0), ([270, 288], 0), ([290, 290], 2), ([384, 384], 2),
    ([257] * 3, 3), ([300] * 4, 4), ([300] * 10, 10), ([430] * 10, 10), ([260] * 15, 15), ([200] * 8 + [400] * 4, 4), ([64] * 8, 0),
], ids=str)
def test_prompts_go_to_pairs_where_these_are_faster(prompts, on_pairs):
    assert att_plan.prompts_on_pairs([(0, p) for p in prompts], 8, 148) == on_pairs


def test_rows_behind_long_contexts_stay_on_pairs():
    assert att_plan.prompts_on_pairs([(3500, 512)], 8, 148) == 1
    assert att_plan.prompts_on_pairs([(700, 270), (700, 270)], 8, 148) == 2   # one round of single CTAs, each over 970 keys


@pytest.mark.parametrize("rows, keys, way", [
    (1, 300, "cta"), (17, 300, "cta"), (17, 4000, "cta"), (24, 40, "units"), (37, 40, "units"), (37, 100, "units"), (48, 40, "units"),
    (24, 100, "half"), (24, 300, "half"), (24, 1500, "half"), (30, 300, "half"), (30, 4000, "half"), (37, 300, "half"), (37, 1500, "half"), (37, 4000, "half"),
    (48, 300, "stream"), (100, 40, "units"), (200, 700, "stream")])
def test_single_rows_go_the_way_that_was_fastest(rows, keys, way):
    assert att_plan.decode_way([keys] * rows, 8, 148) == way


def test_single_rows_of_very_different_contexts_are_cut():
    assert att_plan.decode_way([100 + 3900 * i // 23 for i in range(24)], 8, 148) == "stream"
