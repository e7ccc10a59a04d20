"""Which layers take items that are equal parts of one image (host only)."""
import pytest


@pytest.mark.parametrize("layer,crop", [
    ((32, 256, 14, 14, 256, 3, 3), 1), ((64, 128, 32, 32, 128, 7, 7), 1), ((16, 256, 7, 139, 256, 7, 1), 1),
    ((128, 256, 11, 139, 6, 3, 3), 0),                    # narrower items stage more pixels than the MMAs take time
    ((128, 64, 30, 30, 200, 3, 3), 0),                    # the estimate falls by less than 4 %
])
def test_cropped_items_are_taken_by_the_rule(layer, crop):
    import paper_1705_10591_b200 as lib
    assert lib.conv2d_fwd_plan_describe(*layer, lib.ALGO_TF32)["crop"] == crop
