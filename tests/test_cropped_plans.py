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


def test_the_cropped_test_layers_take_cropped_items(monkeypatch):
    import paper_1705_10591_b200 as lib
    from test_gpu_cropped_images import CASES
    monkeypatch.setenv("CONV2D_B200_TF32_CROP", "2")
    monkeypatch.setenv("CONV2D_B200_TF32_RESIDENT", "0")
    for case in CASES:
        for algo in (lib.ALGO_TF32, lib.ALGO_16BIT):
            assert lib.conv2d_fwd_plan_describe(*case, algo)["crop"] == 1, case
