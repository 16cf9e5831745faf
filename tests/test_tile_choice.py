"""The static choice of a tile basis against measured training steps: for each layer the bases whose step was within 8 % of
the fastest one on B200 (steps in us in the comment)."""
import pytest

import paper_1412_7580_b200 as fc

CASES = [
    # (S, f, f', h, w, k, n), bases
    ((16, 128, 256, 32, 32, 7, 32), (16,)),             # untiled 251, 8: 649, 16: 197
    ((1, 64, 16, 64, 64, 11, 64), (16,)),               # 117, 16: 56, 32: 63
    ((16, 64, 256, 32, 32, 3, 32), (8,)),               # 161, 8: 128, 16: 143
    ((1, 3, 256, 57, 57, 3, 64), (8,)),                 # 263, 8: 57, 16: 81, 32: 120
    ((1, 384, 1, 120, 120, 13, 128), (32,)),            # 1373, 16: 576, 32: 249, 64: 425
    ((16, 16, 256, 128, 94, 13, 128), (64,)),           # 1549, 16: 5906, 32: 1108, 64: 897
    ((16, 128, 1, 120, 120, 7, 128), (32, 64)),         # 730, 8: 4528, 16: 621, 32: 454, 64: 490
    ((1, 3, 16, 200, 200, 5, 256), (32,)),              # 8: 319, 16: 84, 32: 68, 64: 90
    ((121, 71, 80, 58, 58, 3, 64), (32,)),              # 676, 32: 625
    ((64, 64, 64, 64, 64, 3, 64), (0,)),                # 357, 8: 640, 16: 406, 32: 589
    ((64, 64, 64, 128, 128, 5, 128), (32, 0)),          # 1805, 8: 4818, 16: 1862, 32: 1667, 64: 2128
    ((16, 256, 256, 128, 128, 3, 128), (16,)),          # 10419, 8: 2252, 16: 1834, 32: 2276, 64: 3790
]


@pytest.mark.parametrize("dims,bases", CASES)
def test_static_choice_is_among_the_fast_bases(dims, bases):
    S, f, fp, h, w, k, n = dims
    p = fc.conv_plan(S, f, fp, h, w, k, k, n)
    fc.conv_plan_set_tiling(p, fc.TILE_AUTO)
    assert fc.conv_plan_tile_basis(p) in bases
    fc.conv_plan_destroy(p)
