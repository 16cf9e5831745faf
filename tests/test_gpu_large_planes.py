"""Transforms of planes that need the bases 64 and 128: the kernels choose their loads by the parity of the row length
and by the alignment of the tensor, split the rows over work items and clip ragged tiles of 8 planes."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


# (S, f, f', h, w, kh, kw, n), samples by which the tensors are shifted in memory, tile basis
@pytest.mark.parametrize("dims,shift,tile", [
    ((2, 9, 3, 128, 128, 5, 5, 128), 0, 0),   # pairs of columns; every row and column in use
    ((2, 9, 3, 128, 128, 5, 5, 128), 1, 0),   # the same from an address that is no multiple of 8 bytes
    ((1, 8, 10, 66, 127, 3, 4, 128), 0, 0),   # odd rows, the last column has no partner; dy's rows are even
    ((3, 1, 17, 127, 66, 2, 3, 128), 0, 0),   # one plane in a tile, tiles of 8 + 8 + 1
    ((1, 7, 8, 40, 101, 9, 3, 128), 2, 0),    # fewer rows than half the basis
    ((2, 3, 5, 97, 20, 97, 2, 128), 0, 0),    # narrow planes, kernel as high as the plane
    ((2, 9, 12, 64, 64, 14, 5, 64), 0, 0),
    ((2, 9, 12, 64, 64, 5, 14, 64), 1, 0),
    ((1, 8, 10, 33, 63, 3, 4, 64), 0, 0),
    ((3, 5, 17, 61, 20, 15, 3, 64), 3, 0),    # narrow planes and filters too high for the small-plane kernel
    ((2, 4, 3, 57, 58, 3, 3, 64), 0, 0),      # no tile more than half full
    ((19, 33, 30, 64, 63, 14, 2, 64), 0, 0),  # more tiles of 4 planes than SMs, the last of a row not full
    ((19, 30, 33, 57, 64, 2, 13, 64), 1, 0),
    ((2, 9, 6, 128, 128, 5, 7, 128), 0, 64),  # windows of 64 x 64: pairs inside or outside as a whole,
    ((2, 9, 6, 128, 128, 7, 6, 128), 1, 64),  # odd origins and addresses,
    ((9, 17, 18, 100, 128, 5, 7, 128), 0, 64),
    ((1, 3, 9, 97, 125, 13, 2, 128), 0, 64),  # odd planes, windows that hang over the edge
])
def test_passes_against_oracle(dims, shift, tile):
    import torch
    import oracle
    import paper_1412_7580_b200 as fc
    from paper_1412_7580_b200 import workloads as wl
    s = wl.ConvShape("large_planes", *dims, cfg=9, point=sum(dims) + shift)
    host = wl.make_x(s), wl.make_w(s), wl.make_dy(s)

    def shifted(a):
        flat = torch.empty(a.size + shift, device="cuda")
        flat[shift:] = torch.from_numpy(a.ravel()).cuda()
        return flat[shift:].view(a.shape)

    x, w, dy = host
    xd, wd, dyd = (shifted(a) for a in host)
    p = fc.conv_plan(*s.args())
    fc.conv_plan_set_math(p, fc.binding.MATH_FP32)
    fc.conv_plan_set_tiling(p, tile)
    fc.conv_plan_alloc_workspace(p)
    y, dx, dw = (shifted(np.full(shape, np.nan, np.float32)) for shape in
                 ((s.S, s.fp, s.oh, s.ow), x.shape, w.shape))
    fc.conv_fprop(p, xd, wd, y)
    fc.conv_bprop(p, dyd, wd, dx)
    fc.conv_accgrad(p, dyd, xd, dw)
    torch.cuda.synchronize()
    assert fc.conv_plan_status(p) == 0
    # FP32 end to end: 2 x 14 butterfly stages and sums of at most 4 x 54 products (9 planes x 6 windows), each rounded at
    # 2^-24 of its value, signs at random: 2^-24 (28 + sqrt(216)) = 2.5e-6 of the largest result; four times that
    for got, ref in ((y, oracle.fprop(x, w)), (dx, oracle.bprop(dy, w, s.h, s.w)), (dw, oracle.accgrad(dy, x, s.kh, s.kw))):
        g = got.cpu().numpy().astype(np.float64)
        assert np.max(np.abs(g - ref)) <= 1e-5 * np.max(np.abs(ref))
    fc.conv_plan_destroy(p)


# Spectra beyond the L2 whose rows are no whole sectors (12 planes), by tiles in even numbers (the plain kernel) and in odd ones
# (clusters of eight, the last one not full), and ones so large that two CTAs keep step
@pytest.mark.parametrize("dims", [(668, 12, 2, 33, 34, 14, 2, 64), (667, 12, 2, 33, 34, 14, 2, 64), (4003, 7, 1, 33, 35, 14, 2, 64)])
def test_forward_transform_of_spectra_beyond_the_l2(dims):
    import torch
    import oracle
    import paper_1412_7580_b200 as fc
    from paper_1412_7580_b200 import workloads as wl
    s = wl.ConvShape("beyond_l2", *dims, cfg=9, point=sum(dims))
    x, w, dy = wl.make_x(s), wl.make_w(s), wl.make_dy(s)
    p = fc.conv_plan(*s.args())
    fc.conv_plan_set_math(p, fc.binding.MATH_FP32)
    fc.conv_plan_alloc_workspace(p)
    y = torch.full((s.S, s.fp, s.oh, s.ow), float("nan"), device="cuda")
    dw = torch.full(w.shape, float("nan"), device="cuda")
    xd = torch.from_numpy(x).cuda()
    fc.conv_fprop(p, xd, torch.from_numpy(w).cuda(), y)
    fc.conv_accgrad(p, torch.from_numpy(dy).cuda(), xd, dw)
    torch.cuda.synchronize()
    assert fc.conv_plan_status(p) == 0
    # 2 x 12 butterfly stages and sums of 12 (y) or at most 4,003 products (dw), each rounded at 2^-24 of its value, signs at
    # random: 2^-24 (24 + sqrt(4003)) = 5.2e-6 of the largest result; four times that
    for got, ref in ((y, oracle.fprop(x, w)), (dw, oracle.accgrad(dy, x, s.kh, s.kw))):
        assert np.max(np.abs(got.cpu().numpy().astype(np.float64) - ref)) <= 2.1e-5 * np.max(np.abs(ref))
    fc.conv_plan_destroy(p)


# The gradient that is added to: pairs of columns (even crop, even address) and single samples, n = 64 with more tiles than SMs
# (no square crop that the small-crop kernel takes) and n = 128
@pytest.mark.parametrize("dims,shift", [
    ((2, 33, 30, 64, 63, 14, 2, 64), 0),
    ((2, 33, 30, 64, 63, 14, 2, 64), 1),
    ((2, 30, 33, 57, 64, 2, 13, 64), 0),
    ((2, 33, 30, 40, 40, 13, 13, 64), 0),
    ((2, 9, 11, 120, 120, 7, 6, 128), 0),
    ((2, 9, 11, 120, 120, 7, 6, 128), 1),
])
def test_accumulated_filter_gradient(dims, shift):
    import torch
    import oracle
    import paper_1412_7580_b200 as fc
    from paper_1412_7580_b200 import workloads as wl
    s = wl.ConvShape("accumulate", *dims, cfg=9, point=sum(dims) + shift)
    x, dy, before = wl.make_x(s), wl.make_dy(s), wl.make_w(s)
    p = fc.conv_plan(*s.args())
    fc.conv_plan_set_math(p, fc.binding.MATH_FP32)
    fc.conv_plan_alloc_workspace(p)
    flat = torch.empty(before.size + shift, device="cuda")
    flat[shift:] = torch.from_numpy(before.ravel()).cuda()
    dw = flat[shift:].view(before.shape)
    fc.conv_accgrad(p, torch.from_numpy(dy).cuda(), torch.from_numpy(x).cuda(), dw, accumulate=True)
    torch.cuda.synchronize()
    assert fc.conv_plan_status(p) == 0
    # the bound of test_passes_against_oracle and one rounding more
    ref = before.astype(np.float64) + oracle.accgrad(dy, x, s.kh, s.kw)
    assert np.max(np.abs(dw.cpu().numpy().astype(np.float64) - ref)) <= 1e-5 * np.max(np.abs(ref))
    fc.conv_plan_destroy(p)


# one tile of 4 planes for every SM (the plain inverse kernel) and one more (two teams per tile)
@pytest.mark.parametrize("dims", [(37, 2, 16, 33, 40, 5, 7, 64), (149, 2, 3, 34, 33, 6, 5, 64)])
def test_inverse_of_as_many_tiles_as_sms(dims):
    import torch
    import oracle
    import paper_1412_7580_b200 as fc
    from paper_1412_7580_b200 import workloads as wl
    s = wl.ConvShape("sms", *dims, cfg=9, point=sum(dims))
    x, w = wl.make_x(s), wl.make_w(s)
    p = fc.conv_plan(*s.args())
    fc.conv_plan_set_math(p, fc.binding.MATH_FP32)
    fc.conv_plan_alloc_workspace(p)
    y = torch.full((s.S, s.fp, s.oh, s.ow), float("nan"), device="cuda")
    fc.conv_fprop(p, torch.from_numpy(x).cuda(), torch.from_numpy(w).cuda(), y)
    torch.cuda.synchronize()
    ref = oracle.fprop(x, w)
    assert np.max(np.abs(y.cpu().numpy().astype(np.float64) - ref)) <= 1e-5 * np.max(np.abs(ref))
    fc.conv_plan_destroy(p)
