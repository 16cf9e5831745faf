"""Run-to-run determinism and memory-safety checks that stand in for a sanitizer.

* The same pass run twice, and once more on another stream, gives bit-identical
  results (no kernel depends on scheduling order: every output element has one
  writer and a fixed summation order).
* Outputs and the workspace sit between canary bands; after all three passes the
  bands are untouched and every output element has been written.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# With math = 1 the first five run the FP32 kernel for small matrices in most passes, the last two the one for large
# matrices in all three; with math = 2 every pass runs on the tensor cores.
SHAPES = [(6, 20, 24, 13, 13, 3, 3, 16), (3, 18, 20, 31, 31, 5, 5, 32), (2, 9, 10, 64, 64, 11, 11, 64),
          (1, 5, 6, 120, 121, 7, 5, 128), (5, 3, 2, 7, 6, 3, 2, 8),
          (70, 66, 65, 13, 11, 3, 3, 16), (65, 67, 66, 29, 31, 5, 5, 32)]
LARGE = SHAPES[5:]
CANARY = 1024          # floats on either side


def _banded(torch, numel, fill):
    buf = torch.full((numel + 2 * CANARY,), 777.25, device="cuda")
    inner = buf[CANARY:CANARY + numel]
    inner.fill_(fill)
    return buf, inner


@pytest.mark.parametrize("dims", SHAPES)
@pytest.mark.parametrize("math", [1, 2])
def test_bit_identical_reruns_and_untouched_canaries(dims, math):
    import torch
    import paper_1412_7580_b200 as fc
    from paper_1412_7580_b200 import workloads as wl
    s = wl.ConvShape("det", *dims, cfg=10, point=sum(dims))
    x, w, dy = wl.make_x(s), wl.make_w(s), wl.make_dy(s)
    xd, wd, dyd = (torch.from_numpy(a).cuda() for a in (x, w, dy))
    p = fc.conv_plan(*s.args())
    fc.conv_plan_set_math(p, math)
    kernels = [fc.conv_plan_pass_kernel(p, k) for k in range(3)]
    if math == 2:
        assert kernels == [fc.binding.KERNEL_TENSOR] * 3
    elif dims in LARGE:
        assert kernels == [fc.binding.KERNEL_FP32_LARGE] * 3
    need = fc.conv_plan_workspace_bytes(p)
    # workspace between canary bands (256-byte aligned start: the band is 4096 bytes)
    ws_buf = torch.full((need // 4 + 2 * CANARY + 64,), 777.25, device="cuda")
    off = CANARY
    while (ws_buf.data_ptr() + 4 * off) % 256:
        off += 1
    ws = ws_buf[off:off + need // 4]
    fc.conv_plan_set_workspace(p, ws)
    shapes = ((s.S, s.fp, s.oh, s.ow), (s.S, s.f, s.h, s.w), (s.fp, s.f, s.kh, s.kw))

    def run(stream=None):
        outs = []
        ctx = torch.cuda.stream(stream) if stream is not None else None
        if ctx is not None:
            ctx.__enter__()
        try:
            for shp in shapes:
                outs.append(_banded(torch, int(np.prod(shp)), float("nan")))
            (yb, y), (dxb, dx), (dwb, dw) = outs
            fc.conv_fprop(p, xd, wd, y.view(shapes[0]))
            fc.conv_bprop(p, dyd, wd, dx.view(shapes[1]))
            fc.conv_accgrad(p, dyd, xd, dw.view(shapes[2]))
        finally:
            if ctx is not None:
                ctx.__exit__(None, None, None)
        torch.cuda.synchronize()
        return outs

    first = run()
    second = run()
    other = torch.cuda.Stream()
    other.wait_stream(torch.cuda.current_stream())
    third = run(other)
    assert fc.conv_plan_status(p) == 0
    for (b1, o1), (b2, o2), (b3, o3) in zip(first, second, third):
        assert bool(torch.isfinite(o1).all())                     # every element written
        assert torch.equal(o1, o2) and torch.equal(o1, o3)        # bit-identical reruns
        for b in (b1, b2, b3):
            assert bool((b[:CANARY] == 777.25).all()) and bool((b[-CANARY:] == 777.25).all())
    assert bool((ws_buf[:off] == 777.25).all())
    assert bool((ws_buf[off + need // 4:] == 777.25).all())
    fc.conv_plan_destroy(p)


# n = 64 with more tiles than SMs in all three inverse transforms (two teams per tile)
@pytest.mark.parametrize("math", [1, 2])
def test_bit_identical_reruns_of_many_tiles(math):
    test_bit_identical_reruns_and_untouched_canaries((19, 33, 30, 64, 63, 14, 2, 64), math)
