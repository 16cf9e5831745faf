"""The per-bin complex contraction alone (Table 1, the Cgemm row) against the
oracle's plain sum, in both arithmetic modes and on ragged shapes."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

TOL = {1: 1e-4, 2: 5e-3}


def run(bins, M, N, K, math, seed=0, transA=False, transB=False, conjA=False, conjB=False):
    import torch
    import oracle
    import paper_1412_7580_b200 as fc
    rng = np.random.default_rng([14127580, 55, seed, bins, M, N, K])
    r4 = lambda v: (v + 3) // 4 * 4

    def operand(rows, trans, fill):
        """Logical [bins][rows][K] complex matrix, stored planar either as
        [2][bins][rows][ld>=K] or, transposed, as [2][bins][K][ld>=rows]."""
        re = rng.standard_normal((bins, rows, K), dtype=np.float32)
        im = rng.standard_normal((bins, rows, K), dtype=np.float32)
        if not trans:
            buf = np.full((2, bins, rows, r4(K)), fill, np.float32)   # padding must never be read as data
            buf[0, :, :, :K], buf[1, :, :, :K] = re, im
        else:
            buf = np.full((2, bins, K, r4(rows)), fill, np.float32)
            buf[0, :, :, :rows], buf[1, :, :, :rows] = re.transpose(0, 2, 1), im.transpose(0, 2, 1)
        return buf, re.astype(np.float64) + 1j * im.astype(np.float64)

    A, Ac = operand(M, transA, 1e30)
    B, Bc = operand(N, transB, -1e30)
    ldc = r4(N)
    Ad, Bd = torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda()
    Cd = torch.full((2, bins, M, ldc), float("nan"), device="cuda")
    status = torch.zeros(64, dtype=torch.int32, device="cuda")
    fc.fftconv_bin_contract(Ad, Bd, Cd, M, N, K, transA, transB, conjA, conjB, math=math,
                            status_word=status)
    torch.cuda.synchronize()
    assert int(status[0].item()) == 0
    C = Cd.cpu().numpy().astype(np.float64)
    got = C[0, :, :, :N] + 1j * C[1, :, :, :N]
    ref = oracle.bin_contract(Ac, Bc, conjA, conjB)
    assert np.all(np.isfinite(got.real)) and np.all(np.isfinite(got.imag))
    # padding columns of C (N..ldc-1) are scratch: untouched or zero, never data
    if ldc > N:
        pad = C[..., N:]
        assert np.all(np.isnan(pad) | (pad == 0))
    return float(np.max(np.abs(got - ref)) / np.max(np.abs(ref)))


SHAPES = [
    # bins, M, N, K
    (3, 8, 8, 4), (5, 128, 128, 32), (7, 128, 64, 64), (4, 128, 256, 96), (2, 64, 64, 128),
    (3, 130, 70, 33), (2, 1, 1, 1), (9, 37, 129, 100), (2, 384, 384, 128), (300, 32, 48, 16),
    (2, 256, 96, 128), (1, 128, 384, 384),
]


@pytest.mark.parametrize("shape", SHAPES)
def test_contraction_fp32(shape):
    assert run(*shape, math=1) <= TOL[1]


@pytest.mark.parametrize("shape", SHAPES)
def test_contraction_tf32_tensor_cores(shape):
    assert run(*shape, math=2) <= TOL[2]


def test_tf32_many_tiles_per_cta():
    # more tiles than SMs: every CTA walks several tiles through both accumulator buffers
    assert run(700, 128, 128, 64, math=2, seed=3) <= TOL[2]


# operand storage / conjugation as used by the three passes, plus the remaining combinations
FLAGS = [
    dict(transA=False, transB=False, conjA=False, conjB=True),    # fprop
    dict(transA=False, transB=True, conjA=False, conjB=False),    # bprop
    dict(transA=True, transB=True, conjA=True, conjB=False),      # accGrad
    dict(transA=True, transB=False, conjA=True, conjB=True),
]


@pytest.mark.parametrize("flags", FLAGS)
@pytest.mark.parametrize("math", [1, 2])
@pytest.mark.parametrize("shape", [(5, 128, 128, 64), (3, 130, 70, 33), (2, 37, 129, 100),
                                   (4, 64, 96, 128), (2, 8, 8, 4)])
def test_contraction_layouts_and_conjugates(shape, math, flags):
    assert run(*shape, math=math, seed=9, **flags) <= TOL[math]


# tiles of one warp (4 x 64 .. 64 x 4): every tile shape, edges and remainders of rows, columns and k-blocks
@pytest.mark.parametrize("flags", FLAGS)
@pytest.mark.parametrize("math", [1, 2])
@pytest.mark.parametrize("shape", [(40, 1, 1, 1), (9, 4, 64, 8), (9, 3, 65, 9), (9, 8, 32, 7), (9, 7, 33, 17), (9, 16, 16, 16),
                                   (9, 15, 17, 3), (9, 32, 8, 24), (9, 33, 7, 2), (9, 64, 4, 8), (9, 70, 3, 5),
                                   (5, 2, 3, 203), (3000, 2, 5, 3)])
def test_contraction_of_small_matrices(shape, math, flags):
    assert run(*shape, math=math, seed=11, **flags) <= TOL[math]


# tensor-core tiles used in part: rows of the boxes (8, 16, 32 at a time), N of the instructions (16), k-steps
# (8) and stages of the ring, and the line at which a tile counts as full (M > 120 and N > 112)
@pytest.mark.parametrize("flags", FLAGS[:3])
@pytest.mark.parametrize("shape", [(200, 121, 113, 33), (200, 120, 113, 64), (200, 121, 112, 40), (200, 33, 97, 65),
                                   (200, 65, 33, 96), (200, 40, 200, 8), (200, 136, 48, 72)])
def test_tf32_tiles_used_in_part(shape, flags):
    assert run(*shape, math=2, seed=13, **flags) <= TOL[2]


# With TF32 operands (10 explicit bits) a product is off by up to 2^-10 of itself, and some of the outputs here by
# more than 2e-5 of the largest; exact FP32 sums of up to K = 200 terms stay within K 2^-24 = 1.2e-5.
@pytest.mark.parametrize("flags", FLAGS[:3])
@pytest.mark.parametrize("shape", [(288, 8, 8, 16), (544, 8, 16, 4), (288, 1, 64, 16), (2112, 16, 16, 16), (2112, 4, 194, 4),
                                   (544, 2, 70, 200)])
def test_the_arithmetic_asked_for_is_the_one_that_runs(shape, flags):
    assert run(*shape, math=1, seed=17, **flags) <= 1.2e-5
    assert 2e-5 <= run(*shape, math=2, seed=17, **flags) <= TOL[2]


# narrow matrices run several CTAs per SM (N <= 32: up to four, N <= 64: two), as many as find shared memory for their
# rows: both lines, rows that fill one to four staging tiles, one and several k-blocks, more tiles than all CTAs
@pytest.mark.parametrize("flags", FLAGS[:3])
@pytest.mark.parametrize("shape", [(1300, 8, 16, 4), (1300, 16, 8, 33), (700, 55, 12, 15), (700, 97, 32, 40), (700, 128, 33, 33),
                                   (400, 130, 64, 16), (400, 64, 65, 8), (650, 121, 5, 130), (1300, 1, 130, 3)])
def test_tf32_several_ctas_per_sm(shape, flags):
    assert run(*shape, math=2, seed=19, **flags) <= TOL[2]


# as many CTAs per SM as there are tiles for: both sides of 1, 2 and 3 tiles per SM, a sum of many k-blocks
@pytest.mark.parametrize("flags", FLAGS[:3])
@pytest.mark.parametrize("shape", [(148, 9, 14, 40), (149, 9, 14, 40), (296, 30, 33, 9), (297, 30, 33, 9), (445, 12, 20, 7),
                                   (34, 45, 10, 700), (130, 130, 12, 100)])
def test_tf32_ctas_per_sm_follow_the_tiles(shape, flags):
    assert run(*shape, math=2, seed=23, **flags) <= TOL[2]
