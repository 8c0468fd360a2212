"""The fused split-K kernel on products that mm_gemm gives it, past the line below
which they run on the CUDA cores: every test asserts that the kernel ran.  One
and several clusters a tile, short and ragged K, scaled blocks, non-finite
entries, exact sums, guard words, streams and the epilogue."""
import numpy as np
import pytest
import torch

import oracle
import synth
from gpu_util import assert_full, dev, full_errors

pytestmark = pytest.mark.gpu

X3, X6 = "MM_MODE_SPLIT_BF16X3", "MM_MODE_SPLIT_BF16X6"
# m just past one K block (on many tiles), K blocks cut short, ragged n and p,
# clusters of several sizes, several clusters a tile (the long ones)
SHAPES = [(1000, 100, 1000), (900, 132, 1100), (520, 700, 388), (512, 512, 512), (300, 2300, 200),
          (257, 6000, 132), (96, 32768, 64), (40, 49152, 40)]
_ids = lambda s: "x".join(map(str, s))


@pytest.fixture
def fused(mmlib):
    """mm_gemm (or another entry point) that must launch the fused kernel once."""
    def call(f, *args):
        torch.cuda.synchronize()  # the synchronous calls run on the library's own stream
        mmlib.mm_trace_reset()
        assert mmlib.mm_trace_enable(True) == 0
        try:
            assert f(*args) == mmlib.MM_OK
            assert mmlib.mm_trace_read("fused_tc")[1] == 1
        finally:
            mmlib.mm_trace_enable(False)
            mmlib.mm_trace_reset()
    return call


def _product(mm, fused, A, B, mode=X3):
    (n, m), p = A.shape, B.shape[1]
    C = torch.full((n, p), float("nan"), device="cuda")
    fused(mm.mm_gemm, n, m, p, dev(A), dev(B), C, mm.MM_F32, getattr(mm, mode))
    return C.cpu().numpy()


def _uniform(seed, n, m, p):
    return synth.uniform_pm1(seed, (n, m)), synth.uniform_pm1(seed + 1, (m, p))


@pytest.mark.parametrize("shape", SHAPES, ids=_ids)
@pytest.mark.parametrize("mode", [X3, X6])
def test_uniform(mmlib, fused, shape, mode):
    A, B = _uniform(10001, *shape)
    assert_full(_product(mmlib, fused, A, B, mode), A, B, "f32")


@pytest.mark.parametrize("shape", [(1000, 100, 1000), (257, 6000, 132), (40, 49152, 40)], ids=_ids)
def test_small_integers_are_exact(mmlib, fused, shape):
    n, m, p = shape
    A, B = synth.small_ints(10011, (n, m)), synth.small_ints(10012, (m, p))
    assert np.array_equal(_product(mmlib, fused, A, B).astype(np.float64),
                          A.astype(np.float64) @ B.astype(np.float64))


@pytest.mark.parametrize("mode", [X3, X6])
def test_scaled_blocks(mmlib, fused, mode):
    """Rows at 2^-70 and 2^60, columns at 2^-45 and 2^45: blocks outside [2^-40, 2^40]
    are scaled; the first row tile's rows stay in range."""
    n, m, p = 400, 1000, 400
    A, B = (x.astype(np.float64) for x in _uniform(10021, n, m, p))
    ea = synth.row_scale_exponents(10023, n, choices=(-70, 60))
    ea[:128] = 0
    eb = synth.row_scale_exponents(10024, p, choices=(-45, 45))
    A = np.ldexp(A, ea[:, None]).astype(np.float32)
    B = np.ldexp(B, eb[None, :]).astype(np.float32)
    C = _product(mmlib, fused, A, B, mode)
    assert np.isfinite(C).all()
    assert_full(C, A, B, "f32")


def test_cancelling_terms_in_a_scaled_block(mmlib, fused):
    """Terms of 2.25e38 that cancel within a K block: their sum out of FP32's range on
    the way, the block's not."""
    A, B = _uniform(10031, 520, 700, 388)
    for k, s in ((0, 1), (1, 1), (2, -1)):
        A[::3, k], B[k] = np.float32(s * 1.5e19), np.float32(1.5e19)
    C = _product(mmlib, fused, A, B)
    ref, absref = oracle.default().gemm(A, B, with_abs=True)
    assert oracle.rel_errors(C, ref, absref).max() <= oracle.tolerance(700, "f32")


def test_magnitudes_over_forty_binades(mmlib, fused):
    A, B = synth.pow2_real(10041, (300, 4096)), synth.pow2_real(10042, (4096, 300))
    assert_full(_product(mmlib, fused, A, B), A, B, "f32")


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_nonfinite_entry(mmlib, fused, bad):
    """Its row of C is not finite; the others keep the tolerance."""
    A, B = _uniform(10051, 400, 1000, 400)
    A[133, 77] = bad
    C = _product(mmlib, fused, A, B)
    assert not np.isfinite(C[133]).any()
    keep = np.arange(400) != 133
    e, _ = full_errors(C[keep], A[keep], B)
    assert e.max() <= oracle.tolerance(1000, "f32")


@pytest.mark.parametrize("shape", [(257, 6000, 132), (1000, 100, 1000)], ids=_ids)
def test_guard_words(mmlib, fused, shape):
    n, m, p = shape
    A, B = _uniform(10061, n, m, p)
    buf = torch.full((n * p + 64,), 7.0, device="cuda")
    fused(mmlib.mm_gemm, n, m, p, dev(A), dev(B), buf[32:32 + n * p], mmlib.MM_F32, getattr(mmlib, X3))
    assert torch.all(buf[:32] == 7.0) and torch.all(buf[32 + n * p:] == 7.0)
    assert_full(buf[32:32 + n * p].reshape(n, p).cpu().numpy(), A, B, "f32")


@pytest.mark.parametrize("shape", [(96, 32768, 64), (520, 700, 388)], ids=_ids)
def test_same_bits_again_and_on_a_stream(mmlib, fused, shape):
    mm, (n, m, p) = mmlib, shape
    A, B = (dev(x) for x in _uniform(10071, n, m, p))
    C = [torch.full((n, p), float("nan"), device="cuda") for _ in range(3)]
    s = torch.cuda.Stream()
    fused(mm.mm_gemm, n, m, p, A, B, C[0], mm.MM_F32, getattr(mm, X3))
    fused(mm.mm_gemm, n, m, p, A, B, C[1], mm.MM_F32, getattr(mm, X3))
    for _ in range(4):
        assert mm.mm_gemm_async(n, m, p, A, B, C[2], mm.MM_F32, getattr(mm, X3), s) == mm.MM_OK
    assert mm.mm_sync(s) == mm.MM_OK
    assert torch.equal(C[0], C[1]) and torch.equal(C[0], C[2])


@pytest.mark.parametrize("shape", [(96, 32768, 64), (520, 700, 388), (1000, 100, 1000)], ids=_ids)
def test_epilogue(mmlib, fused, shape):
    """C = A.B - D, beside C and in place: the product's bits combined once."""
    mm, (n, m, p) = mmlib, shape
    A, B = (dev(x) for x in _uniform(10081, n, m, p))
    D = dev(synth.uniform_pm1(10083, (n, p)))
    C, E = (torch.full((n, p), float("nan"), device="cuda") for _ in range(2))
    fused(mm.mm_gemm, n, m, p, A, B, C, mm.MM_F32, getattr(mm, X3))
    fused(mm.mm_gemm_axpby, n, m, p, 1.0, A, B, -1.0, D, E, mm.MM_F32, getattr(mm, X3))
    assert torch.equal(E, C - D)
    F = D.clone()
    fused(mm.mm_gemm_axpby, n, m, p, 1.0, A, B, -1.0, F, F, mm.MM_F32, getattr(mm, X3))
    assert torch.equal(F, E)
