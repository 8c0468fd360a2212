"""Small products of the split modes on the CUDA cores: entries whose terms stay
in FP32's range but whose running sum does not come out as the terms cancel
(or as the infinity that they add up to), alone, with the epilogue and off C's
16-byte alignment; infinities and NaNs of the operands give MM_MODE_SIMT's bits."""
import numpy as np
import pytest
import torch

import oracle
import synth
from gpu_util import dev

pytestmark = pytest.mark.gpu

MODES = ["MM_MODE_SPLIT_BF16X3", "MM_MODE_SPLIT_BF16X6"]
# one slice, a cluster's slices on both tiles, more slices than a cluster holds
SHAPES = [(1, 4, 4), (40, 100, 60), (64, 512, 64), (256, 256, 256), (33, 2052, 20), (64, 16384, 64)]


def _operands(n, m, p):
    """Rows 0, 3, 6, ... of A and all of B hold terms of +-2.25e38 at K 0, 1
    and m - 1: two of one sign, then one of the other."""
    A, B = synth.uniform_pm1(9801, (n, m)), synth.uniform_pm1(9802, (m, p))
    for k, s in ((0, 1), (1, 1), (m - 1, -1)):
        A[::3, k] = np.float32(s * 1.5e19)
        B[k] = np.float32(1.5e19)
    return A, B


def _gemm(mm, A, B, C, mode):
    n, m = A.shape
    assert mm.mm_gemm(n, m, B.shape[1], A, B, C, mm.MM_F32, mode) == mm.MM_OK


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("mode", MODES)
@pytest.mark.parametrize("offset", [0, 1])
def test_cancelling_sums(mmlib, shape, mode, offset):
    mm, (n, m, p), md = mmlib, shape, getattr(mmlib, mode)
    A, B = _operands(n, m, p)
    ref, absref = oracle.default().gemm(A, B, with_abs=True)
    dA, dB = dev(A), dev(B)
    C = torch.full((n * p + 1,), float("nan"), device="cuda")[offset:n * p + offset].view(n, p)
    _gemm(mm, dA, dB, C, md)
    S = torch.empty(n, p, device="cuda")
    _gemm(mm, dA, dB, S, mm.MM_MODE_SIMT)
    assert not torch.isfinite(S[::3]).any()  # the plain sums do overflow
    e = oracle.rel_errors(C.cpu().numpy(), ref, absref)
    assert e.max() <= oracle.tolerance(m, "f32")
    kept = torch.isfinite(S)
    assert torch.equal(C[kept], S[kept])
    if offset == 0:
        E = torch.from_numpy(synth.uniform_pm1(9803, (n, p))).cuda() * 1e38
        D = E.clone()
        assert mm.mm_gemm_axpby(n, m, p, 1.0, dA, dB, -1.0, E, E, mm.MM_F32, md) == mm.MM_OK
        assert torch.equal(E, C - D)


@pytest.mark.parametrize("shape", [(256, 256, 256), (64, 16384, 64)], ids=lambda s: "x".join(map(str, s)))
def test_overflow_and_nonfinite_operands(mmlib, shape):
    mm, (n, m, p) = mmlib, shape
    A, B = _operands(n, m, p)
    A[6, m - 1] = np.float32(1.5e19)     # row 6: the sum itself is out of range
    A[9, [0, 1, m - 1]] *= np.float32(-1)
    A[9, m - 1] *= np.float32(-1)        # row 9: and below it
    A[12, 5] = np.inf                    # infinite and NaN operands beside sums that cancel
    B[7, 3] = np.nan
    dA, dB = dev(A), dev(B)
    C, S = torch.empty(n, p, device="cuda"), torch.empty(n, p, device="cuda")
    _gemm(mm, dA, dB, C, mm.MM_MODE_SPLIT_BF16X3)
    _gemm(mm, dA, dB, S, mm.MM_MODE_SIMT)
    cols = [j for j in range(p) if j != 3]
    assert torch.all(C[6, cols] == np.inf) and torch.all(C[9, cols] == -np.inf)
    for rows, c in ((12, slice(None)), (slice(None), 3)):
        assert torch.equal(torch.nan_to_num(C[rows, c], nan=7.0, posinf=8.0, neginf=9.0),
                           torch.nan_to_num(S[rows, c], nan=7.0, posinf=8.0, neginf=9.0))
