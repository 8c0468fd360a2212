"""FP64 emulation by sliced e4m3 products: the digit blocks of 32 rows and 32
columns, the column pairs of the final sum (even p of 512 and more) and the
wide loads of the maxima (rows of a multiple of four values), at one short, at
and past each edge, for slice counts on both sides of each word split, equal
bit for bit to the oracle with the accuracy gate off and on (uniform inputs,
which the gate's bound clears for 12 slices), with unaligned operands too."""
import numpy as np
import pytest
import torch

import synth
from gpu_util import dev
from oracle import ozaki

pytestmark = pytest.mark.gpu


@pytest.fixture
def mm(mmlib):
    yield mmlib
    assert mmlib.mm_ozaki_slices(ozaki.DEFAULT_SLICES) == mmlib.MM_OK
    assert mmlib.mm_ozaki_gate(1) == mmlib.MM_OK


def _run(mm, dA, dB, n, m, p):
    dC = torch.full((n, p), float("nan"), dtype=torch.float64, device="cuda")
    assert mm.mm_gemm(n, m, p, dA, dB, dC, mm.MM_F64, mm.MM_MODE_OZAKI) == mm.MM_OK
    return dC.cpu().numpy()


def _off(x, k):
    """The values of x in device memory k doubles past an allocation's start."""
    t = torch.zeros(x.size + k, dtype=torch.float64, device="cuda")
    t[k:] = dev(x, torch.float64).flatten()
    return t[k:].view(*x.shape)


@pytest.mark.parametrize("shape", [(31, 127, 511), (32, 128, 512), (33, 129, 513), (9, 132, 514),
                                   (160, 260, 1026), (129, 64, 33)], ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("S", [2, 3, 4, 6, 7, 9, 10, 12])
def test_edges(mm, shape, S):
    n, m, p = shape
    A, B = synth.uniform_pm1_f64(9501 + S, (n, m)), synth.uniform_pm1_f64(9502 + S, (m, p))
    A[n // 2, m // 3:] = 0.0
    A[0] *= 2.0 ** -70
    ref = ozaki.gemm(A, B, S)
    assert mm.mm_ozaki_slices(S) == mm.MM_OK
    for gate in (0, 1) if S == 12 else (0,):
        assert mm.mm_ozaki_gate(gate) == mm.MM_OK
        assert np.array_equal(_run(mm, dev(A, torch.float64), dev(B, torch.float64), n, m, p), ref)


@pytest.mark.parametrize("k", [1, 2, 3])
def test_unaligned(mm, k):
    n, m, p = 65, 136, 516
    A, B = synth.uniform_pm1_f64(9511, (n, m)), synth.uniform_pm1_f64(9512, (m, p))
    assert mm.mm_ozaki_gate(0) == mm.MM_OK
    ref = ozaki.gemm(A, B, ozaki.DEFAULT_SLICES)
    assert np.array_equal(_run(mm, _off(A, k), _off(B, 4 - k), n, m, p), ref)


def test_infinite_rows_and_columns(mm):
    """A row or column with an infinity or a NaN is NaN, as are both of a pair
    of columns only where each is."""
    n, m, p = 40, 64, 600
    A, B = synth.uniform_pm1_f64(9521, (n, m)), synth.uniform_pm1_f64(9522, (m, p))
    A[7, 3], B[5, 10], B[9, 513] = np.inf, np.nan, -np.inf
    assert mm.mm_ozaki_gate(0) == mm.MM_OK
    C = _run(mm, dev(A, torch.float64), dev(B, torch.float64), n, m, p)
    bad = np.zeros((n, p), bool)
    bad[7], bad[:, 10], bad[:, 513] = True, True, True
    assert np.array_equal(np.isnan(C), bad)
    A[7, 3], B[5, 10], B[9, 513] = 0.0, 0.0, 0.0
    ref = ozaki.gemm(A, B, ozaki.DEFAULT_SLICES)
    assert np.array_equal(C[~bad], ref[~bad])
