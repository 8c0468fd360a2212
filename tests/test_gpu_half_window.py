"""The fp16 window's low end against the accuracy contract: rows of A and columns
of B that lie wholly in its lowest binades (or just below it) meet 1e-6 sqrt(m)
where they meet, for every short inner dimension, alone and in a table; up to
m = 16 the three-part form serves every product."""
import numpy as np
import pytest
import torch

import oracle
import synth
from gpu_util import dev, full_errors

pytestmark = pytest.mark.gpu


def _grouped(mm, A, B, mode, extra=()):
    """C = A.B in a grouped call, beside `extra` products."""
    outs = [torch.full((a.shape[0], b.shape[1]), float("nan"), device="cuda") for a, b in ((A, B), *extra)]
    tab = [(a.shape[0], a.shape[1], b.shape[1], dev(a), dev(b), c) for (a, b), c in zip(((A, B), *extra), outs)]
    assert mm.mm_gemm_grouped(tab, mm.MM_F32, mode) == 0
    return outs[0].cpu().numpy()


def _pair(seed, n, m, p):
    """Magnitudes in [1/2, 1): the largest sampled one is brought to [2^13, 2^14)."""
    mag = lambda s, shape: (np.abs(synth.uniform_pm1(s, shape)) * 0.5 + 0.5).astype(np.float32)
    return np.minimum(mag(seed, (n, m)), np.float32(1 - 2.0 ** -24)), np.minimum(
        mag(seed + 1, (m, p)), np.float32(1 - 2.0 ** -24))


@pytest.mark.parametrize("m", [1, 2, 4, 8, 16, 17, 32, 33, 36, 63, 64, 65])
@pytest.mark.parametrize("e", [-27, -28, -29, -30])
@pytest.mark.parametrize("table", [False, True], ids=["alone", "table"])
def test_small_rows_meet_small_columns(mmlib, m, e, table):
    """A few rows and columns in [2^e, 2^(e + 1)), with random bits and with bits
    whose low parts are largest (1 + 2^-9 at 2^-30)."""
    n, p = 700, 520
    A, B = _pair(9701, n, m, p)
    A[3:5] *= np.float32(2.0 ** (e + 1))
    B[:, 5:7] *= np.float32(2.0 ** (e + 1))
    A[13] = np.float32(2.0 ** e * (1 + 2.0 ** (-39 - e)))
    B[:, 15] = np.float32(2.0 ** e * (1 + 2.0 ** (-39 - e)))
    extra = [_pair(9711, 130, 70, 40)] if table else ()
    C = _grouped(mmlib, A, B, mmlib.MM_MODE_SPLIT_BF16X3, extra)
    err, _ = full_errors(C, A, B)
    assert err.max() <= oracle.tolerance(m, "f32")


@pytest.mark.parametrize("m", [1, 8, 16])
def test_few_k_take_three_parts(mmlib, m):
    A, B = _pair(9721, 300, m, 260)
    assert np.array_equal(_grouped(mmlib, A, B, mmlib.MM_MODE_SPLIT_BF16X3),
                          _grouped(mmlib, A, B, mmlib.MM_MODE_SPLIT_BF16X6))


@pytest.mark.parametrize("m,low", [(17, -28), (63, -28), (64, -30), (700, -30)])
def test_low_end(mmlib, m, low):
    """An entry at the window's end (2^-14, from m = 64 on 2^-16, after 2^14) keeps
    the fp16 form, one just below it gives the three-part form's bits."""
    A, B = _pair(9731, 300, m, 260)
    six = lambda: _grouped(mmlib, A, B, mmlib.MM_MODE_SPLIT_BF16X6)
    three = lambda: _grouped(mmlib, A, B, mmlib.MM_MODE_SPLIT_BF16X3)
    A[217, m - 1] = 2.0 ** low
    assert not np.array_equal(three(), six())
    A[217, m - 1] = np.nextafter(np.float32(2.0 ** low), np.float32(0))
    assert np.array_equal(three(), six())
