"""FP64 products in 32 x 32 tiles (chosen where they take fewer rounds of the
SMs than 64 x 64 ones): the sums run in the same order, so integer products are
exact and a product equals its rows computed apart, whichever tile each takes;
edges of both tile sizes, one slice of K and several, with the epilogue."""
import numpy as np
import pytest
import torch

import synth
from gpu_util import assert_full, dev, run_gemm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(1024, 70, 1024), (1000, 33, 1030), (832, 17, 833), (31, 300, 33),
                                   (65, 700, 97), (342, 1266, 192), (1, 129, 1)],
                         ids=lambda s: "x".join(map(str, s)))
def test_matches_the_oracle(mmlib, shape):
    n, m, p = shape
    A = synth.uniform_pm1_f64(9401, (n, m))
    B = synth.uniform_pm1_f64(9402, (m, p))
    assert_full(run_gemm(mmlib, A, B, mmlib.MM_MODE_DGEMM, f64=True), A, B, "f64")


def test_same_bits_in_either_tile(mmlib):
    """1024 x 40 x 1024 takes 32 x 32 tiles on 148..152 SMs, 2048 rows of it
    64 x 64 or 32 x 32 ones: the shared rows agree bit for bit."""
    n, m, p = 1024, 40, 1024
    A = synth.uniform_pm1_f64(9403, (3 * n, m))
    B = synth.uniform_pm1_f64(9404, (m, p))
    part = run_gemm(mmlib, A[:n], B, mmlib.MM_MODE_DGEMM, f64=True)
    for k in (2, 3):
        whole = run_gemm(mmlib, A[:k * n], B, mmlib.MM_MODE_DGEMM, f64=True)
        assert np.array_equal(whole[:n], part)


def test_epilogue_in_place(mmlib):
    n, m, p = 1001, 50, 1023
    A, B = dev(synth.uniform_pm1_f64(9405, (n, m))), dev(synth.uniform_pm1_f64(9406, (m, p)))
    D = dev(synth.uniform_pm1_f64(9407, (n, p)))
    C = torch.empty_like(D)
    assert mmlib.mm_gemm(n, m, p, A, B, C, mmlib.MM_F64, mmlib.MM_MODE_DGEMM) == 0
    E = D.clone()
    assert mmlib.mm_gemm_axpby(n, m, p, 1.0, A, B, -1.0, E, E, mmlib.MM_F64, mmlib.MM_MODE_DGEMM) == 0
    assert torch.equal(E, C - D)
