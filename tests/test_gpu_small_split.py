"""The smallest products of the split modes run on the CUDA cores: MM_MODE_SIMT's
bits, plain and with the epilogue, up to the line, and within the tolerance on
both sides of it."""
import pytest
import torch

import synth
from gpu_util import assert_full, dev, run_gemm

pytestmark = pytest.mark.gpu

MODES = ["MM_MODE_SPLIT_BF16X3", "MM_MODE_SPLIT_BF16X6"]


@pytest.mark.parametrize("shape", [(1, 4, 4), (64, 512, 64), (256, 256, 256), (128, 4096, 128), (64, 16384, 64),
                                   (33, 2052, 20)], ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("mode", MODES)
def test_simt_bits(mmlib, shape, mode):
    mm, (n, m, p), md = mmlib, shape, getattr(mmlib, mode)
    A, B = dev(synth.uniform_pm1(9991, (n, m))), dev(synth.uniform_pm1(9992, (m, p)))
    D = dev(synth.uniform_pm1(9993, (n, p)))
    out = [torch.full((n, p), float("nan"), device="cuda") for _ in range(2)]
    for C, k in zip(out, (md, mm.MM_MODE_SIMT)):
        assert mm.mm_gemm(n, m, p, A, B, C, mm.MM_F32, k) == mm.MM_OK
    assert torch.equal(*out)
    E = D.clone()
    assert mm.mm_gemm_axpby(n, m, p, 1.0, A, B, -1.0, E, E, mm.MM_F32, md) == mm.MM_OK
    assert torch.equal(E, out[1] - D)


@pytest.mark.parametrize("shape", [(448, 384, 608), (480, 384, 608), (64, 32768, 64), (96, 32768, 64)],
                         ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("mode", MODES)
def test_both_sides_of_the_line(mmlib, shape, mode):
    n, m, p = shape
    A, B = synth.uniform_pm1(9995, (n, m)), synth.uniform_pm1(9996, (m, p))
    assert_full(run_gemm(mmlib, A, B, getattr(mmlib, mode)), A, B, "f32")
