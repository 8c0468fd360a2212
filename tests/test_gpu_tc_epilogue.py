"""The tensor-core kernel's stores: whole sectors (rows of a multiple of eight
floats), half sectors (of four) and rows off both, through shared memory, with
scale exponents inside and outside of +-60, edges of tiles, and the epilogue in
place.  One entry does not depend on how its row is stored, and a power of two
on a row or column scales it exactly, so the results are compared bit for bit."""
import pytest
import torch

import synth
from gpu_util import dev

pytestmark = pytest.mark.gpu


def _at(x, k):
    """x, k floats past an allocation's start."""
    t = torch.zeros(x.numel() + k, device="cuda")
    t[k:] = x.flatten()
    return t[k:].view(*x.shape)


@pytest.mark.parametrize("p,off", [(264, 0), (264, 4), (264, 1), (260, 0), (260, 2), (257, 0), (130, 0), (7, 3)])
@pytest.mark.parametrize("e", [0, 60, 75])
def test_fp8_rows_and_columns(mmlib, p, off, e):
    n, m = 161, 384
    A, B = dev(synth.uniform_pm1(9901, (n, m))), dev(synth.uniform_pm1(9902, (m, 264)))
    ref = torch.empty(n, 264, device="cuda")
    assert mmlib.mm_gemm(n, m, 264, A, B, ref, mmlib.MM_F32, mmlib.MM_MODE_FP8) == mmlib.MM_OK
    A, B = A.clone(), B[:, :p].contiguous()
    A[3], B[:, p // 2] = A[3] * 2.0 ** e, B[:, p // 2] * 2.0 ** -e
    ref = ref[:, :p].clone()
    ref[3] *= 2.0 ** e
    ref[:, p // 2] *= 2.0 ** -e
    C = _at(torch.full((n, p), float("nan"), device="cuda"), off)
    assert mmlib.mm_gemm(n, m, p, A, B, C, mmlib.MM_F32, mmlib.MM_MODE_FP8) == mmlib.MM_OK
    assert torch.equal(C, ref)


@pytest.mark.parametrize("p,off", [(1608, 0), (1604, 0), (1601, 0), (1608, 2)])
@pytest.mark.parametrize("mode", ["MM_MODE_SPLIT_BF16X3", "MM_MODE_SPLIT_BF16X6"])
def test_epilogue_in_place(mmlib, mode, p, off):
    mm, n, m, md = mmlib, 1537, 2304, getattr(mmlib, mode)
    A, B = dev(synth.uniform_pm1(9911, (n, m))), dev(synth.uniform_pm1(9912, (m, p)))
    D = dev(synth.uniform_pm1(9913, (n, p)))
    C = _at(torch.zeros(n, p, device="cuda"), off)
    assert mm.mm_gemm(n, m, p, A, B, C, mm.MM_F32, md) == mm.MM_OK
    E = _at(D, off)
    assert mm.mm_gemm_axpby(n, m, p, 1.0, A, B, -1.0, E, E, mm.MM_F32, md) == mm.MM_OK
    assert torch.equal(E, C - D)
    assert mm.mm_gemm_axpby(n, m, p, -0.5, A, B, 0.0, None, E, mm.MM_F32, md) == mm.MM_OK
    assert torch.equal(E, -0.5 * C)
