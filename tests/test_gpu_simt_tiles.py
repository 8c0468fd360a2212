"""FP32 SIMT products in 32 x 32 and 64 x 64 tiles: whichever tile, cluster or
kernel a product takes, an entry is the sum of its K slices' ascending sums in
the plan's order.  A product of one slice gives the slices' bits, so the
expected result is put together from those, bit for bit, at tile edges, for
each way the slices are added, with 16-byte and 4-byte copies and the epilogue."""
import pytest
import torch

import synth
from gpu_util import dev

pytestmark = pytest.mark.gpu


def _gemm(mm, A, B):
    (n, m), p = A.shape, B.shape[1]
    C = torch.full((n, p), float("nan"), device="cuda")
    assert mm.mm_gemm(n, m, p, A, B, C, mm.MM_F32, mm.MM_MODE_SIMT) == mm.MM_OK
    return C


def _plan(mm, n, m, p):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    st, S, ks, _ = mm.mm_simt_plan(n, m, p, mm.MM_F32, sms)
    assert st == mm.MM_OK
    return (S, ks) if S > 0 else (1, m)


def _expected(mm, A, B, S, ks):
    """Slices of A and B as products of their own (one slice each: ks values),
    added in eight groups of consecutive slices."""
    m = A.shape[1]
    parts = []
    for z in range(S):
        a, b = A[:, z * ks:min(m, (z + 1) * ks)], B[z * ks:(z + 1) * ks]
        if a.shape[1] >= 256:  # would be cut again: in one pass below many rows
            pad = torch.zeros(4096, a.shape[1], device="cuda")
            pad[:a.shape[0]] = a
            wide = torch.zeros(a.shape[1], 2048, device="cuda")
            wide[:, :b.shape[1]] = b
            assert _plan(mm, 4096, a.shape[1], 2048)[0] == 1
            parts.append(_gemm(mm, pad, wide)[:a.shape[0], :b.shape[1]].contiguous())
        else:
            assert _plan(mm, a.shape[0], a.shape[1], b.shape[1])[0] == 1
            parts.append(_gemm(mm, a.contiguous(), b.contiguous()))
    G = min(8, S)
    total = None
    for g in range(G):
        acc = parts[g * S // G]
        for s in range(g * S // G + 1, (g + 1) * S // G):
            acc = acc + parts[s]
        total = acc if total is None else total + acc
    return total


@pytest.mark.parametrize("shape", [(31, 4, 33), (32, 128, 32), (33, 129, 31), (1, 255, 257), (256, 256, 256),
                                   (255, 383, 259), (100, 100, 100), (512, 512, 512), (63, 1024, 65),
                                   (300, 1100, 129), (768, 768, 770), (64, 4096, 64), (47, 3001, 130),
                                   (1152, 90, 1152), (1280, 77, 1281)], ids=lambda s: "x".join(map(str, s)))
def test_slices_bit_for_bit(mmlib, shape):
    n, m, p = shape
    A, B = dev(synth.uniform_pm1(9601, (n, m))), dev(synth.uniform_pm1(9602, (m, p)))
    S, ks = _plan(mmlib, n, m, p)
    C = _gemm(mmlib, A, B)
    if S > 1:
        assert torch.equal(C, _expected(mmlib, A, B, S, ks))
    E = A.double() @ B.double()
    bound = 2.0 ** -24 * (m + 2) * (A.double().abs() @ B.double().abs())
    assert bool(((C.double() - E).abs() <= bound).all())
    # unaligned operands: the same sums through 4-byte copies
    a, b = torch.zeros(n * m + 1, device="cuda"), torch.zeros(m * p + 3, device="cuda")
    a[1:], b[3:] = A.flatten(), B.flatten()
    assert torch.equal(C, _gemm(mmlib, a[1:].view(n, m), b[3:].view(m, p)))


@pytest.mark.parametrize("n", [1152, 1280])
def test_same_bits_as_the_large_tile(mmlib, n):
    """One pass over K in tiles of 32 or 64 and, as part of a larger product, of 128."""
    m = 70
    A, B = dev(synth.uniform_pm1(9611, (2048, m))), dev(synth.uniform_pm1(9612, (m, 2048)))
    whole = _gemm(mmlib, A, B)
    part = _gemm(mmlib, A[:n].contiguous(), B[:, :n].contiguous())
    assert torch.equal(part, whole[:n, :n])


@pytest.mark.parametrize("shape", [(65, 130, 96), (257, 300, 255), (256, 1024, 256), (70, 3000, 64),
                                   (1152, 40, 1152)], ids=lambda s: "x".join(map(str, s)))
def test_epilogue_in_place(mmlib, shape):
    mm, (n, m, p) = mmlib, shape
    A, B = dev(synth.uniform_pm1(9621, (n, m))), dev(synth.uniform_pm1(9622, (m, p)))
    D = dev(synth.uniform_pm1(9623, (n, p)))
    C, E = _gemm(mm, A, B), D.clone()
    assert mm.mm_gemm_axpby(n, m, p, 1.0, A, B, -1.0, E, E, mm.MM_F32, mm.MM_MODE_SIMT) == mm.MM_OK
    assert torch.equal(E, C - D)
