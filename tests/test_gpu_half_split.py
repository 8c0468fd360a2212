"""The fp16 form of the split path (inner dimensions below 2237): products
whose magnitudes fit the fp16 window meet the tolerance against the oracle at
the edges of tiles and K blocks, whatever their common scale; products they do
not fit, by the sample or by a single entry, give the three-part form's bits
(MM_MODE_SPLIT_BF16X6, which never takes fp16 parts), alone and in a table."""
import numpy as np
import pytest
import torch

import oracle
import synth
from gpu_util import dev, full_errors

pytestmark = pytest.mark.gpu


def _grouped(mm, probs, mode):
    """The products of (A, B) pairs through one grouped call (the packed path)."""
    outs = [torch.full((A.shape[0], B.shape[1]), float("nan"), device="cuda") for A, B in probs]
    tab = [(A.shape[0], A.shape[1], B.shape[1], dev(A), dev(B), C) for (A, B), C in zip(probs, outs)]
    assert mm.mm_gemm_grouped(tab, mm.MM_F32, mode) == 0
    return [C.cpu().numpy() for C in outs]


def _pair(seed, n, m, p):
    return synth.uniform_pm1(seed, (n, m)), synth.uniform_pm1(seed + 1, (m, p))


@pytest.mark.parametrize("shape", [(1, 1, 1), (127, 63, 129), (128, 64, 128), (129, 65, 127), (257, 2236, 4),
                                   (300, 191, 260), (5, 640, 1030)], ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("scale", [0, 40, -60])
def test_tile_edges_and_scales(mmlib, shape, scale):
    """A by 2^scale, B by 2^-scale / 2^(scale / 2): one exponent an operand."""
    A, B = _pair(9001, *shape)
    A, B = np.ldexp(A, scale), np.ldexp(B, -(scale // 2))
    C = _grouped(mmlib, [(A, B)], mmlib.MM_MODE_SPLIT_BF16X3)[0]
    e, _ = full_errors(C, A, B)
    assert e.max() <= oracle.tolerance(shape[1], "f32")


@pytest.mark.parametrize("what", ["wide", "one_large", "one_small", "infinite", "rows"])
def test_outside_the_window_gives_the_three_part_bits(mmlib, what):
    n, m, p = 260, 700, 390
    A, B = _pair(9101, n, m, p)
    if what == "wide":  # the sample sees the spread
        A = synth.pow2_real(9103, (n, m))
    elif what == "one_large":  # one entry in 182,000, which a sample of 256 misses
        A[17, 333] = 2.0 ** 40
    elif what == "one_small":
        B[555, 3] = 2.0 ** -37
    elif what == "infinite":
        B[11, 200] = np.inf
    else:  # rows far apart: scaled in the three-part form
        A = np.ldexp(A, synth.row_scale_exponents(9104, n)[:, None]).astype(np.float32)
    C3 = _grouped(mmlib, [(A, B)], mmlib.MM_MODE_SPLIT_BF16X3)[0]
    C6 = _grouped(mmlib, [(A, B)], mmlib.MM_MODE_SPLIT_BF16X6)[0]
    assert np.array_equal(C3, C6, equal_nan=True)
    if what != "infinite":
        e, _ = full_errors(C3, A, B)
        assert e.max() <= oracle.tolerance(m, "f32")


def test_table_of_both_forms_equals_the_single_calls(mmlib):
    """Products of both forms and of both split kinds in one table, one of
    them with a single entry outside the window; C odd-sized (plain stores)
    beside C with a tensor map."""
    probs = [_pair(9201, 130, 300, 132), _pair(9203, 200, 640, 77), _pair(9205, 64, 2304, 96),
             _pair(9207, 300, 65, 260), (np.zeros((40, 70), np.float32), synth.uniform_pm1(9209, (70, 33)))]
    probs[1][0][100, 5] = 2.0 ** 30
    probs[3] = (synth.pow2_real(9211, (300, 65)), probs[3][1])
    outs = _grouped(mmlib, probs, mmlib.MM_MODE_SPLIT_BF16X3)
    for (A, B), C in zip(probs, outs):
        assert np.array_equal(C, _grouped(mmlib, [(A, B)], mmlib.MM_MODE_SPLIT_BF16X3)[0])
        e, _ = full_errors(C, A, B)
        assert e.max() <= oracle.tolerance(A.shape[1], "f32")


@pytest.mark.parametrize("p", [260, 261])
def test_split_tail_and_epilogue(mmlib, p):
    """A product of one partial wave whose K loop is split (tail plan), with
    C = alpha A.B + beta D through the tiled and the plain stores: the
    product's bits combined once."""
    n, m = 2600, 2100
    A, B = _pair(9301, n, m, p)
    D = synth.uniform_pm1(9303, (n, p))
    st, _, _, split_s = mmlib.mm_tune_query_tail(n, m, p)
    assert st == 0 and split_s > 1
    dA, dB, dD = dev(A), dev(B), dev(D)
    C = torch.full((n, p), float("nan"), device="cuda")
    E = torch.full((n, p), float("nan"), device="cuda")
    mode = mmlib.MM_MODE_SPLIT_BF16X3
    assert mmlib.mm_gemm_grouped([(n, m, p, dA, dB, C)], mmlib.MM_F32, mode) == 0
    assert mmlib.mm_gemm_axpby(n, m, p, 1.0, dA, dB, -1.0, dD, E, mmlib.MM_F32, mode) == 0
    e, _ = full_errors(C.cpu().numpy(), A, B)
    assert e.max() <= oracle.tolerance(m, "f32")
    assert torch.equal(E, C - dD)


@pytest.mark.parametrize("shape", [(1024, 1024, 1024), (640, 1280, 768)], ids=lambda s: "x".join(map(str, s)))
def test_wide_products_keep_short_sums(mmlib, shape):
    """Magnitudes over 40 binades take three bf16 parts; products that the fused
    kernel's plan covers add them every 64 K, so that a sum's error stays that of
    m / 64 roundings to nearest and of 24 truncations within a block: 2^-24
    (sqrt(m / 64) + 24 / sqrt(m / 64)) of the result's norm, doubled here (one sum
    over K loses 3.7e-6)."""
    n, m, p = shape
    g = torch.Generator(device="cuda").manual_seed(77)
    spread = lambda r, c: (torch.rand(r, c, device="cuda", generator=g) * 2 - 1) * torch.exp2(
        torch.randint(-20, 21, (r, c), device="cuda", generator=g).float())
    A, B = spread(n, m), spread(m, p)
    C = torch.empty(n, p, device="cuda")
    assert mmlib.mm_tune_query_splitk(n, m, p)[2] > 0
    assert mmlib.mm_gemm(n, m, p, A, B, C, mmlib.MM_F32, mmlib.MM_MODE_SPLIT_BF16X3) == mmlib.MM_OK
    E = A.double() @ B.double()
    b = (m / 64) ** 0.5
    assert ((C.double() - E).norm() / E.norm()).item() <= 2 * 2.0 ** -24 * (b + 24 / b)
