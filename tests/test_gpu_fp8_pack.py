"""FP8 operands as they are packed, in quarters of a tile (32 rows of A, 64
columns of B) by 128 values of K: every product against an FP64 product of the
operands rounded to e4m3 with the documented power-of-two factors (the block's
own where it lies two or more binades below its row or column, else the
whole row's), at the edges of quarters, tiles and K blocks, aligned and not."""
import pytest
import torch

import synth
from gpu_util import dev

pytestmark = pytest.mark.gpu


def _rounded(X):
    """X (rows by K) with each (row, 128 of K) block rounded to e4m3 at its factor."""
    n, m = X.shape
    P = torch.nn.functional.pad(X, (0, -m % 128)).view(n, -1, 128)
    top = lambda v: torch.frexp(v)[1].to(torch.float64) - 1 - 7  # floor(log2) - 7
    blk, row = P.abs().amax(2, keepdim=True), P.abs().amax((1, 2), keepdim=True)
    e = torch.where((blk == 0) | (top(blk) >= top(row) - 1), top(row).expand_as(blk), top(blk))
    s = torch.exp2(e)
    q = (P.double() / s).float().to(torch.float8_e4m3fn).double() * s
    return q.view(n, -1)[:, :m]


@pytest.mark.parametrize("shape", [(31, 127, 63), (32, 128, 64), (33, 129, 65), (96, 256, 192), (129, 260, 257),
                                   (160, 383, 321), (1, 1, 320), (257, 132, 1)], ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("off", [0, 1])
@pytest.mark.parametrize("spread", [0, 6])
def test_product_of_the_rounded_operands(mmlib, shape, off, spread):
    n, m, p = shape
    A, B = dev(synth.uniform_pm1(9951, (n, m))), dev(synth.uniform_pm1(9952, (m, p)))
    A[:, m // 2:] *= 2.0 ** -spread
    B[:m // 3] *= 2.0 ** -spread
    a, b = torch.zeros(n * m + off, device="cuda"), torch.zeros(m * p + off, device="cuda")
    a[off:], b[off:] = A.flatten(), B.flatten()
    C = torch.full((n, p), float("nan"), device="cuda")
    assert mmlib.mm_gemm(n, m, p, a[off:].view(n, m), b[off:].view(m, p), C, mmlib.MM_F32,
                         mmlib.MM_MODE_FP8) == mmlib.MM_OK
    QA, QB = _rounded(A), _rounded(B.t().contiguous()).t()
    # products exact; m FP32 additions, a rounding a K block and the last one
    bound = (m + m // 128 + 4) * 2.0 ** -23 * (QA.abs() @ QB.abs())
    assert bool(((C.double() - QA @ QB).abs() <= bound).all())
