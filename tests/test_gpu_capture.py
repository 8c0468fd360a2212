"""Split products under stream capture: a captured call allocates nothing once
its scratch is there, whichever call made it, and replays follow their operands."""
import pytest
import torch

import synth
from gpu_util import dev

pytestmark = pytest.mark.gpu


def _pair(seed, n, m, p):
    return dev(synth.uniform_pm1(seed, (n, m))), dev(synth.uniform_pm1(seed + 1, (m, p)))


def _capture(mm, n, m, p, A, B, C, stream):
    g = torch.cuda.CUDAGraph(keep_graph=True)
    torch.cuda.synchronize()
    with torch.cuda.graph(g, stream=stream):
        st = mm.mm_gemm_async(n, m, p, A, B, C, mm.MM_F32, mm.MM_MODE_SPLIT_BF16X3, stream)
    assert st == mm.MM_OK, mm.mm_strerror(st)
    g.instantiate()
    return g


@pytest.mark.parametrize("warm", ["grouped", "single", "host"])
def test_single_product_after_a_warm_up(mmlib, warm):
    """The library is fresh; a table of products, the product itself or a larger one
    with host operands makes the scratch, then the product is captured."""
    mm = mmlib
    n, m, p = 2600, 640, 2600
    A, B = _pair(9901, n, m, p)
    A2, B2 = _pair(9903, n, m, p)
    want = [torch.empty(n, p, device="cuda") for _ in range(2)]
    for (a, b), c in zip(((A, B), (A2, B2)), want):
        assert mm.mm_gemm(n, m, p, a, b, c, mm.MM_F32, mm.MM_MODE_SPLIT_BF16X3) == mm.MM_OK
    mm.mm_shutdown()
    assert mm.mm_init(device=0) == mm.MM_OK
    C = torch.zeros(n, p, device="cuda")
    X = torch.zeros(n, p, device="cuda")
    md = mm.MM_MODE_SPLIT_BF16X3
    if warm == "grouped":
        assert mm.mm_gemm_grouped([(n, m, p, A, B, C), (n, m, p, A, B, X)], mm.MM_F32, md) == mm.MM_OK
    elif warm == "single":
        assert mm.mm_gemm(n, m, p, A, B, C, mm.MM_F32, md) == mm.MM_OK
    else:
        h = [torch.zeros(r, c) for r, c in ((2 * n, m), (m, p), (2 * n, p))]
        assert mm.mm_gemm(2 * n, m, p, *h, mm.MM_F32, md) == mm.MM_OK
    s = torch.cuda.Stream()
    g = _capture(mm, n, m, p, A, B, X, s)
    A1, B1 = A.clone(), B.clone()
    for k in (0, 1, 1, 0):
        A.copy_((A1, A2)[k])
        B.copy_((B1, B2)[k])
        X.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(X, want[k])
        # an eager call between the replays
        assert mm.mm_gemm(n, m, p, A2, B2, C, mm.MM_F32, md) == mm.MM_OK
        assert torch.equal(C, want[1])
