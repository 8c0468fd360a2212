"""Which kernel an under-filled product of the split modes runs on, by its fused
plan: slices of eight K blocks take the packed form in MM_MODE_SPLIT_BF16X3 for
m < 2237, shorter ones and MM_MODE_SPLIT_BF16X6 the fused kernel; the packed form's
sums are no further off there than the fused kernel's."""
import pytest
import torch

from gpu_util import fused_slices

pytestmark = pytest.mark.gpu


def _launches(mm, kernels, call):
    torch.cuda.synchronize()  # mm_gemm runs on the library's own stream
    mm.mm_trace_reset()
    assert mm.mm_trace_enable(True) == 0
    try:
        call()
        return [mm.mm_trace_read(k)[1] for k in kernels]
    finally:
        mm.mm_trace_enable(False)
        mm.mm_trace_reset()


# (n, m, p), slices of the plan, whether they have eight K blocks: two to four
# slices, the ends of each range of m and the tiles' edges
CASES = [((1024, 1024, 1024), 2, True), ((960, 900, 960), 2, True), ((1024, 896, 1024), 2, False),
         ((896, 1352, 896), 3, True), ((896, 1344, 896), 3, False),
         ((768, 2048, 768), 4, True), ((770, 1860, 640), 4, True), ((768, 1792, 768), 4, False)]


@pytest.mark.parametrize("shape,slices,longest", CASES, ids=lambda v: "x".join(map(str, v)) if isinstance(v, tuple) else None)
@pytest.mark.parametrize("wide", [False, True], ids=["uniform", "wide"])
def test_long_slices(mmlib, shape, slices, longest, wide):
    mm, (n, m, p) = mmlib, shape
    assert fused_slices(mm, n, m, p) == slices
    assert (-(-(-(-m // 64)) // slices) >= 8) == longest
    g = torch.Generator(device="cuda").manual_seed(n + m)

    def values(r, c):
        x = torch.rand(r, c, device="cuda", generator=g) * 2 - 1
        return x * torch.exp2(torch.randint(-20, 21, (r, c), device="cuda", generator=g).float()) if wide else x

    A, B = values(n, m), values(m, p)
    exact = A.double() @ B.double()
    err = {}
    for mode, packed in (("MM_MODE_SPLIT_BF16X3", longest), ("MM_MODE_SPLIT_BF16X6", False)):
        C = torch.full((n, p), float("nan"), device="cuda")
        got = _launches(mm, ("split_tc", "fused_tc"),
                        lambda: mm.mm_gemm(n, m, p, A, B, C, mm.MM_F32, getattr(mm, mode)))
        assert got == ([1, 0] if packed else [0, 1])
        err[mode] = ((C.double() - exact).norm() / exact.norm()).item()
    # the same terms, in sums as long: one part in twenty for their order
    assert err["MM_MODE_SPLIT_BF16X3"] <= 1.05 * err["MM_MODE_SPLIT_BF16X6"]
