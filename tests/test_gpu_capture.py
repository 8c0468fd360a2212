"""Split products under stream capture: a captured call allocates nothing once
its scratch is there, whichever call made it, replays follow their operands, and no
call depends on what another one left in the words that start at zero."""
import ctypes

import pytest
import torch

import synth
from gpu_util import dev

pytestmark = pytest.mark.gpu


def _pair(seed, n, m, p):
    return dev(synth.uniform_pm1(seed, (n, m))), dev(synth.uniform_pm1(seed + 1, (m, p)))


def _capture(mm, n, m, p, A, B, C, stream, mode=None):
    g = torch.cuda.CUDAGraph(keep_graph=True)
    torch.cuda.synchronize()
    with torch.cuda.graph(g, stream=stream):
        st = mm.mm_gemm_async(n, m, p, A, B, C, mm.MM_F32, mm.MM_MODE_SPLIT_BF16X3 if mode is None else mode, stream)
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


@pytest.mark.parametrize("shape,first_call", [((256, 256, 256), True), ((64, 1100, 64), True), ((40, 100, 60), True),
                                              ((64, 16384, 64), False)], ids=lambda v: "x".join(map(str, v)) if isinstance(v, tuple) else None)
@pytest.mark.parametrize("mode", ["MM_MODE_SIMT", "MM_MODE_SPLIT_BF16X3"])
def test_small_products_in_a_cluster_need_no_scratch(mmlib, shape, first_call, mode):
    """Up to eight K slices are added within a cluster: such a product may be the
    library's first call and captured.  More slices need one call before."""
    mm, (n, m, p), md = mmlib, shape, getattr(mmlib, mode)
    A, B = _pair(9907, n, m, p)
    want, C = torch.empty(n, p, device="cuda"), torch.zeros(n, p, device="cuda")
    assert mm.mm_gemm(n, m, p, A, B, want, mm.MM_F32, md) == mm.MM_OK  # (loads the kernels, too)
    mm.mm_shutdown()
    assert mm.mm_init(device=0) == mm.MM_OK
    if not first_call:
        assert mm.mm_gemm(n, m, p, A, B, C, mm.MM_F32, md) == mm.MM_OK
    g = _capture(mm, n, m, p, A, B, C, torch.cuda.Stream(), md)
    C.zero_()
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(C, want)


class _Memset(ctypes.Structure):
    _fields_ = [("dst", ctypes.c_uint64), ("pitch", ctypes.c_size_t), ("value", ctypes.c_uint),
                ("elementSize", ctypes.c_uint), ("width", ctypes.c_size_t), ("height", ctypes.c_size_t)]


def _memsets(graph):
    """(address, bytes) of the memset nodes of a captured graph."""
    cu = ctypes.CDLL("libcuda.so.1")
    handle, count = ctypes.c_void_p(graph.raw_cuda_graph()), ctypes.c_size_t(0)
    assert cu.cuGraphGetNodes(handle, None, ctypes.byref(count)) == 0
    nodes = (ctypes.c_void_p * count.value)()
    assert cu.cuGraphGetNodes(handle, nodes, ctypes.byref(count)) == 0
    out = []
    for node in nodes:
        kind = ctypes.c_int(-1)
        assert cu.cuGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(kind)) == 0
        if kind.value == 2:  # CU_GRAPH_NODE_TYPE_MEMSET
            x = _Memset()
            assert cu.cuGraphMemsetNodeGetParams(ctypes.c_void_p(node), ctypes.byref(x)) == 0
            out.append((x.dst, x.elementSize * x.width * max(1, x.height)))
    return out


@pytest.mark.parametrize("m", [2100, 4096])
def test_replays_clear_the_tail_counters(mmlib, m):
    """The words that a replay needs at zero, a word at least for every tile that
    is split along K, are cleared by the graph itself: whatever an aborted launch
    left in them (all ones here), the next replay gives the product."""
    mm = mmlib
    n, p = 2600, 260
    st, tiles, split_from, split_s = mm.mm_tune_query_tail(n, m, p)
    assert st == mm.MM_OK and split_s > 1 and tiles - split_from > 16
    A, B = _pair(9911, n, m, p)
    want, C = torch.empty(n, p, device="cuda"), torch.zeros(n, p, device="cuda")
    assert mm.mm_gemm(n, m, p, A, B, want, mm.MM_F32, mm.MM_MODE_SPLIT_BF16X3) == mm.MM_OK
    g = _capture(mm, n, m, p, A, B, C, torch.cuda.Stream())
    cleared = _memsets(g)
    assert sum(size for _, size in cleared) >= 4 * (tiles - split_from)
    cu = ctypes.CDLL("libcuda.so.1")
    for _ in range(2):
        for at, size in cleared:
            assert cu.cuMemsetD32_v2(ctypes.c_uint64(at), ctypes.c_uint(1), ctypes.c_size_t(size // 4)) == 0
        torch.cuda.synchronize()
        C.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(C, want)


def test_products_in_turn_on_one_scratch(mmlib):
    """Products with and without split tiles, of both forms and sizes of their
    counters, one after the other: each call's words are clear again."""
    mm, md = mmlib, mmlib.MM_MODE_SPLIT_BF16X3
    shapes = [(2600, 2100, 260), (3000, 640, 3000), (2600, 4096, 260), (2600, 2100, 390), (2600, 2100, 260)]
    ops = [_pair(9921 + 2 * k, *s) for k, s in enumerate(shapes)]
    ops[3][0][5, 7] = 2.0 ** 60  # six products, scaled
    want = [torch.empty(n, p, device="cuda") for n, _, p in shapes]
    for (n, m, p), (A, B), W in zip(shapes, ops, want):
        mm.mm_shutdown()
        assert mm.mm_init(device=0) == mm.MM_OK
        assert mm.mm_gemm(n, m, p, A, B, W, mm.MM_F32, md) == mm.MM_OK
    outs = [torch.zeros_like(W) for W in want]
    for _ in range(3):
        for (n, m, p), (A, B), C in zip(shapes, ops, outs):
            C.zero_()
            assert mm.mm_gemm_async(n, m, p, A, B, C, mm.MM_F32, md, torch.cuda.current_stream()) == mm.MM_OK
        assert mm.mm_sync(torch.cuda.current_stream()) == mm.MM_OK
        for C, W in zip(outs, want):
            assert torch.equal(C, W)
