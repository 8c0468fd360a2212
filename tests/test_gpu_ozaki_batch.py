"""Emulated FP64 requests that the serving loop launches together: each has the
bits of its own call, whatever shares its launches - another slice count, the
accuracy gate off, several K chunks, tiles of 128 and 256 columns, an empty
inner dimension, a product that the gate sends to the FP64 units, and more
requests than one launch takes."""
import pytest
import torch

import synth
from gpu_util import dev

pytestmark = pytest.mark.gpu


@pytest.fixture
def mm(mmlib):
    yield mmlib
    assert mmlib.mm_ozaki_slices(12) == mmlib.MM_OK
    assert mmlib.mm_ozaki_gate(1) == mmlib.MM_OK


def _operands(k, n, m, p, wide):
    A, B = synth.uniform_pm1_f64(9700 + k, (n, m)), synth.uniform_pm1_f64(9800 + k, (m, p))
    if wide:  # 2^-60 beside 1 in every row: the gate's bound fails
        A[:, ::2] *= 2.0 ** -60
        B[1::2, :] *= 2.0 ** -60
    return dev(A, torch.float64), dev(B, torch.float64)


SHAPES = [(33, 70, 40), (300, 517, 260), (1, 1, 1), (129, 5500, 70), (64, 11000, 33), (500, 128, 1026),
          (257, 1000, 300), (5, 0, 9), (96, 130, 512), (128, 128, 514)]


@pytest.mark.parametrize("copies", [1, 5])
def test_batch_has_the_bits_of_single_calls(mm, copies):
    jobs = []
    for k, (n, m, p) in enumerate(SHAPES * copies):
        S, gate, wide = (12, 8, 6, 12, 3)[k % 5], k % 7 != 3, k % 4 == 1
        A, B = _operands(k, n, m, p, wide)
        jobs.append((n, m, p, A, B, S, gate))
    big = dev(synth.uniform_pm1_f64(9699, (2048, 2048)), torch.float64)
    outs = [torch.full((j[0], j[2]), float("nan"), dtype=torch.float64, device="cuda") for j in jobs]
    spare = [torch.empty(2048, 2048, dtype=torch.float64, device="cuda") for _ in range(2)]
    torch.cuda.synchronize()
    ids = []
    for C in spare:  # keep the streams busy while the others queue up
        st, rid = mm.mm_submit(2048, 2048, 2048, big, big, C, mm.MM_F64, mm.MM_MODE_OZAKI)
        assert st == mm.MM_OK
        ids.append(rid)
    for (n, m, p, A, B, S, gate), C in zip(jobs, outs):
        assert mm.mm_ozaki_slices(S) == mm.MM_OK and mm.mm_ozaki_gate(int(gate)) == mm.MM_OK
        st, rid = mm.mm_submit(n, m, p, A, B, C, mm.MM_F64, mm.MM_MODE_OZAKI)
        assert st == mm.MM_OK
        ids.append(rid)
    for rid in ids:
        st, res, _, _ = mm.mm_wait(rid, 60.0)
        assert (st, res) == (mm.MM_OK, mm.MM_OK)
    assert torch.equal(spare[0], spare[1])
    for (n, m, p, A, B, S, gate), C in zip(jobs, outs):
        assert mm.mm_ozaki_slices(S) == mm.MM_OK and mm.mm_ozaki_gate(int(gate)) == mm.MM_OK
        ref = torch.full_like(C, float("nan"))
        assert mm.mm_gemm(n, m, p, A, B, ref, mm.MM_F64, mm.MM_MODE_OZAKI) == mm.MM_OK
        assert torch.equal(C, ref), (n, m, p, S, gate)
