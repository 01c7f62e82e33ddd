"""The float64 kernel at the edges of its work split: rows shorter than a 16-byte chunk, chunk and warp-part remainders,
the V at which a row goes from one block to a cluster of 2, 4 and 8, student, teacher and gradient rows on different
16-byte boundaries, more rows than resident blocks (rows taken over from launches that are cancelled), warps whose
first elements lie so far below the row's maximum that pass "sums" is repeated; against the oracle."""
import numpy as np
import pytest
import torch

import oracle as O
import paper_2609_36601_b200 as P
from paper_2609_36601_b200 import synth
from parity import compare_rows, grad_check, oracle_inputs, to_np64

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _shift(x, off):
    """The same values in rows that start `off` elements after a 16-byte boundary."""
    n, V = x.shape
    ld = (V + 15) // 8 * 8
    y = torch.zeros(n * ld + 8, dtype=x.dtype, device=x.device)[off:off + n * ld].view(n, ld)[:, :V]
    y.copy_(x)
    return y


def _check(d, w, rows, offsets=(0, 0, 0)):
    s, t, g = (_shift(x, o) for x, o in zip((d["s"], d["t"], torch.zeros_like(d["s"])), offsets))
    prev = P.set_kernel(1)
    try:
        out, g = P.route_fwd_bwd(s, t, d["proposal"], w.eps, w.temperature, w.seed, grad_scale=0.25, dlogits=g)
    finally:
        P.set_kernel(prev)
    s64, t64 = oracle_inputs(d)
    ref = O.route(s64, t64, d["proposal"].cpu().numpy(), w.eps, w.temperature, w.seed, grad_scale=0.25, want_grad=True,
                  grad_dtype=w.dtype, rows=rows)
    compare_rows(out, ref, rows)
    # (eps and temperature are exact in float32) lambda is good to ~1e-10 before it is rounded to float32 (half an ulp below 1: 3e-8)
    assert np.abs(out["lambda"].cpu().numpy()[rows] - ref["lam"]).max() <= 4e-8
    same = out["corrected"].cpu().numpy()[rows] == ref["corrected"]
    tok = np.where(ref["corrected"] == 1, ref["teacher_top1"], ref["token"])[same]
    grad_check(to_np64(g)[rows][same], ref["grad"][same], w.dtype, tok)


@pytest.mark.parametrize("V,dtype,N", [(2, "bf16", 700), (3, "f32", 600), (7, "bf16", 5), (9, "bf16", 3), (17, "f32", 3),
                                       (255, "bf16", 450), (2047, "bf16", 3), (2049, "bf16", 3), (4097, "f32", 3),
                                       (8191, "bf16", 2), (8193, "f32", 2), (40001, "bf16", 2)])
@pytest.mark.parametrize("offsets", [(0, 0, 0), (3, 3, 3), (1, 2, 0)])
def test_split_edges(V, dtype, N, offsets):
    w = synth.Workload("t", N, V, dtype, 0.078125, 1.2, V > 100, 300 + V, 17, temperature=0.875)
    rows = list(range(N)) if N < 10 else list(range(0, N, 37)) + [N - 1]
    _check(synth.generate(w, DEV), w, rows, offsets)


@pytest.mark.parametrize("drop", [150.0, 2000.0])
def test_maximum_far_above_the_first_elements(drop):
    """Each warp's shift comes from its first 128 elements: here every one of them is `drop` nats below the peaks."""
    w = synth.Workload("t", 4, 6000, "f32", 0.125, 1.0, False, 41, 5)
    d = synth.generate(w, DEV)
    peaks = torch.arange(700, 6000, 750, device=DEV)
    low = torch.ones(6000, dtype=torch.bool, device=DEV)
    low[peaks] = False
    for k in ("s", "t"):
        d[k][:, low] -= drop
    d["proposal"][:] = peaks[:4].to(torch.int32)
    _check(d, w, list(range(4)))
