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


def _check(d, w, rows, offsets=(0, 0, 0), kernel=1):
    s, t, g = (_shift(x, o) for x, o in zip((d["s"], d["t"], torch.zeros_like(d["s"])), offsets))
    prev = P.set_kernel(kernel)
    try:
        out, g = P.route_fwd_bwd(s, t, d["proposal"], w.eps, w.temperature, w.seed, grad_scale=0.25, dlogits=g)
    finally:
        P.set_kernel(prev)
    s64, t64 = oracle_inputs(d)
    ref = O.route(s64, t64, d["proposal"].cpu().numpy(), w.eps, w.temperature, w.seed, grad_scale=0.25, want_grad=True,
                  grad_dtype=w.dtype, rows=rows)
    compare_rows(out, ref, rows)
    # (eps and temperature are exact in float32) at these radii lambda is good to ~1e-13 before it is rounded to float32 (half an ulp
    # below 1: 3e-8)
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


@pytest.mark.parametrize("N,V,dtype,layout", [(296, 1024, "f32", (1, 2)), (297, 1024, "f32", (1, 3)), (1100, 1024, "f32", (1, 3)),
                                              (148, 8000, "f32", (2, 2)), (149, 8000, "f32", (1, 2)), (148, 7999, "f32", (1, 2)),
                                              (222, 10000, "f32", (2, 3)), (223, 10000, "f32", (1, 2)), (99, 20000, "f32", (4, 3)),
                                              (100, 20001, "bf16", (4, 3)), (46, 64001, "f32", (8, 3)), (46, 64001, "bf16", (8, 3)),
                                              (47, 64001, "bf16", (8, 3)), (74, 16000, "f32", (2, 2)), (37, 32001, "f32", (4, 2)),
                                              (160, 151936, "f32", (2, 3)), (700, 50000, "f32", (2, 2)), (512, 151936, "f32", (4, 4)),
                                              (400, 2049, "bf16", (1, 3)), (700, 2049, "bf16", (1, 3)), (148, 8001, "bf16", (2, 2)),
                                              (37, 33001, "bf16", (4, 2))])
def test_layouts(N, V, dtype, layout):
    """Blocks per row and per SM as an unpinned call takes them on 148 SMs: either side of two blocks on each of them, of 4000
    elements a block, of what L2 holds, and calls of more rows than are resident, which go by the cost model."""
    w = synth.Workload("t", N, V, dtype, 0.0625, 1.2, True, 600 + N + V, 29, temperature=0.875)
    _check(synth.generate(w, DEV), w, sorted({0, 1, N // 2, N - 2, N - 1}), kernel=0)
    assert P.last_kernel() == 1
    if torch.cuda.get_device_properties(0).multi_processor_count == 148:
        assert P.last_layout()[:2] == layout


@pytest.mark.parametrize("N,V,dtype", [(33, 32000, "f32"), (34, 32000, "f32"), (37, 64000, "f32"), (37, 33001, "bf16"), (70, 16000, "f32"),
                                       (72, 16000, "f32"), (74, 40001, "bf16"), (104, 20000, "f32"), (111, 20000, "f32")])
def test_rows_of_a_few_clusters_are_resident_at_once(N, V, dtype):
    """Clusters of four and eight do not fill every SM: a call that is laid out in one turn of them has room for all its rows."""
    w = synth.Workload("t", N, V, dtype, 0.0625, 1.2, True, 700 + N + V, 31, temperature=0.875)
    _check(synth.generate(w, DEV), w, sorted({0, N // 2, N - 2, N - 1}), kernel=0)
    cs, k, resident = P.last_layout()
    assert P.last_kernel() == 1 and cs in (2, 4, 8) and k in (2, 3) and N <= resident


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


@pytest.mark.parametrize("V,dtype", [(9, "bf16"), (20, "f32"), (33, "bf16"), (600, "bf16"), (2049, "f32"), (32003, "bf16")])
@pytest.mark.parametrize("off", [1, 2, 3])
def test_argmax_ties(V, dtype, off):
    """The teacher's maximum several times over: among the elements before the row's first 16-byte boundary, in the chunks
    behind it (those of the same thread and of others) and in the elements after the last chunk.  The lowest index counts."""
    w = synth.Workload("t", 24, V, dtype, 0.125, 1.2, False, 320 + V, 18)
    d = synth.generate(w, DEV)
    top = d["t"].float().max() + 2.0
    head = 16 // d["t"].element_size() - off % (16 // d["t"].element_size())
    for r in range(w.N):
        at = [r % 2 * V // 2, r % (head + 1), head + r % 8, min(head + 8 * 32 + r % 8, V - 1), V - 1 - r % 3]
        for v in at[r % 3:]:
            d["t"][r, min(v, V - 1)] = top
    d["t"][0] = 1.0                                    # every element
    _check(d, w, list(range(w.N)), (off, (off * 3) % 8, 0))


@pytest.mark.parametrize("V,N,dtype,off", [(2, 5, "f32", 0), (5, 3, "bf16", 1), (1023, 4, "bf16", 3), (1024, 700, "f32", 0),
                                           (8191, 3, "bf16", 0), (8192, 3, "bf16", 2), (40003, 3, "f32", 1)])
@pytest.mark.parametrize("scale", [1.0, 40.0])
def test_proposal_edges(V, N, dtype, off, scale):
    """Gumbel-max by float32 bounds: partial last Philox block, unaligned rows, one block and a cluster per row, peaked
    rows (scale 40: the winner's Gumbel term is small, where the bound is loose)."""
    w = synth.Workload("t", N, V, dtype, 0.1, 1.0, V > 100, 500 + V, 23)
    s = _shift((synth.generate(w, DEV)["s"].float() * scale).to(w.torch_dtype), off)
    x = P.sample_proposal(s, 0.75, 23, row_offset=(1 << 32) - 2).cpu().numpy()
    rows = list(range(N)) if N < 10 else list(range(0, N, 41))
    ref, gaps = O.sample_proposal(to_np64(s), 0.75, 23, row_offset=(1 << 32) - 2, rows=rows)
    assert np.array_equal(x[rows][gaps >= 1e-12], ref[gaps >= 1e-12])     # float64 keys: a few ulp of ~100


def test_proposal_of_unusual_logits():
    """NaN and -inf are never drawn, +inf is (the first), a row of nothing else gives 0x7fffffff."""
    s = torch.randn(5, 9000, device=DEV)
    s[0, 5:] = float("-inf"); s[1, 7000] = s[1, 8000] = float("inf"); s[2, :] = float("nan"); s[3, ::2] = float("nan")
    s[4] = 3e38 + 0 * s[4]
    x = P.sample_proposal(s, 0.5, 1).cpu().numpy()
    ref, _ = O.sample_proposal(to_np64(s[4:5]), 0.5, 1, row_offset=4)
    assert x[0] < 5 and x[1] == 7000 and x[2] == 0x7fffffff and x[3] % 2 == 1
    assert x[4] == ref[0]
