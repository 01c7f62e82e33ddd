"""Row-per-SM kernel with more rows than run at once: blocks take over rows whose block has not started yet.  Which block routes
a row must not show in its results: they are, to the bit, those of the same rows in calls that are small enough for every
row to have a block of its own from the start.  And the variants with two blocks to a row."""
import numpy as np
import pytest
import torch

import paper_2609_36601_b200 as P
from paper_2609_36601_b200 import binding as B, synth
import oracle as O
from parity import compare_rows, force_second_tier, grad_check, oracle_inputs, to_np64

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


# rows per SM at once: four up to V = 49152, two up to 98304, then one; one row more than that, one turn and a bit, many turns
@pytest.mark.parametrize("V,per_sm,extra", [(2048, 4, 1), (2056, 4, 37), (8192, 4, 2000), (49160, 2, 1), (65536, 2, 150), (98312, 1, 1), (98312, 1, 200)])
def test_rows_in_one_call_and_in_pieces(V, per_sm, extra):
    at_once = per_sm * torch.cuda.get_device_properties(0).multi_processor_count
    N = at_once + extra
    w = synth.Workload("t", N, V, "bf16", 0.08, 1.5, True, 800 + V % 97, 29)
    d = synth.generate(w, DEV)
    if V >= 8192:                       # (shorter rows have no place for it)
        force_second_tier(d, [0, N - 1])
    P.check()
    prev = P.set_kernel(3)              # pinned: pieces and the whole on the same variant
    try:
        for _ in range(2):              # (a call leaves nothing behind for the next)
            out, g = P.route_fwd_bwd(d["s"], d["t"], d["proposal"], w.eps, seed=w.seed)
            torch.cuda.synchronize()
            assert P.last_kernel() == 3 and P.check() == 0
            for r0 in range(0, N, at_once):
                r1 = min(N, r0 + at_once)
                po, pg = P.route_fwd_bwd(d["s"][r0:r1], d["t"][r0:r1], d["proposal"][r0:r1], w.eps, seed=w.seed, row_offset=r0)
                for k in out:
                    assert torch.equal(out[k][r0:r1], po[k]), (k, r0)
                assert torch.equal(g[r0:r1], pg), r0
    finally:
        P.set_kernel(prev)


# two blocks to a row, as dispatched: up to half as many rows as SMs in blocks of 512 threads, then of 256; the last and the first
# row of each rule, more rows than are in flight, segments of one step, ragged last steps, and the longest row
@pytest.mark.parametrize("V,N", [(20000, 74), (20000, 75), (24576, 148), (57344, 33), (98304, 74), (98312, 74), (151936, 148), (151936, 149), (100352, 447), (262144, 40), (262144, 150)])
@pytest.mark.parametrize("eps", [0.0, 0.1, 40.0])      # no evaluation, one or more, none (saturated): other barriers between the blocks
def test_two_blocks_per_row(V, N, eps):
    w = synth.Workload("t", N, V, "bf16", eps, 1.5, True, 900 + V % 97, 31, temperature=0.875)
    d = synth.generate(w, DEV)
    mask = (torch.arange(N, device=DEV) % 5 != 0).to(torch.uint8)
    d["s"][3, V - 1] = float("nan")
    d["proposal"][4] = V
    if eps == 0.1:
        force_second_tier(d, [6])
    P.check()
    out, g = P.route_fwd_bwd(d["s"], d["t"], d["proposal"], w.eps, w.temperature, w.seed, mask=mask, grad_scale=0.25)
    fwd = P.route_fwd(d["s"], d["t"], d["proposal"], w.eps, w.temperature, w.seed, mask=mask)
    torch.cuda.synchronize()
    assert P.last_kernel() == 3
    assert P.check() == 4                  # two flagged rows, two calls
    for k in out:
        assert torch.equal(out[k], fwd[k]), k
    assert int(out["row_status"][3]) & B.ROW_NONFINITE and int(out["row_status"][4]) & B.ROW_BAD_ID
    assert not g[3].any() and not g[4].any() and not g[5].any()
    rows = sorted({0, 1, 2, 6, N // 2, N - 2, N - 1})
    s64, t64 = oracle_inputs(d)
    ref = O.route(s64, t64, d["proposal"].cpu().numpy(), w.eps, w.temperature, w.seed, mask=mask.cpu().numpy(), grad_scale=0.25, want_grad=True,
                  grad_dtype=w.dtype, rows=rows)
    compare_rows(out, ref, rows)
    same = (out["corrected"].cpu().numpy()[rows] == ref["corrected"]) & (mask.cpu().numpy()[rows] != 0)
    tok = np.where(ref["corrected"] == 1, ref["teacher_top1"], ref["token"])[same]
    grad_check(to_np64(g)[rows][same], ref["grad"][same], w.dtype, tok)
    # the same rows with one block each: whatever the order of the sums, the same to the tolerance
    prev = P.set_kernel(3)
    try:
        one = P.route_fwd(d["s"], d["t"], d["proposal"], w.eps, w.temperature, w.seed, mask=mask)
    finally:
        P.set_kernel(prev)
    assert torch.equal(out["row_status"], one["row_status"]) and torch.equal(out["teacher_top1"], one["teacher_top1"])
    assert float((out["lambda"] - one["lambda"]).abs().max()) <= 1e-5 and float((out["tv"] - one["tv"]).abs().max()) <= 1e-5
