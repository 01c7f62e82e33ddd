"""Where a call goes from one form of a kernel to the next: cluster kernel with 1, 2, 4, 8 and 16 CTAs per row, the
row-per-SM kernel with one, two or four rows per SM by the number of rows, the float64 kernel with one to eight blocks
per row, the lm-head GEMM with one CTA or two per
tile, proposals with one to eight blocks per row, slices whose maxima lie behind lower logits.  Against the oracle; float outputs and decisions at the tolerances of the parity tests."""
import numpy as np
import pytest
import torch

import oracle as O
import paper_2609_36601_b200 as P
from paper_2609_36601_b200 import synth
from paper_2609_36601_b200.vshard import route_vocab_sharded_local, split_columns
from parity import bf16_ulp, compare_rows, grad_check, oracle_inputs, to_np64

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _check(w, rows, kernel, used):
    d = synth.generate(w, DEV)
    prev = P.set_kernel(kernel)
    try:
        out, g = P.route_fwd_bwd(d["s"], d["t"], d["proposal"], w.eps, w.temperature, w.seed, grad_scale=0.25)
        torch.cuda.synchronize()
        assert P.last_kernel() == used
    finally:
        P.set_kernel(prev)
    s64, t64 = oracle_inputs(d)
    ref = O.route(s64, t64, d["proposal"].cpu().numpy(), w.eps, w.temperature, w.seed, grad_scale=0.25, want_grad=True,
                  grad_dtype=w.dtype, rows=rows)
    compare_rows(out, ref, rows)
    same = out["corrected"].cpu().numpy()[rows] == ref["corrected"]
    tok = np.where(ref["corrected"] == 1, ref["teacher_top1"], ref["token"])[same]
    grad_check(to_np64(g)[rows][same], ref["grad"][same], w.dtype, tok)


# pinned, the number of CTAs goes by V alone (1, 1, 2, 4, 4, 8, 8); rows end in chunk remainders, and the last CTA's slice
# is short or (8200: a chunk more than 4 x 2048) all but one chunk of a thread's share is empty
@pytest.mark.parametrize("V,N", [(2048, 5), (4088, 5), (4096, 5), (8200, 5), (16376, 4), (16384, 4), (163840, 2)])
def test_cluster_sizes_by_v(V, N):
    _check(synth.Workload("t", N, V, "bf16", 0.125, 1.5, True, 401, 51, temperature=0.875), list(range(N)), 2, 2)


# as dispatched: 16 CTAs per row up to 18 rows (148 SMs), 8 from 19 on; the shortest and the longest row of the rule
@pytest.mark.parametrize("V,N", [(32768, 1), (32768, 18), (32776, 19), (65528, 32), (151936, 9), (163840, 18), (163840, 32)])
def test_cluster_sizes_by_rows(V, N):
    _check(synth.Workload("t", N, V, "bf16", 0.125, 1.5, True, 402, 52), sorted({0, N // 2, N - 1}), 0, 2)


# the last row that fits a turn and the first that does not, for one, two and four rows per SM
@pytest.mark.parametrize("V", [8192, 16384, 30008, 49152])
@pytest.mark.parametrize("N", [148, 149, 296, 297, 592, 593])
def test_rows_per_sm_by_rows(V, N):
    _check(synth.Workload("t", N, V, "bf16", 0.125, 1.5, True, 403, 53), [0, N // 2, N - 1], 0, 3)


# the float64 kernel with one, two, four and eight blocks per row, by V and, at the last call size that is resident at once
# (444 bf16 or 592 fp32 blocks on 148 SMs) and the first that is not, by the number of rows
@pytest.mark.parametrize("V,N,dtype", [(4095, 5, "f32"), (4096, 5, "f32"), (8191, 3, "bf16"), (8193, 3, "f32"), (16387, 3, "bf16"),
                                       (16384, 74, "f32"), (16384, 75, "f32"), (9001, 111, "bf16"), (9001, 112, "bf16"),
                                       (5001, 222, "bf16"), (5001, 223, "bf16"), (4097, 445, "bf16"), (4100, 593, "f32")])
def test_float64_blocks_per_row(V, N, dtype):
    _check(synth.Workload("t", N, V, dtype, 0.125, 1.5, True, 405, 55, temperature=0.875), sorted({0, 1, N // 2, N - 1}), 0, 1)


@pytest.mark.parametrize("N", [1, 127, 128, 129, 255, 256, 257, 511, 513])
@pytest.mark.parametrize("V", [264, 4096])
def test_lmhead_tiles_by_rows(N, V):
    d = 72
    gen = torch.Generator(device=DEV).manual_seed(N)
    h = torch.randn((N, d), generator=gen, device=DEV).to(torch.bfloat16)
    w = (torch.randn((V, d), generator=gen, device=DEV) * 0.25).to(torch.bfloat16)
    logits, row_max, lse = P.lmhead_lse(h, w, 1.0)
    h64, w64 = to_np64(h), to_np64(w)
    ref, _, _ = O.lmhead_lse(h64, w64, 1.0)
    got = to_np64(logits)
    # a bf16 step, plus the float32 accumulation of d products: d 2^-24 of the sum of their magnitudes, here under 2^-17 of it
    assert np.all(np.abs(got - ref) <= bf16_ulp(ref) * 1.0000001 + 2.0 ** -17 * (np.abs(h64) @ np.abs(w64).T))
    m = got.max(axis=1)
    own = m + np.log(np.exp(got - m[:, None]).sum(axis=1))
    assert np.array_equal(row_max.cpu().numpy().astype(np.float64), m)
    assert np.max(np.abs(lse.cpu().numpy() - own)) <= 2e-6 * (1 + np.max(np.abs(own)))


# one, two, four and eight blocks per row; a thread's groups of eight logits paired, with one left over, with a partial one
@pytest.mark.parametrize("V,N", [(2048, 3), (4088, 149), (4104, 3), (6147, 3), (32008, 70), (30003, 30), (24008, 9), (40003, 18)])
@pytest.mark.parametrize("dtype", ["bf16", "f32"])
def test_proposal_blocks_per_row(V, N, dtype):
    s = (torch.randn((N, V), generator=torch.Generator(device=DEV).manual_seed(V), device=DEV) * 2).to(torch.bfloat16 if dtype == "bf16" else torch.float32)
    x = P.sample_proposal(s, 0.75, 29).cpu().numpy()
    rows = sorted({0, 1, N // 2, N - 1})
    ref, gaps = O.sample_proposal(to_np64(s), 0.75, 29, rows=rows)
    assert np.array_equal(x[rows][gaps >= 1e-12], ref[gaps >= 1e-12])     # float64 keys: a few ulp of ~100


# slices whose first 1024 logits lie `drop` nats below the others.  (Not far below: KL is a difference of terms of lambda D, D
# the distance of the two models' logits, whose float32 sums leave 2^-23 D of it, as measured at D = 100, where that passes
# the tolerance of 1e-5.)
@pytest.mark.parametrize("drop", [30.0, 60.0])
@pytest.mark.parametrize("sides", ["st", "s", "t"])
def test_slices_whose_first_logits_are_low(drop, sides):
    w = synth.Workload("t", 6, 8000, "bf16", 0.125, 1.0, False, 404, 54)
    d = synth.generate(w, DEV)
    for k in sides:
        for c in (0, 4000):
            d[k][:, c:c + 1024] -= drop
    d["proposal"][:] = torch.arange(1500, 1506, device=DEV, dtype=torch.int32)
    out, gs, _ = route_vocab_sharded_local([(d["s"][:, a:a + n], d["t"][:, a:a + n], a) for a, n in split_columns(8000, 2)], 8000,
                                           d["proposal"], w.eps, w.temperature, w.seed, grad_scale=0.5)
    s64, t64 = oracle_inputs(d)
    ref = O.route(s64, t64, d["proposal"].cpu().numpy(), w.eps, w.temperature, w.seed, grad_scale=0.5, want_grad=True,
                  grad_dtype=w.dtype)
    compare_rows(out, ref)
    same = out["corrected"].cpu().numpy() == ref["corrected"]
    tok = np.where(ref["corrected"] == 1, ref["teacher_top1"], ref["token"])[same]
    grad_check(to_np64(torch.cat(gs, dim=1))[same], ref["grad"][same], w.dtype, tok)


# The sums of a slice are taken under its own maxima wherever these lie, so that the exponent argument of the largest terms is
# exact: a block of 1024 logits (a chunk for every thread) 40 nats below the others may come first or last, to the bit.  Its
# terms, below 2^-57 of the largest, vanish in every thread's sum beside the others, which lie within 2^-25 of it; under shifts
# taken from a slice's first logits the arguments, and with them the log-sum-exps, would move by some 1e-7.
@pytest.mark.parametrize("sides", ["st", "s", "t"])
def test_sums_do_not_depend_on_where_the_maxima_lie(sides):
    V, N, world = 32768, 32, 4
    w = synth.Workload("t", N, V, "bf16", 0.125, 1.0, False, 406, 56)
    d = synth.generate(w, DEV)
    got = []
    for shift in (0, -1024):
        rows = {k: d[k].float().clamp(-8.0, 8.0).view(N, world, V // world) for k in "st"}
        for k in sides:
            rows[k][:, :, :1024] -= 40.0
        s, t = (torch.roll(rows[k], shift, dims=2).reshape(N, V).to(torch.bfloat16) for k in "st")
        state = []
        route_vocab_sharded_local([(s[:, a:a + n], t[:, a:a + n], a) for a, n in split_columns(V, world)], V, d["proposal"], w.eps,
                                  w.temperature, w.seed, state_out=state)
        got.append(state[0][:, [dict(s=5, t=6)[k] for k in sides]])          # the log-sum-exps of the lowered rows
    assert torch.equal(got[0], got[1])
