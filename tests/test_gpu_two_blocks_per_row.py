"""Rows on two SMs, as dispatched.  Rows of more than 98304 elements in calls of up to a row per SM take two blocks of eight
warps; pinned they take one block of sixteen.  Both add the sums of the sixteen warps in the same order."""
import pytest
import torch

import oracle as O
import paper_2609_36601_b200 as P
from paper_2609_36601_b200 import binding as B, synth
from parity import MARGIN, force_second_tier, oracle_inputs, to_np64
from test_gpu_late_answers import check_rows, limited_call

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def spread_over_warps(d, V, seed):
    """Lowers each sixteenth of a row (a warp's part) by up to 80 nats, so that the warps' sums differ by many binary orders."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    part = torch.arange(V, device=DEV) // 256 * 16 // ((V + 255) // 256)
    off = -80.0 * torch.rand((d["s"].shape[0], 16), generator=gen, device=DEV) ** 2
    for k in ("s", "t"):
        d[k].copy_((d[k].float() + off[:, part]).to(torch.bfloat16))


@pytest.mark.parametrize("V", [98312, 131072, 151936])
@pytest.mark.parametrize("eps", [0.002, 0.1])
@pytest.mark.parametrize("apart", [False, True])
def test_pair_of_blocks_agrees_with_one_block_to_the_bit(V, eps, apart):
    N = torch.cuda.get_device_properties(0).multi_processor_count
    w = synth.Workload("pair", N, V, "bf16", eps, 1.5, True, 1200 + V % 97, 33)
    d = synth.generate(w, DEV)
    if apart:
        spread_over_warps(d, V, 5)
    out, g = P.route_fwd_bwd(d["s"], d["t"], d["proposal"], w.eps, seed=w.seed)
    assert P.last_kernel() == 3
    prev = P.set_kernel(3)
    try:
        one, g_one = P.route_fwd_bwd(d["s"], d["t"], d["proposal"], w.eps, seed=w.seed)
    finally:
        P.set_kernel(prev)
    torch.cuda.synchronize()
    for k in out:
        assert torch.equal(out[k], one[k]), k
    assert torch.equal(g, g_one)


# (blocks per row, blocks per SM), as dispatched and with the kernel pinned
@pytest.mark.parametrize("V,N,layout,pinned", [(8192, 100, (1, 2), (1, 4)), (8192, 2000, (1, 4), (1, 4)), (8192, 304, (1, 4), (1, 4)),
                                               (9200, 320, (1, 4), (1, 4)), (24000, 156, (1, 2), (1, 4)), (65536, 74, (2, 1), (1, 2)), (65536, 148, (2, 2), (1, 2)),
                                               (65536, 900, (1, 2), (1, 2)), (98304, 74, (2, 1), (1, 2)), (98312, 74, (2, 2), (1, 1)), (151936, 40, (2, 2), (1, 1)),
                                               (151936, 447, (2, 2), (1, 1)), (262144, 150, (2, 2), (1, 1))])
def test_layouts(V, N, layout, pinned):
    assert torch.cuda.get_device_properties(0).multi_processor_count == 148, "the shapes are chosen for 148 SMs"
    w = synth.Workload("layout", N, V, "bf16", 0.1, 1.5, True, 7, 7)
    d = synth.generate(w, DEV)
    for which, want in ((0, layout), (3, pinned)):
        prev = P.set_kernel(which)
        try:
            P.route_fwd(d["s"], d["t"], d["proposal"], w.eps, seed=w.seed)
            assert P.last_kernel() == 3 and P.last_rowsm_layout() == want, which
        finally:
            P.set_kernel(prev)
    prev = P.set_kernel(1)
    try:
        P.route_fwd(d["s"], d["t"], d["proposal"], w.eps, seed=w.seed)
        assert P.last_rowsm_layout() == (0, 0)
    finally:
        P.set_kernel(prev)
    torch.cuda.synchronize()


# three turns and more of rows that take other ways through the kernel, each after each: no evaluation (saturated), one or more,
# flagged (NaN, bad id), handed to the second tier, masked
@pytest.mark.parametrize("V,N", [(104000, 447), (151936, 600)])
def test_long_chains_on_the_pair(V, N):
    w = synth.Workload("chains", N, V, "bf16", 0.1, 1.5, True, 1300 + V % 97, 35)
    d = synth.generate(w, DEV)
    saturated, nan, bad, second = range(2, N, 5), range(3, N, 17), range(4, N, 19), range(5, N, 59)
    for r in saturated:
        d["t"][r] = d["s"][r]
    force_second_tier(d, list(second))
    for r in nan:
        d["s"][r, (r * 977) % V] = float("nan")
    for r in bad:
        d["proposal"][r] = -1 - r
    flagged = sorted(set(nan) | set(bad))
    mask = (torch.arange(N, device=DEV) % 7 != 0).to(torch.uint8)
    P.check()
    out, g = P.route_fwd_bwd(d["s"], d["t"], d["proposal"], w.eps, seed=w.seed, mask=mask, grad_scale=0.25)
    assert P.last_kernel() == 3 and P.last_rowsm_layout() == (2, 2)
    assert P.redo_count() >= len(set(second) - set(flagged))
    assert P.check() == len(flagged)
    prev = P.set_kernel(3)
    try:
        one, g_one = P.route_fwd_bwd(d["s"], d["t"], d["proposal"], w.eps, seed=w.seed, mask=mask, grad_scale=0.25)
        assert P.last_rowsm_layout() == (1, 1)
    finally:
        P.set_kernel(prev)
    torch.cuda.synchronize()
    P.check()
    assert torch.all(out["row_status"][flagged] & (B.ROW_NONFINITE | B.ROW_BAD_ID) != 0) and not g[flagged].any()
    for k in out:
        assert torch.equal(out[k], one[k]), k
    assert torch.equal(g, g_one)
    rows = [0, 1, 5, 7, N // 2, N - 2, N - 1]
    s64, t64 = oracle_inputs(d, rows)
    for i, r in enumerate(rows):
        ref = O.route_row(s64[i], t64[i], int(d["proposal"][r]), w.eps, 1.0, w.seed, r, int(mask[r]))
        assert abs(float(out["lambda"][r]) - ref["lam"]) <= 1e-5 and abs(float(out["tv"][r]) - ref["tv"]) <= 1e-5
        assert int(out["teacher_top1"][r]) == ref["teacher_top1"] and int(out["row_status"][r]) == ref["status"]


# a limit that every copy misses, and limits that some of a row's blocks miss and others do not
@pytest.mark.parametrize("V,N,layout", [(65536, 74, (2, 1)), (65536, 148, (2, 2)), (104000, 300, (2, 2)), (151936, 320, (2, 2))])
def test_expired_waits_on_two_blocks(V, N, layout):
    w = synth.Workload("limit", N, V, "bf16", 0.1, 1.5, True, 4100 + V % 97, 9)
    d = synth.generate(w, DEV)
    P.check()
    ref, g_ref = P.route_fwd_bwd(d["s"], d["t"], d["proposal"], w.eps, seed=w.seed)
    torch.cuda.synchronize()
    assert P.last_kernel() == 3 and P.last_rowsm_layout() == layout and P.check() == 0
    for limit in (2, 300, 800, 1500, 2500, 4000):
        late, out, g = limited_call(d, w, limit)
        assert limit > 2 or late.any(), "no wait ran out: the limit did not reach the kernel"
        check_rows(late, out, g, ref, g_ref)
    late, out, g = limited_call(d, w, 0)
    assert not late.any()
    check_rows(late, out, g, ref, g_ref)


def test_phase_clock_on_two_blocks():
    w = synth.Workload("clock", 300, 151936, "bf16", 0.05, 1.0, True, 77, 5)
    d = synth.generate(w, DEV)
    ref, g_ref = P.route_fwd_bwd(d["s"], d["t"], d["proposal"], w.eps, seed=w.seed)
    prev = P.set_phase_clock(True)
    try:
        out, g = P.route_fwd_bwd(d["s"], d["t"], d["proposal"], w.eps, seed=w.seed)
        assert P.last_rowsm_layout() == (2, 2)
        cycles = P.phase_cycles()
    finally:
        P.set_phase_clock(prev)
    assert cycles["rows"] == w.N                             # the rows' first blocks carry the clock
    passes, total = cycles["lse"] + cycles["solve"] + cycles["final"], sum(v for k, v in cycles.items() if k != "rows")
    assert 0.3 * total < passes < total and 1e4 < total / w.N < 4e5
    for k in ref:
        assert torch.equal(out[k], ref[k]), k
    assert torch.equal(g, g_ref)


def test_block_verification_with_early_out_on_the_pair():
    Bs, K, V = 2 * torch.cuda.get_device_properties(0).multi_processor_count + 4, 2, 151936
    w = synth.Workload("t", Bs * (K + 1), V, "bf16", 0.1, 1.5, True, 93, 23, K=K)
    d = synth.generate(w, DEV)
    force_second_tier(d, [5 * (K + 1), 30 * (K + 1) + 1])
    s3, t3 = d["s"].view(Bs, K + 1, V), d["t"].view(Bs, K + 1, V)
    draft = d["proposal"].view(Bs, K + 1)[:, :K].contiguous()
    s3[3, 1, 17] = float("nan")
    draft[20, 1] = V
    P.check()
    res = {}
    prev = P.set_spec_early_out(True)
    try:
        for on in (True, False):
            P.set_spec_early_out(on)
            res[on] = P.spec_verify(s3, t3, draft, w.eps, seed=w.seed)
            assert P.last_kernel() == 3 and P.last_rowsm_layout() == (2, 2)
            assert P.redo_count() >= 1 and (P.spec_positions_routed() > 0) == on
            P.check()
    finally:
        P.set_spec_early_out(prev)
    a, b = res[True], res[False]
    for k in ("n_accept", "next_token", "next_is_correction"):
        assert torch.equal(a[k], b[k]), k
    for k in a["per_pos"]:
        assert k == "loss" or torch.equal(a["per_pos"][k], b["per_pos"][k]), k
    assert int(a["n_accept"][3]) <= 1 and int(a["n_accept"][20]) <= 1
    for q in (0, 3, 5, 20, 30, Bs - 1):
        ref = O.spec_verify(to_np64(s3[q:q + 1]), to_np64(t3[q:q + 1]), draft[q:q + 1].cpu().numpy(), w.eps, seed=w.seed, seq_offset=q)
        if ref["margin"][0] >= MARGIN:
            assert int(a["n_accept"][q]) == int(ref["n_accept"][0]) and int(a["next_token"][q]) == int(ref["next_token"][0]), q
            assert int(a["next_is_correction"][q]) == int(ref["next_is_correction"][0]), q
