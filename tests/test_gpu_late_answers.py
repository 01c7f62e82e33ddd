"""Row-per-SM kernel: a block that is done asks for the row of one that has not started.  If the answer comes later than the
wait limit, the row that it took over is flagged TIMEOUT with zero outputs and a zero gradient row, and counted: no row ends
without a status.  Nothing is withheld: the limit is set below the time that an answer takes."""
import pytest
import torch

import paper_2609_36601_b200 as P
from paper_2609_36601_b200 import binding, synth

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
UNWRITTEN = 77


def limited_call(d, w, limit):
    """One call under a wait limit, into buffers that show what was not written.  Returns (flagged rows, outputs, gradient)."""
    out = P.alloc_outputs(w.N, torch.device(DEV))
    for v in out.values():
        v.fill_(UNWRITTEN)
    g = torch.full_like(d["s"], float(UNWRITTEN))
    try:
        P.set_wait_limit(limit)
        P.route_fwd_bwd(d["s"], d["t"], d["proposal"], w.eps, seed=w.seed, out=out, dlogits=g)
    finally:
        P.set_wait_limit(0)
    n_flagged = P.check()                                # synchronises: the kernel came back
    late = (out["row_status"] & binding.ROW_TIMEOUT) != 0
    assert n_flagged == int(late.sum())
    return late, out, g


def check_rows(late, out, g, ref, g_ref):
    """Flagged rows carry nothing but the status, the others are those of the undisturbed call to the bit."""
    assert torch.all(out["row_status"][late] == binding.ROW_TIMEOUT)
    assert torch.all(out["token"][late] == -1) and torch.all(out["corrected"][late] == 0)
    for k in ("lambda", "kl", "tv", "accept_prob", "loss", "logp_x", "logq_y"):
        assert torch.all(out[k][late] == 0), k
    assert torch.all(g[late] == 0)
    for k in out:
        assert torch.equal(out[k][~late], ref[k][~late]), k
    assert torch.equal(g[~late], g_ref[~late])


def test_a_row_whose_answer_is_late_is_flagged():
    at_once = 4 * torch.cuda.get_device_properties(0).multi_processor_count       # rows of 2048 elements in flight
    w = synth.Workload("late", at_once + 108, 2048, "bf16", 0.1, 1.5, True, 4100, 9)
    d = synth.generate(w, DEV)
    prev = P.set_kernel(3)
    P.check()
    by_answer = 0
    try:
        ref, g_ref = P.route_fwd_bwd(d["s"], d["t"], d["proposal"], w.eps, seed=w.seed)
        torch.cuda.synchronize()
        assert P.last_kernel() == 3 and P.check() == 0
        # the rows are in L2: their copies have landed by the time they are waited for, an answer takes some hundred cycles
        for limit in (100, 150, 200, 250):
            late, out, g = limited_call(d, w, limit)
            check_rows(late, out, g, ref, g_ref)
            if not late[:at_once].any():                 # every copy was in time: it is answers that were late
                by_answer += int(late[at_once:].sum())
        again, g_again = P.route_fwd_bwd(d["s"], d["t"], d["proposal"], w.eps, seed=w.seed)
        torch.cuda.synchronize()
        assert P.check() == 0
    finally:
        P.set_kernel(prev)
    assert by_answer > 0, "no answer was waited for under the limit"
    for k in ref:
        assert torch.equal(again[k], ref[k]), k
    assert torch.equal(g_again, g_ref)


def test_a_limit_beyond_any_wait_changes_nothing():
    w = synth.Workload("patient", 20000, 2048, "bf16", 0.1, 1.5, True, 4101, 9)          # thirty rows taken over per block
    d = synth.generate(w, DEV)
    prev = P.set_kernel(3)
    P.check()
    try:
        ref, g_ref = P.route_fwd_bwd(d["s"], d["t"], d["proposal"], w.eps, seed=w.seed)
        late, out, g = limited_call(d, w, 2 ** 63 - 1)
    finally:
        P.set_kernel(prev)
    assert not late.any()
    check_rows(late, out, g, ref, g_ref)
