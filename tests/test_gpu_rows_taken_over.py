"""Row-per-SM kernel with more rows than run at once: blocks take over rows whose block has not started yet.  Which block routes
a row must not show in its results: they are, to the bit, those of the same rows in calls that are small enough for every
row to have a block of its own from the start."""
import pytest
import torch

import paper_2609_36601_b200 as P
from paper_2609_36601_b200 import synth
from parity import force_second_tier

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


# rows per SM at once: four up to V = 49152, two up to 98304, then one; one row more than that, one turn and a bit, many turns
@pytest.mark.parametrize("V,per_sm,extra", [(2048, 4, 1), (2056, 4, 37), (8192, 4, 2000), (49160, 2, 1), (65536, 2, 150), (98312, 1, 1), (98312, 1, 200)])
def test_rows_in_one_call_and_in_pieces(V, per_sm, extra):
    at_once = per_sm * torch.cuda.get_device_properties(0).multi_processor_count
    N = at_once + extra
    w = synth.Workload("t", N, V, "bf16", 0.08, 1.5, True, 800 + V % 97, 29)
    d = synth.generate(w, DEV)
    force_second_tier(d, [0, N - 1])
    prev = P.set_kernel(3)              # pinned: pieces and the whole on the same variant
    try:
        for _ in range(2):              # (a call leaves nothing behind for the next)
            out, g = P.route_fwd_bwd(d["s"], d["t"], d["proposal"], w.eps, seed=w.seed)
            torch.cuda.synchronize()
            assert P.last_kernel() == 3
            P.check()
            for r0 in range(0, N, at_once):
                r1 = min(N, r0 + at_once)
                po, pg = P.route_fwd_bwd(d["s"][r0:r1], d["t"][r0:r1], d["proposal"][r0:r1], w.eps, seed=w.seed, row_offset=r0)
                for k in out:
                    assert torch.equal(out[k][r0:r1], po[k]), (k, r0)
                assert torch.equal(g[r0:r1], pg), r0
    finally:
        P.set_kernel(prev)
