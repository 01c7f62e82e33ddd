"""A routing call in a CUDA graph on a stream that the library has not seen: its scratch is allocated while the stream is
captured (in the mode that lets memory be allocated), and has to be fit for use by ordinary calls on that stream before the
graph is launched for the first time, and by the graph after them."""
import pytest
import torch

import paper_2609_36601_b200 as P
from paper_2609_36601_b200 import synth
from parity import force_second_tier

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def test_first_call_on_a_stream_is_a_captured_one():
    w = synth.Workload("t", 300, 8192, "bf16", 0.125, 1.5, True, 420, 61)
    d = synth.generate(w, DEV)
    force_second_tier(d, [3, 70, 299])                 # rows for the list that the scratch holds
    ref, g_ref = P.route_fwd_bwd(d["s"], d["t"], d["proposal"], w.eps, seed=w.seed)
    assert P.redo_count() == 3
    side = torch.cuda.Stream()
    graph = torch.cuda.CUDAGraph()
    out, g = P.alloc_outputs(w.N, DEV), torch.empty_like(d["s"])
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=side, capture_error_mode="relaxed"):
        P.route_fwd_bwd(d["s"], d["t"], d["proposal"], w.eps, seed=w.seed, out=out, dlogits=g)
    torch.cuda.synchronize()

    def same(o, grad):
        for k in ref:
            assert torch.equal(o[k], ref[k]), k
        assert torch.equal(grad, g_ref)

    with torch.cuda.stream(side):                      # an ordinary call before the graph is ever launched
        o, grad = P.route_fwd_bwd(d["s"], d["t"], d["proposal"], w.eps, seed=w.seed)
    side.synchronize()
    same(o, grad)
    for _ in range(3):
        for t in (*out.values(), g):
            t.zero_()
        torch.cuda.synchronize()
        with torch.cuda.stream(side):
            graph.replay()
        side.synchronize()
        same(out, g)
