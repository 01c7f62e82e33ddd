"""saki_route_host over more chunks than staging buffers, with gradients in pinned, pageable and strided memory and
forward only; against the device entry, to the bit (the same kernel serves both)."""
import pytest
import torch

import paper_2609_36601_b200 as P
from paper_2609_36601_b200 import synth

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("V,N,dtype", [(4000, 3001, "bf16"), (4001, 3001, "bf16"), (3000, 2000, "f32"), (70000, 181, "bf16")])
@pytest.mark.parametrize("grad", ["pinned", "pageable", "strided", "none"])
def test_chunked_call_equals_the_device_entry(V, N, dtype, grad):
    w = synth.Workload("t", N, V, dtype, 0.1, 1.5, True, 700 + V, 19)
    d = synth.generate(w, DEV)
    mask = (torch.arange(N, device=DEV) % 7 != 3).to(torch.uint8)
    out, g = P.route_fwd_bwd(d["s"], d["t"], d["proposal"], w.eps, seed=w.seed, mask=mask, grad_scale=0.5)
    hs, ht, hx, hm = (a.cpu().pin_memory() for a in (d["s"], d["t"], d["proposal"], mask))
    hg = None
    if grad in ("pinned", "pageable"):
        hg = torch.empty((N, V), dtype=w.torch_dtype, pin_memory=grad == "pinned")
    elif grad == "strided":
        hg = torch.empty((N, V + 3), dtype=w.torch_dtype, pin_memory=True)[:, :V]
    hout, hg = P.route_host(hs, ht, hx, w.eps, seed=w.seed, mask=hm, grad_scale=0.5, backward=grad != "none", dlogits=hg)
    for k in out:
        assert torch.equal(out[k].cpu(), hout[k]), k
    if grad != "none":
        assert torch.equal(g.cpu(), hg)
