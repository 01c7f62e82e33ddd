"""The output tensors that the binding allocates: every field with memory of its own, so that it can be saved, resized and
kept without the others."""
import io

import pytest
import torch

import paper_2609_36601_b200 as P
from paper_2609_36601_b200 import synth


def _own_memory(out):
    assert len({t.untyped_storage().data_ptr() for t in out.values()}) == len(out)
    for t in out.values():
        assert t.untyped_storage().nbytes() == t.numel() * t.element_size() and t.storage_offset() == 0
    buf = io.BytesIO()
    torch.save(out, buf)
    buf.seek(0)
    back = torch.load(buf)
    for k, t in out.items():
        assert back[k].dtype == t.dtype and torch.equal(back[k], t), k


def test_allocated_outputs_have_memory_of_their_own():
    out = P.alloc_outputs(37, "cpu")
    for k, t in enumerate(out.values()):
        t.fill_(k + 1)
    _own_memory(out)
    out["token"].resize_(4096).fill_(0)
    assert all(bool((t == k + 1).all()) for k, (f, t) in enumerate(out.items()) if f != "token")


@pytest.mark.gpu
def test_returned_outputs_have_memory_of_their_own():
    w = synth.Workload("t", 24, 2048, "bf16", 0.125, 1.0, True, 410, 60)
    d = synth.generate(w, "cuda:0")
    out = P.route_fwd(d["s"], d["t"], d["proposal"], w.eps, seed=w.seed)
    _own_memory(out)
    meta, _ = P.route_bwd_from_meta(d["s"], out["corrected"], d["proposal"], out["teacher_top1"], out["logT_x"] - out["logp_x"])
    _own_memory(meta)
    host, _ = P.route_host(*(d[k].cpu() for k in ("s", "t", "proposal")), w.eps, seed=w.seed)
    _own_memory(host)
