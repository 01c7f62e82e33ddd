"""Logits masked with the lowest value of their type, as constrained decoding and padded vocabularies leave them: finite
values whose differences have no square in float32.  Every kernel the automatic choice comes to, against the oracle."""
import numpy as np
import pytest
import torch

import oracle as O
import paper_2609_36601_b200 as P
from paper_2609_36601_b200 import synth
from parity import compare_rows, grad_check, oracle_inputs, to_np64

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
CALLS = [(2048, 4, "bf16"), (32768, 4, "bf16"), (40960, 32, "bf16"), (65536, 4, "bf16"), (151936, 8, "bf16"), (40960, 40, "bf16"),
         (32003, 4, "bf16"), (1024, 4, "f32")]


def _workload(V, N, dtype, eps):
    w = synth.Workload("t", N, V, dtype, eps, 1.2, V > 1024, 700 + V % 89, 21)
    d = synth.generate(w, DEV)
    return w, d, torch.finfo(w.torch_dtype).min


def _check(w, d, rows):
    out, g = P.route_fwd_bwd(d["s"], d["t"], d["proposal"], w.eps, w.temperature, w.seed, grad_scale=0.25)
    s64, t64 = oracle_inputs(d)
    ref = O.route(s64, t64, d["proposal"].cpu().numpy(), w.eps, w.temperature, w.seed, grad_scale=0.25, want_grad=True,
                  grad_dtype=w.dtype, rows=rows)
    compare_rows(out, ref, rows)
    same = out["corrected"].cpu().numpy()[rows] == ref["corrected"]
    tok = np.where(ref["corrected"] == 1, ref["teacher_top1"], ref["token"])[same]
    grad_check(to_np64(g)[rows][same], ref["grad"][same], w.dtype, tok)
    return out


@pytest.mark.parametrize("V,N,dtype", CALLS)
@pytest.mark.parametrize("eps", [0.0, 0.125, 4.0])
def test_masked_student(V, N, dtype, eps):
    """The student's row masked where the teacher's is not (row 1: a quarter of it; row 2: its end), both masked alike
    (row 3), and beside them a row that is not finite, which is flagged."""
    w, d, lowest = _workload(V, N, dtype, eps)
    d["s"][1, V // 4:V // 2] = lowest
    d["s"][2, V - V // 8:] = lowest
    d["s"][3, V // 4:V // 2] = lowest
    d["t"][3, V // 4:V // 2] = lowest
    d["s"][0, V // 3] = float("-inf")
    d["proposal"][1:4] = 5
    out = _check(w, d, list(range(4)))
    st = out["row_status"].cpu().numpy()
    assert st[0] == 8 and not np.any(st[1:4] & 8)
