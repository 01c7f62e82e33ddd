"""Rows on which the two models disagree by hundreds of nats: each has its mass where the other is far below its maximum, so
that every term of q_beta lies far below a shift made of the two maxima.  Every kernel the automatic choice comes to, against
the oracle."""
import pytest
import torch

import oracle as O
import paper_2609_36601_b200 as P
from paper_2609_36601_b200 import synth
from parity import compare_rows, oracle_inputs

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _rows(V, N, dtype="bf16"):
    w = synth.Workload("t", N, V, dtype, 0.125, 1.2, False, 800 + V % 89, 22)
    d = synth.generate(w, DEV)
    for r, (a, b, ds, dt) in enumerate([(0, V // 4, -500.0, -300.0), (0, V // 2, -300.0, -500.0), (V // 2, V, -90.0, -120.0)]):
        d["s"][r, a:b] += ds                           # the student's mass outside [a, b), the teacher's inside
        d["t"][r, :a] += dt
        d["t"][r, b:] += dt
    d["proposal"][:3] = d["s"][:3].float().argmax(dim=1).to(torch.int32)
    s64, t64 = oracle_inputs(d, range(4))
    ref = O.route(s64, t64, d["proposal"][:4].cpu().numpy(), w.eps, w.temperature, w.seed)
    assert (ref["lam"][:3] > 0.1).all() and (ref["lam"][:3] < 0.7).all()
    return w, d, ref


@pytest.mark.parametrize("V,N,dtype", [(2048, 4, "bf16"), (4096, 300, "bf16"), (8192, 700, "bf16"), (32768, 4, "bf16"),
                                       (40960, 40, "bf16"), (65536, 32, "bf16"), (151936, 4, "bf16"), (151936, 40, "bf16"),
                                       (32003, 4, "bf16"), (1024, 4, "f32")])
def test_rows_whose_models_are_apart(V, N, dtype):
    w, d, ref = _rows(V, N, dtype)
    out = P.route_fwd(d["s"], d["t"], d["proposal"], w.eps, w.temperature, w.seed)
    compare_rows(out, ref, range(4))
