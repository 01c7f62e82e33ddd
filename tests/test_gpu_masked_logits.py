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


def _largest_coefficient(s, t, eps):
    """Of one row, in float64: the largest beta with KL(q_beta || p) <= eps, by bisection of its exponent (the oracle's bisection
    ends at 1e-15; here the root may lie at 1e-39), with KL and TV there."""
    lp, lT = (x - (x.max() + np.log(np.exp(x - x.max()).sum())) for x in (s, t))

    def at(beta):
        z = lp + beta * (lT - lp)
        lq = z - (z.max() + np.log(np.exp(z - z.max()).sum()))
        q = np.exp(lq)
        return float((q * np.where(q > 0, lq - lp, 0.0)).sum()), float(np.maximum(q - np.exp(lp), 0.0).sum())

    if at(1.0)[0] <= eps:
        return 1.0, *at(1.0)
    lo, hi = -150.0, 0.0                               # of log2
    for _ in range(200):
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if at(2.0 ** mid)[0] <= eps else (lo, mid)
    return 2.0 ** lo, *at(2.0 ** lo)


@pytest.mark.parametrize("V,N,dtype", CALLS)
@pytest.mark.parametrize("mask,kernel", [("lowest", 0), ("lowest", 1), (-1e9, 1)])
def test_masked_teacher(V, N, dtype, mask, kernel):
    """The teacher's row masked where the student's is not.  Where the student has more than 1 - exp(-eps) there, every lambda
    that moves mass away from it in earnest is beyond the radius, and the root lies at the scale of the mask (rows 0 and 1);
    where it has less, the root is an ordinary one (rows 2 and 3)."""
    w, d, lowest = _workload(V, N, dtype, 0.125)
    for r, (a, b) in enumerate([(V // 4, V // 2), (0, V // 2), (V - V // 40, V), (V // 2, V // 2 + 3)]):
        d["t"][r, a:b] = lowest if mask == "lowest" else mask
        d["s"][r, a:b] += 2.0 if r < 2 else -6.0
    d["proposal"][:4] = d["t"][:4].float().argmax(dim=1).to(torch.int32)
    prev = P.set_kernel(kernel)
    try:
        out = P.route_fwd(d["s"], d["t"], d["proposal"], w.eps, w.temperature, w.seed)
    finally:
        P.set_kernel(prev)
    s64, t64 = oracle_inputs(d, range(4))
    got = {k: out[k].double().cpu().numpy() for k in ("lambda", "kl", "tv")}
    for r in range(4):
        lam, kl, tv = _largest_coefficient(s64[r], t64[r], w.eps)
        assert (lam < 1e-7) == (r < 2), (r, lam)
        print(f"row {r}: lambda {lam:.3e} {got['lambda'][r]:.3e} kl {kl:.6f} {got['kl'][r]:.6f} tv {tv:.6f} {got['tv'][r]:.6f}")
        assert abs(got["lambda"][r] - lam) <= 1e-5 and abs(got["kl"][r] - kl) <= 1e-5 and abs(got["tv"][r] - tv) <= 1e-5, r
