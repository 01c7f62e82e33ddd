"""The float64 kernels at radii where every digit counts: KL(q_beta || p) = beta m1 - log Z(beta) is a difference of numbers of
the size of 1, so an error E of its terms moves lambda by E / (d KL / d log beta): a relative error of E / (2 eps) as a rule.
Against a solve in extended precision."""
import numpy as np
import pytest
import torch

import paper_2609_36601_b200 as P
from paper_2609_36601_b200.vshard import route_vocab_sharded_local, split_columns

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
L = np.longdouble


def _solve(s, t, eps):
    """lambda, d KL / d beta there, and the student's log-sum-exp."""
    s, t = s.astype(L), t.astype(L)
    lse = s.max() + np.log(np.exp(s - s.max()).sum())
    lp = s - lse
    d = t - t.max() - np.log(np.exp(t - t.max()).sum()) - lp
    p = np.exp(lp)

    def kl(b):
        e = p * np.exp(b * d)
        z = e.sum()
        m = (e * d).sum() / z
        return b * m - np.log(z), b * ((e * d * d).sum() / z - m * m)

    assert kl(L(1))[0] > eps                     # (else lambda = 1)
    lo, hi = L(0), L(1)
    b = min(L(0.5), np.sqrt(2 * L(eps) / ((p * d * d).sum() - (p * d).sum() ** 2)))
    for _ in range(200):                         # Newton inside a bracket
        k, slope = kl(b)
        lo, hi = (lo, b) if k > eps else (b, hi)
        nb = b - (k - L(eps)) / slope if slope > 0 else (lo + hi) / 2
        if not lo < nb < hi:
            nb = (lo + hi) / 2
        if abs(nb - b) < 1e-17 * b:
            break
        b = nb
    return float(b), float(slope), float(lse)


@pytest.mark.parametrize("sharded", [False, True])
@pytest.mark.parametrize("kind", ["gauss", "one_hot"])
@pytest.mark.parametrize("V,N", [(64, 100), (1025, 40)])
@pytest.mark.parametrize("eps", [2.0 ** -20, 2.0 ** -27, 2.0 ** -30])
def test_lambda_to_the_last_digits(eps, V, N, kind, sharded):
    g = torch.Generator().manual_seed(5 + V)
    s = 2.0 * torch.randn(N, V, generator=g)
    t = s + torch.randn(N, V, generator=g)
    if kind == "one_hot":
        s[:, 3] += 14.0
        t[:, 3] += 12.0
    x = torch.zeros(N, dtype=torch.int32, device=DEV)
    prev = P.set_kernel(1)
    try:
        if sharded:
            slices = [(s[:, a:a + n].contiguous().to(DEV), t[:, a:a + n].contiguous().to(DEV), a) for a, n in split_columns(V, 3)]
            out = route_vocab_sharded_local(slices, V, x, eps, 1.0, 3)[0]
        else:
            out = P.route_fwd_bwd(s.to(DEV), t.to(DEV), x, eps, 1.0, 3)[0]
    finally:
        P.set_kernel(prev)
    ref = np.array([_solve(s[i].numpy(), t[i].numpy(), eps) for i in range(N)])
    # The normaliser of p is one number of the size of the log-sum-exp that four roundings of 2^-53 have gone through; with the
    # exponential, the sums and the logarithm of Z, a few more of a number of the size of 1.  Lambda is then rounded to float32.
    E = 2.0 ** -53 * (4.0 * np.abs(ref[:, 2]) + 8.0)
    err = np.abs(out["lambda"].cpu().numpy().astype(np.float64) - ref[:, 0])
    assert (err <= E / ref[:, 1] + 2.0 ** -24 * ref[:, 0]).all(), (err * ref[:, 1] / E).max()


@pytest.mark.parametrize("V", [64, 1024])
def test_log_sum_exps_of_logits_far_from_zero(V):
    """Student logits about 1000, the teacher's about -500: KL takes the roundings of the student's log-sum-exp one to one."""
    N, eps = 100, 2.0 ** -30
    g = torch.Generator().manual_seed(5 + V)
    s = 2.0 * torch.randn(N, V, generator=g)
    t = s + torch.randn(N, V, generator=g)
    s += 1000.0
    t -= 500.0
    prev = P.set_kernel(1)
    try:
        out = P.route_fwd_bwd(s.to(DEV), t.to(DEV), torch.zeros(N, dtype=torch.int32, device=DEV), eps, 1.0, 3)[0]
    finally:
        P.set_kernel(prev)
    ref = np.array([_solve(s[i].numpy(), t[i].numpy(), eps) for i in range(N)])
    assert (ref[:, 2] < 1024).all()
    # The log-sum-exp, below 1024, rounded once (2^-44); log2(e) times it, below 2048, once more (2^-43 of log2); ln 2 and log2(e) as
    # float64 numbers, each good to 2.4e-17 and used on numbers of about 1450; the bound of the test above for what has no offset.
    E = 2.0 ** -44 + np.log(2.0) * 2.0 ** -43 + 2 * 2.4e-17 * 1450 * np.log(2.0) + 2.0 ** -53 * (4.0 * (ref[:, 2] - 1000.0) + 8.0)
    err = np.abs(out["lambda"].cpu().numpy().astype(np.float64) - ref[:, 0])
    assert (err <= E / ref[:, 1] + 2.0 ** -24 * ref[:, 0]).all(), (err * ref[:, 1] / E).max()
