"""Vocabulary-sharded routing on the GPU: the rows' columns cut into 2, 8 and uneven slices, every slice
reduced as by a rank of its own (the slices of all ranks in one launch per stage: the same stages, in the same
order, that one rank per GPU runs around its all-gather), against the float64 oracle on the whole rows and
against the unsharded call.  Both families of slice kernels: the float32 ones (bf16 slices on 16-byte
boundaries, eps >= 0.02; the default) and the float64 ones (everything else, and under set_kernel(1))."""
import numpy as np
import pytest
import torch

import oracle as O
import paper_2609_36601_b200 as P
from paper_2609_36601_b200 import synth
from paper_2609_36601_b200.vshard import route_vocab_sharded_local, split_columns
from parity import compare_rows, grad_check, oracle_inputs, to_np64

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _slices(d, cuts):
    return [(d["s"][:, a:a + n], d["t"][:, a:a + n], a) for a, n in cuts]


def _special_rows(d, w):
    mask = torch.ones(w.N, dtype=torch.uint8, device=DEV)
    mask[3] = 0
    d["proposal"][5] = w.V + 1                                    # bad id
    d["s"][6, w.V // 2 + 11] = float("nan")                        # non-finite, in the second half of the row
    d["t"][8] = (d["s"][8].float() + 0.01).to(d["t"].dtype)        # teacher = student up to a constant: lambda = 1
    return mask


@pytest.mark.parametrize("tier", ["f32", "f64"])
@pytest.mark.parametrize("V,world", [(151936, 2), (151936, 8), (32000, 3), (1000, 7)])
def test_sliced_rows_match_the_oracle_and_the_unsharded_call(V, world, tier):
    w = synth.Workload("vs", 40, V, "bf16", 0.1, 1.5, True, 900 + world, 40 + world)
    d = synth.generate(w, DEV)
    mask = _special_rows(d, w)
    cuts = split_columns(V, world)
    if world == 7:                                               # uneven, with an empty slice in the middle
        cuts = [(0, 100), (100, 0), (100, 250), (350, 1), (351, 349), (700, 299), (999, 1)]
    prev = P.set_kernel(1 if tier == "f64" else 0)
    try:
        out, gs, waves = route_vocab_sharded_local(_slices(d, cuts), V, d["proposal"], w.eps, w.temperature, w.seed, mask=mask,
                                                   grad_scale=0.5)
        torch.cuda.synchronize()
    finally:
        P.set_kernel(prev)
    g = torch.cat(gs, dim=1)
    assert 1 <= waves <= 6
    s64, t64 = oracle_inputs(d)
    ref = O.route(s64, t64, d["proposal"].cpu().numpy(), w.eps, w.temperature, w.seed, 0, mask=mask.cpu().numpy(),
                  grad_scale=0.5, want_grad=True, grad_dtype=w.dtype)
    n_exempt = compare_rows(out, ref)
    assert n_exempt <= 2
    same = out["corrected"].cpu().numpy() == ref["corrected"]
    live = same & (ref["status"] & (8 | 16) == 0)
    tok = np.where(ref["corrected"] == 1, ref["teacher_top1"], ref["token"])
    grad_check(to_np64(g)[live], ref["grad"][live], w.dtype, tok[live])
    assert torch.all(g[5] == 0) and torch.all(g[6] == 0) and torch.all(g[3] == 0)      # flagged and masked rows
    # float64 all the way: far inside the tolerance on lambda (1e-5), which is what the float32 kernels are held to
    tol = 1e-6 if tier == "f64" else 1e-5
    assert np.max(np.abs(out["lambda"].cpu().numpy() - ref["lam"])) <= tol
    st = ref["status"]
    assert st[3] & 4 and st[5] == 16 and st[6] == 8 and st[8] & 1
    # the unsharded float64 kernel on the same rows: same flags and ids, floats to float32 rounding
    prev = P.set_kernel(1)
    try:
        whole, g_whole = P.route_fwd_bwd(d["s"], d["t"], d["proposal"], w.eps, w.temperature, w.seed, mask=mask, grad_scale=0.5)
        torch.cuda.synchronize()
    finally:
        P.set_kernel(prev)
    ok = torch.as_tensor(np.minimum(ref["margin_accept"], ref["margin_draw"]) >= 1e-6, device=DEV)
    for k in ("corrected", "token", "teacher_top1", "row_status"):
        assert torch.equal(out[k][ok], whole[k][ok]), k
    for k in ("lambda", "tv", "kl", "accept_prob", "loss", "logp_x", "logq_y"):
        assert float((out[k] - whole[k]).abs().max()) <= tol * (1 + float(whole[k].abs().max())), k
    print(f"\n[parity] vocabulary-sharded V={V} world={world} {tier} slice kernels: {waves} evaluation waves, margin-exempt "
          f"{n_exempt}, corrected {int(ref['corrected'].sum())} of {w.N}, max |dlambda| "
          f"{np.max(np.abs(out['lambda'].cpu().numpy() - ref['lam'])):.2e}")


@pytest.mark.parametrize("eps", [0.0, 5.0])
def test_endpoints_need_no_evaluation_wave(eps):
    w = synth.Workload("vs", 16, 8192, "bf16", eps, 1.0, True, 77, 9)
    d = synth.generate(w, DEV)
    out, gs, waves = route_vocab_sharded_local(_slices(d, split_columns(w.V, 4)), w.V, d["proposal"], eps, seed=w.seed)
    torch.cuda.synchronize()
    s64, t64 = oracle_inputs(d)
    ref = O.route(s64, t64, d["proposal"].cpu().numpy(), eps, 1.0, w.seed, want_grad=True, grad_dtype=w.dtype)
    compare_rows(out, ref)
    if eps == 0.0:
        assert waves == 0 and int(out["corrected"].sum()) == 0
    else:
        assert np.all(ref["lam"] == 1.0) and waves == 0
    grad_check(to_np64(torch.cat(gs, dim=1)), ref["grad"], w.dtype, np.where(ref["corrected"] == 1, ref["teacher_top1"], ref["token"]))


@pytest.mark.parametrize("eps", [1e-4, 2e-3, 0.02, 0.1, 3.0])
def test_hard_rows_in_slices(eps):
    """Rows that stress the numerics (near one-hot students and teachers, large magnitudes and offsets, a flat row,
    disjoint peaks) cut into four slices: radii below 0.02 are reduced in float64 altogether; from 0.02 on the
    float32 slice kernels are at work and the combine hands the rows they cannot resolve to the float64 ones."""
    V, N = 4096, 10
    gen = torch.Generator(device=DEV).manual_seed(5)
    s = 2.0 * torch.randn((N, V), generator=gen, device=DEV)
    t = s + 1.5 * torch.randn((N, V), generator=gen, device=DEV)
    s[0, 17] += 40.0
    t[1, 99] += 40.0
    s[2] *= 12.0; t[2] *= 12.0
    t[3] = s[3]
    s[4] = 0.0; t[4] = 0.0; t[4, 5] = 3.0
    s[5] += 300.0; t[5] -= 250.0
    s[6, 7] = 80.0; t[6, 9] = 80.0
    s[7, 100] += 25.0; t[7, 100] += 24.0; t[7, 200] += 18.0       # both nearly one-hot on the same token
    s[8] = 0.0; t[8] = 0.0; s[8, 300] = 17.5; t[8, 300] = 11.8    # p = 0.9999, T = 0.97 on one token: a very flat KL(q_beta || p)
    s, t = s.to(torch.bfloat16), t.to(torch.bfloat16)
    x = torch.tensor([17, 3, 5, 8, 0, 11, 7, 100, 300, 3], dtype=torch.int32, device=DEV)
    d = dict(s=s, t=t, proposal=x)
    state = []
    out, gs, waves = route_vocab_sharded_local(_slices(d, split_columns(V, 4)), V, x, eps, seed=31, state_out=state)
    torch.cuda.synchronize()
    s64, t64 = oracle_inputs(d)
    ref = O.route(s64, t64, x.cpu().numpy(), eps, 1.0, 31, want_grad=True, grad_dtype="bf16")
    n_exempt = compare_rows(out, ref)
    same = out["corrected"].cpu().numpy() == ref["corrected"]
    grad_check(to_np64(torch.cat(gs, dim=1))[same], ref["grad"][same], "bf16",
               np.where(ref["corrected"] == 1, ref["teacher_top1"], ref["token"])[same])
    n64 = int((state[0][:, 30] != 0).sum().item())
    if eps < 0.02:
        assert n64 == 0                    # no row is marked: the whole call runs on the float64 kernels
    if eps == 0.02:
        assert state[0][8, 30] != 0        # the flat row is handed over
    print(f"\n[parity] hard rows in 4 slices, eps={eps}: {waves} waves, {n64} of {N} rows handed to the float64 slice "
          f"kernels, margin-exempt {n_exempt}, max |dlambda| {np.max(np.abs(out['lambda'].cpu().numpy() - ref['lam'])):.2e}")


@pytest.mark.parametrize("dtype,temperature,eps", [("bf16", 0.7, 0.1), ("bf16", 1.6, 0.03), ("f32", 0.9, 0.1)])
def test_temperature_and_dtype_in_slices(dtype, temperature, eps):
    """Temperatures other than 1 (they scale both logit rows, the moments of the logit difference and the gradient)
    on the float32 slice kernels, and fp32 logits, which the float64 kernels take."""
    V = 8192 if dtype == "bf16" else 1024
    w = synth.Workload("vs", 48, V, dtype, eps, 1.5, dtype == "bf16", 1200, 61, temperature=temperature)
    d = synth.generate(w, DEV)
    out, gs, waves = route_vocab_sharded_local(_slices(d, split_columns(V, 4)), V, d["proposal"], eps, temperature, w.seed,
                                               grad_scale=0.25)
    torch.cuda.synchronize()
    s64, t64 = oracle_inputs(d)
    ref = O.route(s64, t64, d["proposal"].cpu().numpy(), eps, temperature, w.seed, grad_scale=0.25, want_grad=True,
                  grad_dtype=dtype)
    n_exempt = compare_rows(out, ref)
    assert n_exempt <= 2
    same = out["corrected"].cpu().numpy() == ref["corrected"]
    grad_check(to_np64(torch.cat(gs, dim=1))[same], ref["grad"][same], dtype,
               np.where(ref["corrected"] == 1, ref["teacher_top1"], ref["token"])[same])


def test_marked_rows_in_more_than_one_group():
    """The float64 slice kernels look through a call's marks in groups of 512 rows per block (16 slices in one launch: 28
    blocks per slice on 148 SMs).  More rows than a group holds, marked ones at both ends of a group and in the next one,
    the rest in between and behind them unmarked; against the unsharded float64 kernel."""
    V, world = 1024, 16
    blocks = (3 * torch.cuda.get_device_properties(0).multi_processor_count + world - 1) // world
    group = 512 * blocks
    N = group + 3 * blocks + 5
    w = synth.Workload("vs", N, V, "bf16", 0.02, 1.5, False, 1300, 71)
    d = synth.generate(w, DEV)
    marked = torch.tensor([0, 1, blocks - 1, blocks, group // 2, group - blocks, group - 1, group, group + 2 * blocks, N - 1], device=DEV)
    for k, peak in (("s", 17.5), ("t", 11.8)):         # p = 0.99997, T = 0.992 on one token: a very flat KL(q_beta || p)
        d[k][marked] = 0.0
        d[k][marked, 300] = peak
    d["proposal"][marked] = 300
    state = []
    out, gs, _ = route_vocab_sharded_local(_slices(d, split_columns(V, world)), V, d["proposal"], w.eps, seed=w.seed, grad_scale=0.5,
                                           state_out=state)
    prev = P.set_kernel(1)
    try:
        ref, g_ref = P.route_fwd_bwd(d["s"], d["t"], d["proposal"], w.eps, seed=w.seed, grad_scale=0.5)
    finally:
        P.set_kernel(prev)
    f64 = torch.nonzero(state[0][:, 30]).flatten()
    assert set(marked.tolist()) <= set(f64.tolist()) and len(f64) < N // 4
    for k in ("lambda", "tv", "kl", "accept_prob", "logp_x"):
        assert float((out[k] - ref[k]).abs().max()) <= 1e-5 * (1 + float(ref[k].abs().max())), k
        assert float((out[k] - ref[k])[f64].abs().max()) <= 1e-6, k             # the same arithmetic to float32 rounding
    for k in ("corrected", "token", "teacher_top1", "row_status"):
        assert torch.equal(out[k][marked], ref[k][marked]), k
    tok = torch.where(ref["corrected"] == 1, ref["teacher_top1"], ref["token"])[marked].cpu().numpy()
    grad_check(to_np64(torch.cat(gs, dim=1)[marked]), to_np64(g_ref[marked]), w.dtype, tok)


def test_a_stream_that_is_not_the_current_one():
    """The caller's stream, busy for a while when the call comes: counters and marks are zeroed, counted up and read in its
    order, so that rows that take more waves and rows for the float64 kernels are routed as on the current stream."""
    V = 4096
    w = synth.Workload("vs", 24, V, "bf16", 0.02, 1.5, False, 1400, 81)
    d = synth.generate(w, DEV)
    for k, peak in (("s", 17.5), ("t", 11.8)):         # very flat rows: marked for the float64 kernels
        d[k][::5] = 0.0
        d[k][::5, 300] = peak
    d["proposal"][::5] = 300
    slices = _slices(d, split_columns(V, 4))
    state = []
    ref, g_ref, waves = route_vocab_sharded_local(slices, V, d["proposal"], w.eps, seed=w.seed, state_out=state)
    assert bool((state[0][::5, 30] != 0).all()) and waves >= 2
    torch.cuda.synchronize()
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        torch.cuda._sleep(50_000_000)                    # some 25 ms
    out, gs, n = route_vocab_sharded_local(slices, V, d["proposal"], w.eps, seed=w.seed, stream=side)
    side.synchronize()
    assert n == waves
    for k in ref:
        assert torch.equal(out[k], ref[k]), k
    for a, b in zip(gs, g_ref):
        assert torch.equal(a, b)


@pytest.mark.parametrize("N,world", [(1, 8), (7, 16), (9, 17), (8, 33)])
def test_combines_at_the_edges_of_their_groups(N, world):
    """A combine takes eight rows a block and holds the records of up to sixteen ranks at once; a launch takes sixteen slices."""
    V = 8192
    w = synth.Workload("vs", N, V, "bf16", 0.125, 1.5, True, 950 + world, 50 + world)
    d = synth.generate(w, DEV)
    out, gs, _ = route_vocab_sharded_local(_slices(d, [(8 * a, 8 * n) for a, n in split_columns(V // 8, world)]), V, d["proposal"], w.eps,
                                           w.temperature, w.seed, grad_scale=0.5)
    s64, t64 = oracle_inputs(d)
    ref = O.route(s64, t64, d["proposal"].cpu().numpy(), w.eps, w.temperature, w.seed, 0, grad_scale=0.5, want_grad=True, grad_dtype=w.dtype)
    compare_rows(out, ref)
    same = out["corrected"].cpu().numpy() == ref["corrected"]
    tok = np.where(ref["corrected"] == 1, ref["teacher_top1"], ref["token"])
    grad_check(to_np64(torch.cat(gs, dim=1))[same], ref["grad"][same], w.dtype, tok[same])
    assert np.max(np.abs(out["lambda"].cpu().numpy() - ref["lam"])) <= 1e-5      # what the float32 kernels are held to


def test_logits_rewritten_right_in_front_of_the_call():
    """Slices of which one is not on 16-byte boundaries (float64 beside float32), the same buffers over and over, new logits and
    proposals copied into them by kernels that the call follows without a pause: to the bit what the call gives after a wait."""
    V, N, sets = 32768, 300, 4
    w = [synth.Workload("vs", N, V, "bf16", 0.125, 1.5, True, 1500 + k, 91) for k in range(sets)]
    d = [synth.generate(x, DEV) for x in w]
    cuts = split_columns(V, 4)
    slices = []
    for r, (a, n) in enumerate(cuts):
        st = [torch.empty(N * (n + 8), dtype=torch.bfloat16, device=DEV)[r == 2:].narrow(0, 0, N * n).view(N, n) for _ in "st"]
        slices.append((*st, a))
    x = torch.empty(N, dtype=torch.int32, device=DEV)

    def call(k, pause):
        for (s, t, a), (_, n) in zip(slices, cuts):
            s.copy_(d[k]["s"][:, a:a + n])
            t.copy_(d[k]["t"][:, a:a + n])
        x.copy_(d[k]["proposal"])
        if pause:
            torch.cuda.synchronize()
        out, gs, _ = route_vocab_sharded_local(slices, V, x, w[k].eps, seed=w[k].seed)
        return [out[f] for f in sorted(out)] + gs

    ref = [call(k, True) for k in range(sets)]
    for i in range(5 * sets):
        for a, b in zip(call(i % sets, False), ref[i % sets]):
            assert torch.equal(a, b)


@pytest.mark.skipif(torch.cuda.device_count() < 2, reason="needs a second GPU to be the current one")
def test_slices_that_are_not_on_the_current_device():
    """Without a stream from the caller the stages and their counters take the current stream of the slices' device, which is busy
    for a while when the call comes."""
    V = 4096
    w = synth.Workload("vs", 24, V, "bf16", 0.02, 1.5, False, 1400, 81)
    d = synth.generate(w, DEV)
    slices = _slices(d, split_columns(V, 4))
    with torch.cuda.device(0):
        ref, g_ref, waves = route_vocab_sharded_local(slices, V, d["proposal"], w.eps, seed=w.seed)
        torch.cuda.synchronize()
        torch.cuda._sleep(50_000_000)                    # some 25 ms
    with torch.cuda.device(1):
        out, gs, n = route_vocab_sharded_local(slices, V, d["proposal"], w.eps, seed=w.seed)
    torch.cuda.synchronize(0)
    assert n == waves
    for k in ref:
        assert torch.equal(out[k], ref[k]), k
    for a, b in zip(gs, g_ref):
        assert torch.equal(a, b)
