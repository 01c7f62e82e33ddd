"""Performance cases: the calls a program that uses this library makes, at the sizes it makes them.

Every case names a call (`call`) and its sizes.  The calls:

  fwd     route_fwd: one decoding step; the caller wants tokens and probabilities, no gradient
  train   route_fwd_bwd into buffers the training loop keeps: routing, losses and the gradient
  spec    spec_verify: verification of a batch of drafted blocks
  meta    select_tm (placement control, where asked for) and route_bwd_from_meta: the trainer's step
  lmhead  lmhead_lse: the lm-head GEMM in front of the path, row statistics in its epilogue
  vshard  route_vocab_sharded_local: rows whose columns are spread over ranks, the ranks in turn on one GPU
  sample  sample_proposal: the student's proposals
  host    route_host: logits, results and gradient in pinned host memory

Logits come from the repository's synthetic workloads (`synth.py`: Gaussian logits with a Zipf rank bias, a
teacher correlated with the student), seeded by the caller.
"""
from __future__ import annotations

import math

import torch

import paper_2609_36601_b200 as saki
from paper_2609_36601_b200 import synth
from paper_2609_36601_b200.vshard import route_vocab_sharded_local, split_columns

DEV = "cuda:0"
# what a training loop keeps of a routing call: the inputs of the trainer's step and the logged statistics
TRAIN_FIELDS = ("corrected", "token", "teacher_top1", "row_status", "lambda", "kl", "tv", "accept_prob", "logp_x",
                "logq_x", "logT_x", "loss")


def listed():
    return [
        # a decoding step of a small serving batch: eight positions, latency and launches count
        dict(name="decode_8", call="fwd", N=8, V=151936, dtype="bf16", eps=0.1, sigma=1.5, temperature=1.0),
        # the tiny fp32 workload (unit-sized batch of a small-vocabulary model)
        dict(name="tiny_f32", call="train", N=64, V=1024, dtype="f32", eps=0.1, sigma=1.5, temperature=1.0, masked=False),
        # a training batch of a 32000-entry vocabulary
        dict(name="train_32k", call="train", N=4096, V=32000, dtype="bf16", eps=0.05, sigma=1.0, temperature=1.0, masked=False),
        # the headline batch: 8 rollouts of 2048 tokens over a 151936-entry vocabulary
        dict(name="train_152k", call="train", N=16384, V=151936, dtype="bf16", eps=0.1, sigma=1.5, temperature=1.0, masked=False),
        # a vocabulary that was extended by a few tokens (rows are not 16-byte aligned), padding positions masked
        dict(name="train_ragged", call="train", N=1024, V=32003, dtype="bf16", eps=0.05, sigma=1.0, temperature=1.0, masked=True),
        # logits kept in fp32 by the engine, long rows, sampled at a temperature below one, late in the radius schedule
        dict(name="train_f32", call="train", N=512, V=151936, dtype="f32", eps=0.02, sigma=1.5, temperature=0.8, masked=False),
        # block verification: 512 sequences of 6 drafted tokens and the bonus position
        dict(name="spec_512x6", call="spec", B=512, K=6, V=151936, dtype="bf16", eps=0.1, sigma=1.5, temperature=1.0),
        # the trainer's step on freshly evaluated logits, with the TV-weighted placement control
        dict(name="trainer_step", call="meta", N=8192, V=151936, dtype="bf16", control="tv", temperature=1.0, masked=True),
        # the lm-head of 4096 positions
        dict(name="lm_head", call="lmhead", N=4096, V=151936, d=2560, temperature=1.0),
        # a tensor-parallel head of 8 ranks
        dict(name="sharded_8", call="vshard", N=1024, V=151936, world=8, dtype="bf16", eps=0.1, sigma=1.5, temperature=1.0),
        # proposals for a batch of 512 sequences
        dict(name="propose_512", call="sample", N=512, V=151936, dtype="bf16", temperature=1.0),
        # a caller whose logits live in host memory
        dict(name="host_512", call="host", N=512, V=32000, dtype="bf16", eps=0.05, sigma=1.0, temperature=1.0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _vocab(rng, lo, hi, multiple=1):
    return max(multiple, _log_int(rng, lo, hi) // multiple * multiple)


def draw(rng):
    call = rng.choice(("fwd", "train", "train", "train", "spec", "meta", "lmhead", "vshard", "sample", "host"))
    eps = float("%.3g" % math.exp(rng.uniform(math.log(2e-3), math.log(1.0))))
    sigma = rng.choice((0.5, 1.0, 1.5, 2.0))
    tau = rng.choice((1.0, 1.0, 0.7, 1.3))
    if call == "fwd":
        ragged = rng.random() < 0.2
        V = _vocab(rng, 2048, 160000, 1 if ragged else 8)
        return dict(call=call, N=_log_int(rng, 1, 512), V=V, dtype="bf16", eps=eps, sigma=sigma, temperature=tau)
    if call == "train":
        kind = rng.choice(("bf16", "bf16", "ragged", "f32"))
        if kind == "bf16":
            V = _vocab(rng, 4096, 160000, 8)
            N = _log_int(rng, 64, max(65, min(16384, int(1.2e9 / V))))
        else:
            V = _vocab(rng, 512, 160000) | (1 if kind == "ragged" else 0)
            N = _log_int(rng, 16, max(17, min(4096, int(6e7 / V))))
        return dict(call=call, N=N, V=V, dtype="f32" if kind == "f32" else "bf16", eps=eps, sigma=sigma, temperature=tau,
                    masked=rng.random() < 0.5)
    if call == "spec":
        K = rng.randint(1, 8)
        V = _vocab(rng, 8192, 160000, 8)
        return dict(call=call, B=_log_int(rng, 4, max(5, min(1024, int(5e8 / V / (K + 1))))), K=K, V=V, dtype="bf16", eps=eps,
                    sigma=sigma, temperature=tau)
    if call == "meta":
        V = _vocab(rng, 4096, 160000, 8)
        return dict(call=call, N=_log_int(rng, 64, max(65, min(16384, int(1.2e9 / V)))), V=V, dtype="bf16",
                    control=rng.choice(("none", "random", "tv")), temperature=tau, masked=rng.random() < 0.5)
    if call == "lmhead":
        return dict(call=call, N=_log_int(rng, 64, 4096), V=_vocab(rng, 16384, 151936, 8), d=rng.choice((1024, 1536, 2048, 2560)),
                    temperature=tau)
    if call == "vshard":
        V = _vocab(rng, 16384, 160000, 64)
        return dict(call=call, N=_log_int(rng, 16, max(17, min(2048, int(1.5e8 / V)))), V=V, world=rng.choice((2, 4, 8)),
                    dtype="bf16", eps=max(eps, 0.02), sigma=sigma, temperature=tau)
    if call == "sample":
        V = _vocab(rng, 2048, 160000)
        return dict(call=call, N=_log_int(rng, 8, max(9, min(2048, int(7e7 / V)))), V=V, dtype=rng.choice(("bf16", "f32")),
                    temperature=tau)
    V = _vocab(rng, 4096, 160000, 8)
    return dict(call=call, N=_log_int(rng, 8, max(9, min(2048, int(3e7 / V)))), V=V, dtype="bf16", eps=eps, sigma=sigma,
                temperature=tau)


def _rows(case, seed, n):
    w = synth.Workload("case", n, case["V"], case["dtype"], case.get("eps", 0.1), case.get("sigma", 1.5), case["V"] > 1024,
                       seed, seed, temperature=case["temperature"])
    return synth.generate(w, DEV)


def _mask(gen, n):
    return (torch.rand(n, generator=gen, device=DEV) > 0.1).to(torch.uint8)     # a tenth of the positions is padding


def prepare(case, seed):
    call, gen = case["call"], torch.Generator(device=DEV)
    gen.manual_seed(seed)
    st = dict(case=case, seed=seed)
    if call == "lmhead":
        N, V, d = case["N"], case["V"], case["d"]
        st["hidden"] = torch.randn((N, d), generator=gen, device=DEV, dtype=torch.float32).to(torch.bfloat16)
        st["weight"] = (torch.randn((V, d), generator=gen, device=DEV, dtype=torch.float32) * (2.0 / math.sqrt(d))).to(torch.bfloat16)
        st["logits"] = torch.empty((N, V), dtype=torch.bfloat16, device=DEV)
        st["scratch"] = torch.empty(int(saki.load_library().saki_lmhead_scratch_bytes(N, V)), dtype=torch.uint8, device=DEV)
        return st
    if call == "spec":
        B, K = case["B"], case["K"]
        d = _rows(case, seed, B * (K + 1))
        st["s"], st["t"] = d["s"].view(B, K + 1, -1), d["t"].view(B, K + 1, -1)
        st["draft"] = d["proposal"].view(B, K + 1)[:, :K].contiguous()
        return st
    N, V = case["N"], case["V"]
    d = _rows(case, seed, N)
    if call == "sample":
        st["s"] = d["s"]
        return st
    if call == "meta":
        # the metadata a routing call of the rollout returns: about a sixth of the positions corrected
        st["s"], st["proposal"] = d["s"], d["proposal"]
        st["tv"] = torch.rand(N, generator=gen, device=DEV).mul_(0.36)
        st["corrected"] = (torch.rand(N, generator=gen, device=DEV) < st["tv"]).to(torch.uint8)
        st["teacher_top1"] = torch.cat([c.argmax(dim=1) for c in d["t"].split(1024)]).to(torch.int32)
        st["advantage"] = torch.randn(N, generator=gen, device=DEV).mul_(0.7).sub_(0.2)
        st["mask"] = _mask(gen, N) if case["masked"] else None
        st["seq_start"] = torch.tensor(sorted(set(list(range(0, N, 512)) + [N])), dtype=torch.int64, device=DEV)
        st["g"] = torch.empty_like(d["s"])
        return st
    st["s"], st["t"], st["proposal"] = d["s"], d["t"], d["proposal"]
    if call == "train":
        out = saki.alloc_outputs(N, torch.device(DEV))
        st["out"] = {k: out[k] for k in TRAIN_FIELDS}
        st["g"] = torch.empty_like(d["s"])
        st["mask"] = _mask(gen, N) if case["masked"] else None
    elif call == "vshard":
        st["slices"] = [(d["s"][:, v0:v0 + n].contiguous(), d["t"][:, v0:v0 + n].contiguous(), v0)
                        for v0, n in split_columns(V, case["world"])]
        del st["s"], st["t"]
    elif call == "host":
        for k in ("s", "t", "proposal"):
            st[k] = d[k].cpu().pin_memory()
        st["out"] = {k: v.cpu().pin_memory() for k, v in saki.alloc_outputs(N, torch.device(DEV)).items()}
        st["g"] = torch.empty(st["s"].shape, dtype=st["s"].dtype, pin_memory=True)
    return st


def run(st):
    c, seed = st["case"], st["seed"]
    call, tau = c["call"], c["temperature"]
    if call == "fwd":
        return saki.route_fwd(st["s"], st["t"], st["proposal"], c["eps"], tau, seed)
    if call == "train":
        return saki.route_fwd_bwd(st["s"], st["t"], st["proposal"], c["eps"], tau, seed, mask=st["mask"],
                                  grad_scale=1.0 / c["N"], out=st["out"], dlogits=st["g"])
    if call == "spec":
        return saki.spec_verify(st["s"], st["t"], st["draft"], c["eps"], tau, seed)
    if call == "meta":
        corrected, selected = st["corrected"], None
        if c["control"] != "none":
            mode = saki.SELECT_TV_WEIGHTED if c["control"] == "tv" else saki.SELECT_RANDOM
            corrected, _ = selected = saki.select_tm(st["seq_start"], corrected, st["tv"], mode, seed, mask=st["mask"])
        return selected, saki.route_bwd_from_meta(st["s"], corrected, st["proposal"], st["teacher_top1"], st["advantage"], tau,
                                                  mask=st["mask"], grad_scale=1.0 / c["N"], dlogits=st["g"])
    if call == "lmhead":
        return saki.lmhead_lse(st["hidden"], st["weight"], tau, logits=st["logits"], scratch=st["scratch"])
    if call == "vshard":
        out, gs, _ = route_vocab_sharded_local(st["slices"], c["V"], st["proposal"], c["eps"], tau, seed, grad_scale=1.0 / c["N"])
        return out, gs
    if call == "sample":
        return saki.sample_proposal(st["s"], tau, seed)
    return saki.route_host(st["s"], st["t"], st["proposal"], c["eps"], tau, seed, grad_scale=1.0 / c["N"], out=st["out"],
                           dlogits=st["g"])


def work(case):
    call = case["call"]
    es = 4 if case.get("dtype") == "f32" else 2
    if call == "lmhead":
        N, V, d = case["N"], case["V"], case["d"]
        return dict(bytes=2 * (N * d + V * d + N * V) + 8 * N, flops=2 * N * V * d)
    if call == "spec":
        # positions up to a sequence's first rejection; a position is rejected with probability TV <= sqrt(eps/2),
        # about four fifths of that bound on these logits
        r = min(0.9, 0.8 * math.sqrt(case["eps"] / 2))
        positions = case["B"] * (1 - (1 - r) ** (case["K"] + 1)) / r
        return dict(bytes=int(positions * 2 * case["V"] * es + case["B"] * (case["K"] + 1) * 53), flops=0)
    N, V = case["N"], case["V"]
    # rows read and written, and the per-position outputs
    rows, scalars = {"fwd": (2, 61), "train": (3, 45), "meta": (2, 30), "vshard": (3, 61), "sample": (1, 4), "host": (3, 61)}[call]
    return dict(bytes=N * (rows * V * es + scalars), flops=0)


def tolerance(case):
    call = case["call"]
    if call == "sample":
        return "exact"                      # keys are formed in float64
    if case.get("dtype") == "f32":
        return dict(rel=1e-5)
    if call in ("meta", "lmhead"):
        return dict(rel=4e-3)               # bf16 gradient / logits: half an ulp is 2^-9
    # bf16 routing: bf16 gradients, and float32 scalars (lambda to 1e-5).  A token drawn by inverse CDF over up to
    # 160000 cells moves to the neighbouring cell where float32 rounding of the running sum crosses its edge: a few in
    # a thousand draws, each with the log-probabilities of its token.
    if call == "train":
        return dict(rel=4e-3, differ=0.005)
    return dict(rel=1e-2, max=0.9, differ=0.005)
