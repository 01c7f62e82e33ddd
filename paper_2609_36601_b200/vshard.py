"""Vocabulary-sharded routing: the exchange around the library's stage calls.

Every rank holds a contiguous column slice of the logit rows (as a tensor-parallel lm-head leaves them).  A
row is routed in four stages; per stage a rank reduces its slice to 16 float64 numbers per row
(`vshard_partial`, a kernel), the ranks all-gather those (128 bytes per row, rank and stage; NCCL over NVLink on
GPUs, no logits ever cross), and every rank folds the gathered partials in rank order into the same per-row
state (`vshard_combine`, a kernel).  Stage 1 (one evaluation of the trust-region constraint) repeats until no
row is still solving: two waves as a rule (each moves to the root of a fourth-order model of the constraint).  This module holds no arithmetic: it
sequences the stages, moves the partials, and reads the counters of the waves.

`route_vocab_sharded` is the one-rank-per-process form over `torch.distributed`; `route_vocab_sharded_local`
runs the stages of all ranks in a single process on one device (the slices of all ranks are at hand), the slices in
one launch per stage, their partials written where the all-gather would put them.
"""
from __future__ import annotations

import torch

from . import binding as B

MAX_WAVES = 128
# Evaluation waves sent off before the host looks at the counters for the first time: two as a rule settle every row, and
# a wave that finds nothing to do costs less than a round trip to the host between waves.
EAGER_WAVES = 2


def _stages(wave, dev, eager):
    """Stage 0, evaluation waves until no row is solving (stage 1), stages 2 and 3.  Returns the number of waves that had
    a row to settle."""
    solving = torch.zeros(eager + 1, dtype=torch.int32, device=dev)
    counts = solving.unbind(0)
    wave(0, counts[0])
    for k in range(eager):
        wave(1, counts[k + 1])
    left = solving.tolist()                      # rows still solving after stage 0 and after each wave
    waves = left.index(0) if 0 in left else eager
    while left[-1] > 0 and waves < MAX_WAVES:
        wave(1, counts[-1])
        waves += 1
        left = [int(counts[-1].item())]
    wave(2)
    wave(3)
    return waves


def split_columns(V: int, world: int):
    """Contiguous, balanced column ranges: [(v0, V_local)] per rank, in rank order, tiling [0, V)."""
    base, extra = divmod(V, world)
    out, v0 = [], 0
    for r in range(world):
        n = base + (1 if r < extra else 0)
        out.append((v0, n))
        v0 += n
    return out


def route_vocab_sharded(s_loc, t_loc, v0: int, V: int, proposal, eps, temperature=1.0, seed=0, row_offset=0, mask=None,
                        grad_scale=1.0, backward=True, group=None, stream=None):
    """One rank's call: `s_loc`, `t_loc` are this rank's columns [v0, v0 + V_local) on its GPU.  Returns (out,
    dlogits_slice): the per-position outputs (identical on every rank) and this rank's columns of the gradient."""
    import torch.distributed as dist
    rank, world = dist.get_rank(group), dist.get_world_size(group)
    dev, N = s_loc.device, s_loc.shape[0]
    si = B.vshard_in(s_loc, t_loc, v0, V, proposal, eps, temperature, seed, row_offset, mask, rank, world)
    out = B.alloc_outputs(N, dev)
    g = torch.empty_like(s_loc) if backward else None
    # the slice's device and the caller's stream are the current ones: the exchange, the zeroing and the reading of the counters
    # are ordered with the stages
    with torch.cuda.device(dev), torch.cuda.stream(stream):
        state = torch.empty((N, B.VSHARD_STATE), dtype=torch.float64, device=dev)
        part = torch.empty((N, B.VSHARD_PARTIALS), dtype=torch.float64, device=dev)
        gathered = torch.empty((world, N, B.VSHARD_PARTIALS), dtype=torch.float64, device=dev)

        def wave(stage, n_solving=None):
            B.vshard_partial(si, stage, state if stage > 0 else None, part, g if stage == 2 else None, grad_scale, stream)
            dist.all_gather_into_tensor(gathered.view(-1), part.view(-1), group=group)
            B.vshard_combine(si, stage, gathered, state, out if stage == 3 else None, n_solving, stream)

        _stages(wave, dev, EAGER_WAVES)
    return out, g


def route_vocab_sharded_local(slices, V: int, proposal, eps, temperature=1.0, seed=0, row_offset=0, mask=None,
                              grad_scale=1.0, backward=True, stream=None, state_out=None):
    """All ranks in one process: `slices` = [(s_loc, t_loc, v0)] in rank order on one device.  Returns (out,
    [dlogits_slice per rank], waves): the stages every rank would run, the slices of all ranks in one launch per stage.
    `state_out`: a list that receives the per-row state tensor (for tests)."""
    out, gs, waves, state = B._tensors().vshard_local(slices, V, proposal, eps, temperature, seed, row_offset, mask, grad_scale,
                                                      backward, B._handle(stream), EAGER_WAVES + 1, MAX_WAVES)
    if state_out is not None:
        state_out.append(state)
    return out, gs, waves
