"""Rows on two SMs, as dispatched.  Rows of more than 98304 elements in calls of up to a row per SM take two blocks of eight
warps; pinned they take one block of sixteen.  Both add the sums of the sixteen warps in the same order."""
import pytest
import torch

import paper_2609_36601_b200 as P
from paper_2609_36601_b200 import synth

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def spread_over_warps(d, V, seed):
    """Lowers each sixteenth of a row (a warp's part) by up to 80 nats, so that the warps' sums differ by many binary orders."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    part = torch.arange(V, device=DEV) // 256 * 16 // ((V + 255) // 256)
    off = -80.0 * torch.rand((d["s"].shape[0], 16), generator=gen, device=DEV) ** 2
    for k in ("s", "t"):
        d[k].copy_((d[k].float() + off[:, part]).to(torch.bfloat16))


@pytest.mark.parametrize("V", [98312, 131072, 151936])
@pytest.mark.parametrize("eps", [0.002, 0.1])
@pytest.mark.parametrize("apart", [False, True])
def test_pair_of_blocks_agrees_with_one_block_to_the_bit(V, eps, apart):
    N = torch.cuda.get_device_properties(0).multi_processor_count
    w = synth.Workload("pair", N, V, "bf16", eps, 1.5, True, 1200 + V % 97, 33)
    d = synth.generate(w, DEV)
    if apart:
        spread_over_warps(d, V, 5)
    out, g = P.route_fwd_bwd(d["s"], d["t"], d["proposal"], w.eps, seed=w.seed)
    assert P.last_kernel() == 3
    prev = P.set_kernel(3)
    try:
        one, g_one = P.route_fwd_bwd(d["s"], d["t"], d["proposal"], w.eps, seed=w.seed)
    finally:
        P.set_kernel(prev)
    torch.cuda.synchronize()
    for k in out:
        assert torch.equal(out[k], one[k]), k
    assert torch.equal(g, g_one)


# (blocks per row, blocks per SM), as dispatched and with the kernel pinned
@pytest.mark.parametrize("V,N,layout,pinned", [(8192, 100, (1, 2), (1, 4)), (8192, 2000, (1, 4), (1, 4)), (8192, 304, (1, 4), (1, 4)),
                                               (9200, 320, (1, 4), (1, 4)), (24000, 156, (1, 2), (1, 4)), (65536, 74, (2, 1), (1, 2)), (65536, 148, (2, 2), (1, 2)),
                                               (65536, 900, (1, 2), (1, 2)), (98304, 74, (2, 1), (1, 2)), (98312, 74, (2, 2), (1, 1)), (151936, 40, (2, 2), (1, 1)),
                                               (151936, 447, (2, 2), (1, 1)), (262144, 150, (2, 2), (1, 1))])
def test_layouts(V, N, layout, pinned):
    assert torch.cuda.get_device_properties(0).multi_processor_count == 148, "the shapes are chosen for 148 SMs"
    w = synth.Workload("layout", N, V, "bf16", 0.1, 1.5, True, 7, 7)
    d = synth.generate(w, DEV)
    for which, want in ((0, layout), (3, pinned)):
        prev = P.set_kernel(which)
        try:
            P.route_fwd(d["s"], d["t"], d["proposal"], w.eps, seed=w.seed)
            assert P.last_kernel() == 3 and P.last_rowsm_layout() == want, which
        finally:
            P.set_kernel(prev)
    prev = P.set_kernel(1)
    try:
        P.route_fwd(d["s"], d["t"], d["proposal"], w.eps, seed=w.seed)
        assert P.last_rowsm_layout() == (0, 0)
    finally:
        P.set_kernel(prev)
    torch.cuda.synchronize()
