"""Softmax kernel with two warpgroups taking turns (64-column softmax heads): every number of key tiles from none to
beyond the ring, against the oracle, and many CTAs in flight giving the same bits every time -- a tile whose
probabilities are multiplied before all of its warps have written them shows up in either."""
import numpy as np
import pytest
import torch

from paper_2602_03681_b200 import inputs
from test_gpu_parity import TOL, check_fwd, dev, run_fwd, run_oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kept", [0, 1, 63, 64, 65, 128, 129, 192, 320, 449])
def test_tile_counts(kept):
    wl = inputs.WORKLOADS["cfg4_bf16_train"]
    B, H, L = 1, 2, 512
    route = np.zeros((B, L, H), np.uint8)
    route[:, :kept, 0] = 1
    route[:, L - kept:, 1] = 1
    x = inputs.make_layer_inputs(wl, B=B, H=H, L=L, route=route)
    check_fwd(wl, run_fwd(wl, x), run_oracle(wl, x), TOL["bf16"])


@pytest.mark.parametrize("d,G", [(128, 2), (64, 1)])
def test_same_bits_every_time(d, G):
    from paper_2602_03681_b200 import binding
    wl = inputs.WORKLOADS["cfg4_bf16_train"]
    gen = torch.Generator(device="cuda").manual_seed(5)
    B, H, L = 8, 6, 2048
    q, k, v = (torch.randn((B, L, H, d), generator=gen, device="cuda").bfloat16() for _ in range(3))
    g = -torch.rand((B, L, H), generator=gen, device="cuda")
    beta = torch.rand((B, L, H), generator=gen, device="cuda")
    route = dev(inputs.route_blocks(3, (B, L, H), 0.3))
    p = binding.make_params(B, H, L, d, binding.NATSL_BF16, d ** -0.5, (d // G) ** -0.5, G=G, norm_eps=1e-6,
                            flags=binding.BLOCK_ROUTING | binding.QK_NORM | binding.SAVE_FOR_BWD)
    ws = binding.alloc_workspace(p, binding.OP_BWD)
    first = None
    for _ in range(20):
        out = torch.empty_like(q)
        binding.natsl_hybrid_fwd(q, k, v, g, beta, route, out, p, ws)
        if first is None:
            first = out
        assert torch.equal(out, first)
    assert torch.isfinite(first.float()).all()
    assert binding.natsl_device_status(ws) == 0
