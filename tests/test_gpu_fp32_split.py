"""fp32 forward on either side of the pair, chunk and block counts at which its kernels cut their work finer, against the
oracle."""
import numpy as np
import pytest
import torch

from paper_2602_03681_b200 import inputs
from test_gpu_parity import TOL, check_fwd, run_fwd, run_oracle

pytestmark = pytest.mark.gpu


# (64 columns: 111 chunks are the last that the prepare kernel cuts into four)
@pytest.mark.parametrize("B,H,L", [(1, 73, 64), (2, 37, 64), (1, 49, 192), (1, 50, 192), (3, 25, 320), (1, 37, 192), (1, 28, 256)])
def test_fp32_forward(B, H, L):
    wl = inputs.WORKLOADS["cfg0_f32_tiny_fwd"]
    x = inputs.make_layer_inputs(wl, B=B, H=H, L=L)
    check_fwd(wl, run_fwd(wl, x), run_oracle(wl, x), TOL["f32"])


# 128 columns: 74 chunks (cut into four by the prepare kernel) and 75, 36 and 37 pairs (narrow and wide scan slices)
@pytest.mark.parametrize("B,H,L", [(1, 37, 128), (1, 25, 192), (1, 36, 64), (1, 2, 704)])
def test_fp32_forward_128_columns(B, H, L):
    import dataclasses
    wl = dataclasses.replace(inputs.WORKLOADS["cfg0_f32_tiny_fwd"], d=128)
    x = inputs.make_layer_inputs(wl, B=B, H=H, L=L)
    check_fwd(wl, run_fwd(wl, x), run_oracle(wl, x), TOL["f32"])


# no retained token at all, and nothing else; one chunk and a ragged number of key tiles
@pytest.mark.parametrize("L", [64, 192])
@pytest.mark.parametrize("retained", [0, 1])
def test_fp32_forward_one_branch_empty(L, retained):
    wl = inputs.WORKLOADS["cfg0_f32_tiny_fwd"]
    x = inputs.make_layer_inputs(wl, B=1, H=2, L=L)
    x["route"] = np.full_like(x["route"], retained)
    check_fwd(wl, run_fwd(wl, x), run_oracle(wl, x), TOL["f32"])


# A value out of range stays causal: the rows before its token are those of a call without it, bit for bit (tokens at edges
# of the kernels' groups of 4, 8, 16 and 32 rows; narrow and wide scan slices).
@pytest.mark.parametrize("value", [np.inf, np.nan])
@pytest.mark.parametrize("d,B,H", [(64, 1, 2), (64, 1, 73), (128, 1, 2), (128, 1, 40)])
def test_fp32_forward_value_out_of_range_reaches_no_earlier_token(d, B, H, value):
    import dataclasses

    from paper_2602_03681_b200 import binding
    from test_gpu_parity import dev
    wl, L, dt = dataclasses.replace(inputs.WORKLOADS["cfg0_f32_tiny_fwd"], d=d), 192, torch.float32
    x = inputs.make_layer_inputs(wl, B=B, H=H, L=L)
    x["route"] = np.zeros_like(x["route"])
    x["route"][:, ::64] = 1

    def fwd(v):
        r = binding.hybrid_fwd(dev(x["q"], dt), dev(x["k"], dt), v, dev(x["g"]), dev(x["beta"]), dev(x["route"]), dev(x["w"]),
                               scale_la=wl.scale_la, scale_sm=wl.scale_sm, want=("o_la",))
        return r["out"], r["o_la"]

    v = dev(x["v"], dt)
    plain = fwd(v)
    for t in (1, 3, 4, 7, 8, 15, 31, 32, 33, 63, 65, 100, 190):
        bad = v.clone()
        bad[:, t, :, 5] = value
        for a, b in zip(fwd(bad), plain):
            assert torch.equal(a[:, :t], b[:, :t]), t
            assert not torch.isfinite(a[:, t, :, 5]).any(), t
