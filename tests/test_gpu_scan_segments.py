"""Segmented scan at the segment counts and lengths its rule gives: three segments and many, the shortest ones, a last one
of the same length and of nearly twice it, an odd number of chunks; weak decay, so that entry states carry through;
against the one-pass scan and the oracle."""
import numpy as np
import pytest

from paper_2602_03681_b200 import binding, inputs
from test_gpu_parity import TOL, check_fwd, rel_err, run_fwd, run_oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,H,L,oracle", [("cfg1_bf16_prefill", 1, 1024, True), ("cfg1_bf16_prefill", 30, 1024, False), ("cfg1_bf16_prefill", 3, 1984, True),
                                             ("cfg1_bf16_prefill", 16, 2112, False), ("cfg1_bf16_prefill", 32, 1088, False),
                                             ("cfg4_bf16_train", 2, 1088, True), ("cfg4_bf16_train", 5, 4160, False)])
def test_segments(name, H, L, oracle):
    wl = inputs.WORKLOADS[name]
    x = inputs.make_layer_inputs(wl, B=1, H=H, L=L)
    x["g"] = np.full((1, L, H), -1e-3, np.float32)
    S0 = (0.2 * np.random.default_rng(5).standard_normal((1, H, wl.d, wl.d))).astype(np.float32)
    seg = run_fwd(wl, x, state_in=S0)
    one = run_fwd(wl, x, state_in=S0, flags=binding.SINGLE_PASS_SCAN)
    for n in ("o_la", "state_out"):
        assert rel_err(seg[n], one[n]) <= TOL["bf16"], n
    if oracle:
        check_fwd(wl, seg, run_oracle(wl, x, state_in=S0), TOL["bf16"])


# the last number of pairs that is cut into segments and the first that is not, 128 and 64 columns, with block-level routing
# too
@pytest.mark.parametrize("name,H,block", [("cfg1_bf16_prefill", 22, False), ("cfg1_bf16_prefill", 23, False),
                                          ("cfg4_bf16_train", 30, False), ("cfg4_bf16_train", 31, False),
                                          ("cfg4_bf16_train", 18, True), ("cfg4_bf16_train", 19, True),
                                          ("cfg1_bf16_prefill", 14, True), ("cfg1_bf16_prefill", 15, True)])
def test_segments_at_the_lines(name, H, block):
    wl = inputs.WORKLOADS[name]
    L = 1536
    x = inputs.make_layer_inputs(wl, B=1, H=H, L=L)
    if block:
        x["route"] = np.repeat((np.random.default_rng(3).random((1, L // 64, H)) < 0.3).astype(np.uint8), 64, axis=1)
    x["g"] = np.full((1, L, H), -1e-3, np.float32)
    flags = binding.BLOCK_ROUTING if block else 0
    seg, one = run_fwd(wl, x, flags=flags), run_fwd(wl, x, flags=flags | binding.SINGLE_PASS_SCAN)
    for n in ("o_la", "state_out"):
        assert rel_err(seg[n], one[n]) <= TOL["bf16"], n
