"""Segmented scan at the segment counts and lengths its rule gives: three segments and many, the shortest ones, a last one
of the same length and of nearly twice it, an odd number of chunks; weak decay, so that entry states carry through;
against the one-pass scan and the oracle.  How many kernels a call launches says which of the two it was: a first pass and the
chaining are two more."""
import numpy as np
import pytest
import torch

from paper_2602_03681_b200 import binding, inputs
from test_gpu_parity import TOL, check_fwd, dev, rel_err, run_oracle, tdtype

pytestmark = pytest.mark.gpu


def both_ways(wl, x, flags=0, G=0, state_in=None):
    """What the call returns by default and with one pass, and whether the default cut the scan into segments."""
    res, launches = [], []
    for f in (0, binding.SINGLE_PASS_SCAN):
        before = binding.natsl_launch_count()
        r = binding.hybrid_fwd(*(dev(x[n], tdtype(wl)) for n in ("q", "k", "v")), dev(x["g"]), dev(x["beta"]), dev(x["route"]),
                               dev(x["w"]), scale_la=wl.scale_la, scale_sm=wl.scale_sm, flags=flags | f, G=G,
                               state_in=None if state_in is None else dev(state_in), want=("o_la", "o_nla", "lse", "state_out"))
        launches.append(binding.natsl_launch_count() - before)
        torch.cuda.synchronize()
        assert binding.natsl_device_status(r["ws"]) == 0
        res.append({n: t.float().cpu().numpy() for n, t in r.items() if n != "ws"})
    assert launches[0] - launches[1] in (0, 2)
    return (*res, launches[0] != launches[1])


# (64 columns, 30 pairs: segments of 8, 8 and 16 chunks; 128 columns, 22 pairs: 8, 8 and 15)
@pytest.mark.parametrize("name,H,L,oracle", [("cfg1_bf16_prefill", 1, 1024, True), ("cfg1_bf16_prefill", 22, 1984, False), ("cfg1_bf16_prefill", 3, 1984, True),
                                             ("cfg1_bf16_prefill", 16, 2112, False), ("cfg1_bf16_prefill", 20, 1088, False),
                                             ("cfg4_bf16_train", 2, 1088, True), ("cfg4_bf16_train", 5, 4160, False),
                                             ("cfg4_bf16_train", 30, 2048, True)])
def test_segments(name, H, L, oracle):
    wl = inputs.WORKLOADS[name]
    x = inputs.make_layer_inputs(wl, B=1, H=H, L=L)
    x["g"] = np.full((1, L, H), -1e-3, np.float32)
    S0 = (0.2 * np.random.default_rng(5).standard_normal((1, H, wl.d, wl.d))).astype(np.float32)
    seg, one, cut = both_ways(wl, x, state_in=S0)
    assert cut
    for n in ("o_la", "state_out"):
        assert rel_err(seg[n], one[n]) <= TOL["bf16"], n
    if oracle:
        check_fwd(wl, seg, run_oracle(wl, x, state_in=S0), TOL["bf16"])


# the last number of pairs that is cut into segments and the first that is not: 128 and 64 columns, with block-level routing too,
# and 128 columns with two softmax heads, below and from 4096 tokens on.  What is not cut is the same call as with one pass and compared with the oracle.
@pytest.mark.parametrize("name,H,L,mode,cut", [("cfg1_bf16_prefill", 22, 1536, "token", True), ("cfg1_bf16_prefill", 23, 1536, "token", False),
                                               ("cfg4_bf16_train", 30, 2048, "token", True), ("cfg4_bf16_train", 31, 2048, "token", False),
                                               ("cfg4_bf16_train", 18, 1536, "block", True), ("cfg4_bf16_train", 19, 1536, "block", False),
                                               ("cfg1_bf16_prefill", 14, 1536, "block", True), ("cfg1_bf16_prefill", 15, 1536, "block", False),
                                               ("cfg1_bf16_prefill", 14, 1536, "two heads", True), ("cfg1_bf16_prefill", 15, 1536, "two heads", False),
                                               ("cfg1_bf16_prefill", 23, 4032, "token", False), ("cfg1_bf16_prefill", 23, 4096, "token", True),
                                               ("cfg1_bf16_prefill", 24, 4096, "token", False),
                                               ("cfg4_bf16_train", 20, 4096, "block", True), ("cfg4_bf16_train", 21, 4096, "block", False),
                                               ("cfg1_bf16_prefill", 18, 4096, "block", True), ("cfg1_bf16_prefill", 19, 4096, "block", False),
                                               ("cfg1_bf16_prefill", 16, 4096, "two heads", True), ("cfg1_bf16_prefill", 17, 4096, "two heads", False),
                                               ("cfg1_bf16_prefill", 15, 4096, "both", True), ("cfg1_bf16_prefill", 16, 4096, "both", False)])
def test_segments_at_the_lines(name, H, L, mode, cut):
    wl = inputs.WORKLOADS[name]
    x = inputs.make_layer_inputs(wl, B=1, H=H, L=L)
    block, heads = mode in ("block", "both"), 2 if mode in ("two heads", "both") else 0
    if block:
        x["route"] = np.repeat((np.random.default_rng(3).random((1, L // 64, H)) < 0.3).astype(np.uint8), 64, axis=1)
    x["g"] = np.full((1, L, H), -1e-3, np.float32)
    seg, one, was_cut = both_ways(wl, x, binding.BLOCK_ROUTING if block else 0, heads)
    assert was_cut == cut
    if cut:
        for n in ("o_la", "state_out"):
            assert rel_err(seg[n], one[n]) <= TOL["bf16"], n
        return
    for n in seg:
        assert np.array_equal(seg[n], one[n]), n
    ref = run_oracle(wl, x, block=64 if block else None)
    if heads:                       # (the linear branch does not see the softmax heads)
        for n in ("o_la", "state_out"):
            assert rel_err(seg[n], ref[n]) <= TOL["bf16"], n
    else:
        check_fwd(wl, seg, ref, TOL["bf16"])
