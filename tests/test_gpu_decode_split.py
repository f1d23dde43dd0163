"""Decode step at the edges of how its work is split: (sequence, head) counts on either side of one resident set
of items, caches of every length from empty to beyond a slice of every part, against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from oracle import grouped
from paper_2602_03681_b200 import inputs
from test_gpu_parity import TOL, check_stored, dev, rel_err, tdtype

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,B,H", [("cfg3_bf16_decode", 1, 1), ("cfg3_bf16_decode", 14, 7),
                                      ("cfg3_bf16_decode", 9, 11), ("cfg4_bf16_train", 25, 12),
                                      ("cfg0_f32_tiny_fwd", 20, 15)])
def test_decode_ragged_caches(name, B, H):
    from paper_2602_03681_b200 import binding
    wl = inputs.WORKLOADS[name]
    cap, T = 600, 2
    x = inputs.make_decode_inputs(wl, B=B, H=H, steps=T, ctx_retained=cap - T, cap=cap)
    lengths = np.array([0, 1, 31, 32, 33, 63, 64, 65, 127, 129, 255, 257, 383, 511, 512, 513, 577, cap - T])
    rng = np.random.default_rng(7)
    x["cache_len"][...] = rng.permutation(np.resize(lengths, B * H)).reshape(B, H)
    dt = tdtype(wl)
    state, kc, vc, n = dev(x["state"]), dev(x["k_cache"], dt), dev(x["v_cache"], dt), dev(x["cache_len"])
    p = binding.make_params(B, H, 0, wl.d, binding._dtype_code(kc), wl.scale_la, wl.scale_sm)
    ws = binding.alloc_workspace(p, binding.OP_DECODE)
    o_state, o_n = x["state"].astype(np.float64), x["cache_len"].copy()
    o_kc, o_vc = x["k_cache"].astype(np.float64), x["v_cache"].astype(np.float64)
    for t in range(T):
        w = dev(x["w"][t])
        p.w = w.data_ptr()
        out = torch.empty((B, H, wl.d), dtype=dt, device="cuda")
        binding.natsl_decode_step(dev(x["q"][t], dt), dev(x["k"][t], dt), dev(x["v"][t], dt), dev(x["g"][t]),
                                  dev(x["beta"][t]), dev(x["route"][t]), state, kc, vc, n, out, p, ws)
        ref = oracle.decode_step(x["q"][t], x["k"][t], x["v"][t], x["g"][t], x["beta"][t], x["route"][t], x["w"][t],
                                 o_state, o_kc, o_vc, o_n, scale_la=wl.scale_la, scale_sm=wl.scale_sm)
        check_stored(out.float().cpu().numpy(), ref["out"], TOL[wl.dtype], wl.dtype, f"step{t}")
    assert binding.natsl_device_status(ws) == 0
    assert np.array_equal(n.cpu().numpy(), o_n)
    assert rel_err(state.cpu().numpy(), o_state) <= 1e-4


@pytest.mark.parametrize("B,H,cap", [(9, 11, 100), (9, 11, 301), (14, 7, 601), (8, 8, 1201), (20, 15, 64)])
def test_decode_split_follows_the_capacity(B, H, cap):
    """Capacities at which a pair's cache is cut differently: a step on caches of mixed lengths, against the oracle."""
    from paper_2602_03681_b200 import binding
    wl = inputs.WORKLOADS["cfg3_bf16_decode"]
    x = inputs.make_decode_inputs(wl, B=B, H=H, steps=1, ctx_retained=cap - 1, cap=cap)
    x["cache_len"][...] = np.resize(np.array([0, 1, cap // 3, cap // 2 + 1, cap - 1]), B * H).reshape(B, H)
    dt = tdtype(wl)
    state, kc, vc, n, w = dev(x["state"]), dev(x["k_cache"], dt), dev(x["v_cache"], dt), dev(x["cache_len"]), dev(x["w"][0])
    p = binding.make_params(B, H, 0, wl.d, binding._dtype_code(kc), wl.scale_la, wl.scale_sm, w=w)
    ws = binding.alloc_workspace(p, binding.OP_DECODE)
    out = torch.empty((B, H, wl.d), dtype=dt, device="cuda")
    binding.natsl_decode_step(dev(x["q"][0], dt), dev(x["k"][0], dt), dev(x["v"][0], dt), dev(x["g"][0]),
                              dev(x["beta"][0]), dev(x["route"][0]), state, kc, vc, n, out, p, ws)
    ref = oracle.decode_step(x["q"][0], x["k"][0], x["v"][0], x["g"][0], x["beta"][0], x["route"][0], x["w"][0],
                             x["state"].astype(np.float64), x["k_cache"].astype(np.float64),
                             x["v_cache"].astype(np.float64), x["cache_len"].copy(),
                             scale_la=wl.scale_la, scale_sm=wl.scale_sm)
    check_stored(out.float().cpu().numpy(), ref["out"], TOL[wl.dtype], wl.dtype, "step")
    assert binding.natsl_device_status(ws) == 0


def _steps(wl, x, n, cap, B, H):
    """Two steps of x's first token on caches of n entries in cap rows: out, state, cache_len, k_cache, v_cache."""
    from paper_2602_03681_b200 import binding
    dt = tdtype(wl)
    kc, vc = (torch.zeros((B, H, cap, wl.d), dtype=dt, device="cuda") for _ in range(2))
    rows = min(cap, x["k_cache"].shape[2])
    kc[:, :, :rows], vc[:, :, :rows] = dev(x["k_cache"], dt)[:, :, :rows], dev(x["v_cache"], dt)[:, :, :rows]
    state, n, w = dev(x["state"]), dev(n), dev(x["w"][0])
    p = binding.make_params(B, H, 0, wl.d, binding._dtype_code(kc), wl.scale_la, wl.scale_sm, w=w)
    ws = binding.alloc_workspace(p, binding.OP_DECODE)
    out = torch.empty((B, H, wl.d), dtype=dt, device="cuda")
    for _ in range(2):          # (the second step finds the first one's tickets and partial results)
        binding.natsl_decode_step(dev(x["q"][0], dt), dev(x["k"][0], dt), dev(x["v"][0], dt), dev(x["g"][0]),
                                  dev(x["beta"][0]), dev(x["route"][0]), state, kc, vc, n, out, p, ws)
    assert binding.natsl_device_status(ws) == 0
    return out, state, n, kc, vc


def _oracle_steps(wl, x, n):
    o = [x["state"].astype(np.float64), x["k_cache"].astype(np.float64), x["v_cache"].astype(np.float64), n.copy()]
    for _ in range(2):
        ref = oracle.decode_step(x["q"][0], x["k"][0], x["v"][0], x["g"][0], x["beta"][0], x["route"][0], x["w"][0], *o,
                                 scale_la=wl.scale_la, scale_sm=wl.scale_sm)
    return ref["out"], o


@pytest.mark.parametrize("name,B,H,most", [("cfg3_bf16_decode", 8, 8, 200), ("cfg3_bf16_decode", 12, 6, 1300),
                                           ("cfg3_bf16_decode", 8, 12, 700), ("cfg4_bf16_train", 9, 11, 900),
                                           ("cfg0_f32_tiny_fwd", 20, 15, 320)])
def test_decode_split_goes_by_length(name, B, H, most):
    """Mixed lengths in caches that hold them just so and in roomy ones: the same bits, because how a pair's cache is cut
    depends on its length alone, and the oracle's values."""
    wl = inputs.WORKLOADS[name]
    x = inputs.make_decode_inputs(wl, B=B, H=H, steps=1, ctx_retained=most, cap=most + 2)
    lengths = np.unique(np.minimum([0, 1, 31, 33, 100, 299, 300, 301, 599, 600, 601, 900, 901, 1199, 1200, 1201, most], most))
    n = np.resize(np.random.default_rng(B).permutation(lengths), B * H).reshape(B, H).astype(np.int32)
    tight, roomy = (_steps(wl, x, n, cap, B, H) for cap in (most + 2, 5000))
    for a, b, what in zip(tight, roomy, ("out", "state", "cache_len", "k_cache", "v_cache")):
        assert torch.equal(a, b[:, :, :a.shape[2]] if what.endswith("cache") else b), what
    ref, o = _oracle_steps(wl, x, n)
    check_stored(roomy[0].float().cpu().numpy(), ref, TOL[wl.dtype], wl.dtype)
    assert np.array_equal(roomy[2].cpu().numpy(), o[3]) and rel_err(roomy[1].cpu().numpy(), o[0]) <= 1e-4


@pytest.mark.parametrize("cap", [8, 400])
def test_decode_more_items_than_a_resident_set_can_list(cap):
    """16384 pairs: the CTAs that list their items are more than are resident at once."""
    wl = inputs.WORKLOADS["cfg4_bf16_train"]
    B, H = 256, 64
    x = inputs.make_decode_inputs(wl, B=B, H=H, steps=1, ctx_retained=6, cap=8)
    n = (np.arange(B * H) % 7).reshape(B, H).astype(np.int32)
    got = _steps(wl, x, n, cap, B, H)
    ref, o = _oracle_steps(wl, x, n)
    check_stored(got[0].float().cpu().numpy(), ref, TOL[wl.dtype], wl.dtype)
    assert np.array_equal(got[2].cpu().numpy(), o[3])


def _grouped_step(x, n, state, kc, vc, G, scale_la, scale_sm, norm_eps, eps=1e-5):
    """One step with normalised q, k and G softmax heads per linear head, from the definitions: out and new state."""
    t = {m: torch.from_numpy(np.asarray(x[m][0], np.float64)) for m in ("q", "k", "v", "g", "beta", "w")}
    route = torch.from_numpy(x["route"][0].astype(np.int64))
    B, H, d = t["q"].shape
    q, k = (grouped.l2_normalise(t[m], norm_eps) for m in ("q", "k"))
    S = torch.exp(t["g"])[..., None, None] * torch.from_numpy(state)
    fold = t["beta"] * (route != 1)
    S = S + fold[..., None, None] * k[..., :, None] * (t["v"] - torch.einsum("bha,bhac->bhc", k, S))[..., None, :]
    o_la = scale_la * torch.einsum("bha,bhac->bhc", q, S)
    sl = lambda a: a.reshape(*a.shape[:-1], G, d // G)
    keys = torch.cat([torch.from_numpy(kc), t["k"][:, :, None]], 2)          # the cache, then the token itself
    values = torch.cat([torch.from_numpy(vc), t["v"][:, :, None]], 2)
    logits = scale_sm * torch.einsum("bhsa,bhmsa->bhsm", grouped.rms_normalise(sl(t["q"]), norm_eps),
                                     grouped.rms_normalise(sl(keys), norm_eps))
    seen = torch.arange(keys.shape[2]) < torch.from_numpy(n.astype(np.int64))[..., None]
    seen[..., -1] = route != 0
    p = torch.softmax(logits.masked_fill(~seen[:, :, None], -torch.inf), -1).nan_to_num(0.0)   # (no key: zero)
    o_nla = torch.einsum("bhsm,bhmsc->bhsc", p, sl(values))
    rms = lambda a: a * torch.rsqrt((a * a).mean(-1, keepdim=True) + eps)
    return (t["w"][..., :1] * rms(o_nla).reshape(B, H, d) + t["w"][..., 1:] * rms(o_la)).numpy(), S.numpy()


@pytest.mark.parametrize("name,B,H,G,cap", [("cfg3_bf16_decode", 9, 12, 2, 500), ("cfg3_bf16_decode", 9, 12, 2, 4000),
                                            ("cfg3_bf16_decode", 12, 8, 2, 1700), ("cfg4_bf16_train", 20, 15, 1, 280),
                                            ("cfg0_f32_tiny_fwd", 20, 6, 2, 1000)])
def test_decode_going_round_with_grouped_heads(name, B, H, G, cap):
    """More pairs than a resident set holds (or long caches of nearly as many), softmax heads of their own and q, k
    normalised as read; mixed lengths and routes."""
    from paper_2602_03681_b200 import binding
    wl = inputs.WORKLOADS[name]
    most = min(cap - 1, 1600)
    x = inputs.make_decode_inputs(wl, B=B, H=H, steps=1, ctx_retained=most, cap=most)
    r = np.random.default_rng(3)
    for m in ("q", "k"):
        x[m] = (x[m] * np.exp(0.5 * r.standard_normal(x[m].shape[:-1] + (1,)))).astype(np.float32)
        if wl.dtype == "bf16":
            x[m] = inputs.round_bf16(x[m])
    x["route"][...] = r.integers(0, 3, x["route"].shape)
    n = np.resize(r.permutation([0, 1, 33, 299, 301, 600, 601, 1201, most]), B * H).reshape(B, H).clip(0, most).astype(np.int32)
    scale_sm, dt = (wl.d // G) ** -0.5, tdtype(wl)
    kc, vc = (torch.zeros((B, H, cap, wl.d), dtype=dt, device="cuda") for _ in range(2))
    kc[:, :, :most], vc[:, :, :most] = dev(x["k_cache"], dt), dev(x["v_cache"], dt)
    state, length, w = dev(x["state"]), dev(n), dev(x["w"][0])
    p = binding.make_params(B, H, 0, wl.d, binding._dtype_code(kc), wl.scale_la, scale_sm, w=w, G=G, norm_eps=1e-6,
                            flags=binding.QK_NORM)
    ws = binding.alloc_workspace(p, binding.OP_DECODE)
    out = torch.empty((B, H, wl.d), dtype=dt, device="cuda")
    binding.natsl_decode_step(dev(x["q"][0], dt), dev(x["k"][0], dt), dev(x["v"][0], dt), dev(x["g"][0]),
                              dev(x["beta"][0]), dev(x["route"][0]), state, kc, vc, length, out, p, ws)
    assert binding.natsl_device_status(ws) == 0
    ref, S = _grouped_step(x, n, x["state"].astype(np.float64), x["k_cache"].astype(np.float64),
                           x["v_cache"].astype(np.float64), G, wl.scale_la, scale_sm, 1e-6)
    check_stored(out.float().cpu().numpy(), ref, TOL[wl.dtype], wl.dtype)
    assert rel_err(state.cpu().numpy(), S) <= 1e-4
    assert np.array_equal(length.cpu().numpy(), n + (x["route"][0] != 0))
