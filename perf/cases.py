"""The calls whose speed counts: generation, prefill, training and the score layer, each through the
entry points of ``paper_2602_03681_b200.binding`` that a program using the layer calls.

A case is a dict of plain values.  ``kind`` says which calls one pass makes:

  decode   ``steps`` generation steps of ``B`` sequences whose caches hold ``ctx`` retained tokens
  block    generation with the decision of a block open (route 2), ``steps`` tokens and the block's end
  prefill  one forward; with ``handoff`` it also returns the final state and the compacted cache
  piece    one forward that continues a sequence: ``ctx`` retained tokens in the cache, carried state
  train    forward that saves for the backward, then the backward: output and every gradient
  score    the attention score layer: features to one route per block and head

``mode`` is how the layer is set up: "token" (a route per token, unit-norm q and k, one softmax head per
linear head) or "paper" (the mode of the paper's models: one route per block of 64 tokens, q and k normalised
inside the kernels, two softmax heads of 64 columns per linear head at d = 128 and one at d = 64).
"""
import math

import torch

from paper_2602_03681_b200 import binding as nb

C = 64
EPS = 1e-5
NORM_EPS = 1e-6


def listed():
    return [
        # one user's chat: a token at a time, 1638 retained tokens (10 % of a context of 16384); latency and launches
        dict(name="decode_one_user", kind="decode", mode="token", dtype="bf16", B=1, H=16, d=128, ctx=1638, steps=8, p=0.1),
        # a serving batch of 64 at the same context: the memory-bound end of generation
        dict(name="decode_batch64", kind="decode", mode="token", dtype="bf16", B=64, H=16, d=128, ctx=1638, steps=8, p=0.1),
        # a block of the paper's mode generated with its decision open, then closed; ragged cache length
        dict(name="decode_block_paper", kind="block", mode="paper", dtype="bf16", B=12, H=6, d=128, ctx=771, steps=64, p=0.2),
        # fp32 storage, the arithmetic that bf16 results are checked against: two heads, 256 tokens
        dict(name="prefill_f32_tiny", kind="prefill", mode="token", dtype="f32", B=1, H=2, L=256, d=64, p=0.25, handoff=False),
        # a short prompt (five chunks) on its way to generation: time to first token
        dict(name="prefill_short", kind="prefill", mode="token", dtype="bf16", B=1, H=16, L=320, d=128, p=0.1, handoff=True),
        # the ordinary prefill: four sequences of 4096 tokens
        dict(name="prefill_4x4096", kind="prefill", mode="token", dtype="bf16", B=4, H=16, L=4096, d=128, p=0.1, handoff=False),
        # a long document: 32768 tokens, softmax tokens in clustered runs, slow decay
        dict(name="prefill_long", kind="prefill", mode="token", dtype="bf16", B=1, H=16, L=32768, d=128, p=0.05, handoff=True, runs=True),
        # the next piece of a long prompt: 8192 tokens behind 1203 retained ones
        dict(name="prefill_piece", kind="piece", mode="token", dtype="bf16", B=1, H=16, L=8192, d=128, p=0.05, ctx=1203, runs=True),
        # scoring text with a model of the paper's mode: six linear heads, twelve softmax heads
        dict(name="prefill_paper", kind="prefill", mode="paper", dtype="bf16", B=10, H=6, L=4096, d=128, p=0.2, handoff=False),
        # the score layer that routes such a model's blocks
        dict(name="score_layer", kind="score", mode="paper", dtype="bf16", B=4, H=16, L=4096, d=128, p=0.5, d_model=2048),
        # training, 64-column heads, a route per token
        dict(name="train_d64", kind="train", mode="token", dtype="bf16", B=8, H=12, L=2048, d=64, p=0.2),
        # training in the paper's mode: the largest case
        dict(name="train_paper", kind="train", mode="paper", dtype="bf16", B=10, H=6, L=4096, d=128, p=0.2),
    ]


def draw(rng):
    """One more case of the same ranges: sizes log-uniform, every kind, mode and head size."""
    def log(a, b):
        return min(b, max(a, int(round(math.exp(rng.uniform(math.log(a), math.log(b + 1)))))))

    most = {k: work(max(listed(), key=lambda c: (c["kind"] == k, work(c)["bytes"]))) for k in ("decode", "train")}
    while True:
        kind = rng.choice(["decode", "block", "prefill", "prefill", "piece", "train", "train", "score"])
        c = dict(kind=kind, mode="paper" if kind in ("block", "score") else rng.choice(["token", "token", "paper"]), dtype="bf16",
                 B=log(1, 16), H=rng.randint(2, 16), d=rng.choice([64, 128, 128]), p=round(math.exp(rng.uniform(math.log(0.05), math.log(0.4))), 3))
        if kind in ("decode", "block"):
            c.update(B=log(1, 64), ctx=log(64, 8192), steps=64 if kind == "block" else log(1, 16))
        else:
            c.update(L=C * log(1, 512 if kind in ("prefill", "piece") else 128))
        if kind == "prefill":
            c.update(handoff=rng.random() < 0.5)
            if c["mode"] == "token" and rng.random() < 0.15:      # fp32 storage: small calls only
                c.update(dtype="f32", B=log(1, 2), H=rng.randint(1, 8), L=C * log(1, 16))
            elif c["mode"] == "token" and rng.random() < 0.3:
                c.update(runs=True)
        if kind == "piece":
            c.update(ctx=log(64, 4096))
        if kind == "score":
            c.update(p=0.5, d_model=64 * log(4, 64))
        w, m = work(c), most["decode" if kind in ("decode", "block") else "train"]
        if w["bytes"] <= m["bytes"] and w["flops"] <= m["flops"]:
            return c


def _groups(c):
    return 2 if c["mode"] == "paper" and c["d"] == 128 else 1


def _flags(c):
    return nb.BLOCK_ROUTING | nb.QK_NORM if c["mode"] == "paper" else 0


def _params(c, L, w, flags=0, **opt):
    """The call's parameter block.  Logit scales: d^-1/2 for the linear read-out; for the softmax branch sqrt(d) on
    unit-norm q and k, (slice width)^-1/2 where the kernels normalise."""
    paper, G = c["mode"] == "paper", _groups(c)
    scale_sm = (c["d"] // G) ** -0.5 if paper else c["d"] ** 0.5
    code = nb.NATSL_F32 if c["dtype"] == "f32" else nb.NATSL_BF16
    return nb.make_params(c["B"], c["H"], L, c["d"], code, c["d"] ** -0.5, scale_sm, EPS, flags=flags, w=w, G=G,
                          norm_eps=NORM_EPS if paper else 0.0, **opt)


def _route(c, gen, shape, p):
    """[B,L,H]: softmax tokens by token, by block of 64 (paper's mode) or in clustered runs of mean length 8; the first
    token, or block, is one."""
    B, L, H = shape
    dev = "cuda"
    if c["mode"] == "paper":
        r = torch.rand((B, L // C, H), generator=gen, device=dev) < p
        r[:, 0] = True
        return r.to(torch.uint8).repeat_interleave(C, dim=1).contiguous()
    if c.get("runs"):
        n = int(L * p / 8 * 2) + 64
        u = torch.rand((B * H, n, 2), generator=gen, device=dev).clamp_(1e-7, 1 - 1e-7)
        mean = torch.tensor([8.0, 8.0 * (1 - p) / p], device=dev)
        length = torch.floor(torch.log(u) / torch.log1p(-1 / mean)) + 1           # geometric: run, gap, run, ...
        ends = length.reshape(B * H, 2 * n).cumsum(1)
        at = torch.arange(L, device=dev, dtype=torch.float32).expand(B * H, L).contiguous()
        r = (torch.searchsorted(ends.contiguous(), at, right=True) % 2 == 0)
        return r.to(torch.uint8).reshape(B, H, L).permute(0, 2, 1).contiguous()
    r = torch.rand((B, L, H), generator=gen, device=dev) < p
    r[:, 0] = True
    return r.to(torch.uint8)


def _tokens(c, gen, lead, H, d, dt):
    """q, k, v [*lead,H,d] and g, beta [*lead,H], w [*lead,H,2]."""
    def n(*s):
        return torch.randn((*lead, H, *s), generator=gen, device="cuda")

    q, k, v = n(d), n(d), n(d)
    if c["mode"] == "token":          # (paper's mode: the kernels normalise)
        q, k = torch.nn.functional.normalize(q, dim=-1), torch.nn.functional.normalize(k, dim=-1)
    g = -torch.nn.functional.softplus(n() - (2.0 if c.get("runs") else 0.0))
    return dict(q=q.to(dt), k=k.to(dt), v=v.to(dt), g=g, beta=torch.sigmoid(n()), w=torch.softmax(n(2), -1).contiguous())


def prepare(case, seed):
    c = case
    gen = torch.Generator(device="cuda").manual_seed(seed)
    dt = torch.float32 if c["dtype"] == "f32" else torch.bfloat16
    B, H, d = c["B"], c["H"], c["d"]
    s = dict(kind=c["kind"])
    if c["kind"] in ("decode", "block"):
        T, n0 = c["steps"], c["ctx"]
        t = _tokens(c, gen, (T, B), H, d, dt)
        if c["kind"] == "block":
            route = torch.full((T, B, H), 2, dtype=torch.uint8, device="cuda")
        else:
            route = (torch.rand((T, B, H), generator=gen, device="cuda") < c["p"]).to(torch.uint8)
        s["state"] = 0.02 * torch.randn((B, H, d, d), generator=gen, device="cuda")
        cap = n0 + T
        for m in ("k_cache", "v_cache"):
            s[m] = torch.zeros((B, H, cap, d), dtype=dt, device="cuda")
            s[m][:, :, :n0] = torch.randn((B, H, n0, d), generator=gen, device="cuda")
        s["ctx"] = torch.full((B, H), n0, dtype=torch.int32, device="cuda")
        s["cache_len"] = s["ctx"].clone()
        s["out"] = torch.empty((T, B, H, d), dtype=dt, device="cuda")
        s["steps"] = []
        for i in range(T):
            p = _params(c, 0, t["w"][i], flags=_flags(c))
            s["steps"].append((t["q"][i], t["k"][i], t["v"][i], t["g"][i], t["beta"][i], route[i], s["out"][i], p))
        s["keep"] = t["w"]
        s["ws"] = nb.alloc_workspace(s["steps"][0][-1], nb.OP_DECODE)
        if c["kind"] == "block":
            s["state_start"] = s["state"].clone()
            s["route_block"] = (torch.rand((B, H), generator=gen, device="cuda") < c["p"]).to(torch.uint8)
            s["g_block"] = t["g"].sum(0).contiguous()
        return s
    L = c["L"]
    if c["kind"] == "score":
        Dm = c["d_model"]
        s["x"] = torch.randn((B, L, Dm), generator=gen, device="cuda").to(dt)
        s["w_score"] = torch.randn((H, 2, Dm), generator=gen, device="cuda") / Dm ** 0.5
        s["scores"] = torch.empty((B, L // C, H, 2), dtype=torch.float32, device="cuda")
        s["route"] = torch.empty((B, L, H), dtype=torch.uint8, device="cuda")
        s["p"] = _params(c, L, None)
        return s
    s.update(_tokens(c, gen, (B, L), H, d, dt))
    s["route"] = _route(c, gen, (B, L, H), c["p"])
    s["out"] = torch.empty_like(s["q"])
    if c["kind"] == "train":
        s["dout"] = torch.randn((B, L, H, d), generator=gen, device="cuda").to(dt)
        s["grads"] = [torch.empty_like(s[m]) for m in ("q", "k", "v", "g", "beta", "w")]
        s["p"] = _params(c, L, s["w"], flags=_flags(c) | nb.SAVE_FOR_BWD)
        s["pb"] = _params(c, L, s["w"], flags=_flags(c) | nb.SAVED_FWD)
        if c["mode"] == "paper":
            s["dscore"] = torch.empty((B, L // C, H, 2), dtype=torch.float32, device="cuda")
            s["p"].dscore = s["pb"].dscore = s["dscore"].data_ptr()
        s["ws"] = nb.alloc_workspace(s["p"], nb.OP_BWD)
        return s
    opt, n0 = {}, c.get("ctx", 0)
    if c["kind"] == "piece" or c["handoff"]:
        opt["k_sm"], opt["v_sm"] = (torch.zeros((B, H, n0 + L, d), dtype=dt, device="cuda") for _ in range(2))
        opt["sm_len"] = torch.full((B, H), n0, dtype=torch.int32, device="cuda")
        opt["state_out"] = torch.empty((B, H, d, d), dtype=torch.float32, device="cuda")
        s["results"] = dict(opt)
    flags = _flags(c)
    if c["kind"] == "piece":
        flags |= nb.APPEND_CACHE
        for m in ("k_sm", "v_sm"):
            x = torch.randn((B, H, n0, d), generator=gen, device="cuda")
            if m == "k_sm" and c["mode"] == "token":
                x = torch.nn.functional.normalize(x, dim=-1)
            opt[m][:, :, :n0] = x
        opt["state_in"] = 0.02 * torch.randn((B, H, d, d), generator=gen, device="cuda")
        s["ctx"] = opt["sm_len"].clone()
    s["opt"] = opt
    s["p"] = _params(c, L, s["w"], flags=flags, sm_cap=n0 + L if opt else 0, **opt)
    s["ws"] = nb.alloc_workspace(s["p"], nb.OP_FWD)
    return s


def run(state):
    s = state
    kind = s["kind"]
    if kind in ("decode", "block"):
        s["cache_len"].copy_(s["ctx"])          # every pass generates from the same context
        for q, k, v, g, beta, route, out, p in s["steps"]:
            nb.natsl_decode_step(q, k, v, g, beta, route, s["state"], s["k_cache"], s["v_cache"], s["cache_len"], out, p, s["ws"])
        if kind == "block":
            nb.natsl_decode_block_end(s["route_block"], s["g_block"], s["state"], s["state_start"], s["cache_len"],
                                      len(s["steps"]), p, s["ws"])
        return dict(out=s["out"], state=s["state"], k_cache=s["k_cache"], v_cache=s["v_cache"], cache_len=s["cache_len"])
    if kind == "score":
        nb.natsl_score_layer(s["x"], s["w_score"], s["scores"], s["route"], s["p"])
        return dict(scores=s["scores"], route=s["route"])
    if kind == "piece":
        s["opt"]["sm_len"].copy_(s["ctx"])      # every pass appends to the same cache
    nb.natsl_hybrid_fwd(s["q"], s["k"], s["v"], s["g"], s["beta"], s["route"], s["out"], s["p"], s["ws"])
    if kind == "train":
        nb.natsl_hybrid_bwd(s["q"], s["k"], s["v"], s["g"], s["beta"], s["route"], s["dout"], *s["grads"], s["pb"], s["ws"])
        return dict(out=s["out"], **dict(zip(("dq", "dk", "dv", "dg", "dbeta", "dw"), s["grads"])), dscore=s.get("dscore"))
    return dict(out=s["out"], **s.get("results", {}))


def work(case):
    """Inputs read once, outputs written once; products of the chunkwise form over the tokens that take part (n linear
    tokens per chunk on average) and of the softmax branch over the keys a query sees, 2 operations per multiply-add."""
    c = case
    B, H, d, p = c["B"], c["H"], c["d"], c["p"]
    e = 4 if c["dtype"] == "f32" else 2
    if c["kind"] in ("decode", "block"):
        T, n = c["steps"], c["ctx"] + (c["steps"] / 2 if c["kind"] == "block" else c["p"] * c["steps"] / 2)
        per = 2 * d * d * 4 + 2 * n * d * e + 4 * d * e + 17
        end = (2 * d * d * 4) if c["kind"] == "block" else 0
        return dict(bytes=B * H * (T * per + end), flops=B * H * T * (8 * d * d + 4 * n * d))
    L = c["L"]
    NC = L // C
    if c["kind"] == "score":
        Dm = c["d_model"]
        return dict(bytes=B * L * Dm * e + 2 * H * Dm * 4 + B * NC * H * 8 + B * L * H, flops=B * L * Dm + 4 * B * NC * H * Dm)
    n = C if c["mode"] == "paper" else C * (1 - p)        # (block-level routing: every token takes part in its own block)
    seen = p * L / 2 + (C / 2 if c["mode"] == "paper" else 0) + c.get("ctx", 0)
    token = 17 + 4 * d * e                                # g, beta, w, route; q, k, v and out
    fwd = B * H * NC * (6 * n * n * d + 4 * C * n * d + 2 * d * d * (2 * n + C)) + B * H * L * 4 * d * seen
    kept = p * L * 2 * d * e if c["kind"] == "piece" or c.get("handoff") else 0
    if c["kind"] == "piece":
        kept += c["ctx"] * 2 * d * e
    state = {"piece": 2, "prefill": int(c.get("handoff", False)), "train": 0}[c["kind"]] * d * d * 4
    if c["kind"] == "train":
        token += 4 * d * e + 16                           # dout; dq, dk, dv; dg, dbeta, dw
        fwd += B * H * NC * (8 * C * n * d + 8 * n * d * d + 4 * C * d * d + 12 * n * n * d + 4 * n ** 3)
        fwd += B * H * L * 10 * d * seen
    return dict(bytes=B * H * (L * token + kept + state), flops=fwd)


def tolerance(case):
    if case["kind"] == "score":       # fp32 sums over 64 tokens and d_model columns; routes: ties
        return {"rel": 1e-5, "max": 1e-4, "differ": 1e-3}
    if case["dtype"] == "f32":
        return {"rel": 1e-5, "max": 1e-4}
    return {"rel": 1e-2, "max": 0.1}  # bf16 storage, 16-bit operands, fp32 accumulation
