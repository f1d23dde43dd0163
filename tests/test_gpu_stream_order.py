"""Which kernels of a captured backward are ordered behind which: the edges of the graph, not the outcome of one run.
(A missing edge between the two streams gives the right bits whenever the reader happens to start late enough.)"""
import ctypes
import glob
import os
import re

import pytest
import torch

pytestmark = pytest.mark.gpu

# (writer, reader): the reader reads what the writer wrote
ALWAYS = [("combine_bwd", "gdn_rscan"), ("combine_bwd", "softmax_bwd_dq"), ("combine_bwd", "softmax_bwd_dkv"),
          ("gdn_rscan", "gdn_chunk_bwd"), ("gdn_scan", "combine_bwd"), ("softmax_combine", "combine_bwd")]
NORMED = [("to_f16_bhld", "softmax_bwd_dq"), ("to_f16_bhld", "softmax_bwd_dkv")]
BLOCK = [("softmax_bwd_dq", "softmax_bwd_own_block"), ("softmax_bwd_own_block", "gdn_chunk_bwd"),
         ("softmax_bwd_dkv", "gdn_chunk_bwd"), ("scatter", "gdn_chunk_bwd"), ("softmax_bwd_dkv", "scatter"),
         ("softmax_bwd_dkv", "dscore")]
TOKEN = [("softmax_bwd_dkv", "scatter"), ("softmax_bwd_dq", "gdn_chunk_bwd")]
TOKEN_NORMED = [("softmax_bwd_dkv", "scatter"), ("softmax_bwd_dq", "qk_norm_bwd"), ("gdn_chunk_bwd", "qk_norm_bwd"),
                ("scatter", "qk_norm_bwd")]


def kernels_and_paths(graph):
    """{node: kernel name}, {node: every node ordered behind it} and the nodes launched as programmatic dependents of a
    captured graph."""
    from cuda.bindings import driver as cu

    def ok(res):
        assert res[0] == cu.CUresult.CUDA_SUCCESS, res[0]
        return res[1] if len(res) == 2 else res[1:]

    g = cu.CUgraph(graph.raw_cuda_graph())
    nodes = ok(cu.cuGraphGetNodes(g, ok(cu.cuGraphGetNodes(g, 0))[1]))[0]
    # (edges by ctypes: the binding returns edge data that it has freed)
    get, m = ctypes.CDLL("libcuda.so.1").cuGraphGetEdges_v2, ctypes.c_size_t()
    h = ctypes.c_void_p(graph.raw_cuda_graph())
    assert get(h, None, None, None, ctypes.byref(m)) == 0
    src, dst = (ctypes.c_void_p * m.value)(), (ctypes.c_void_p * m.value)()
    data = (ctypes.c_ubyte * 8 * m.value)()                   # from_port, to_port, type, 5 reserved bytes
    assert get(h, src, dst, data, ctypes.byref(m)) == 0
    names = {}
    for n in nodes:
        if ok(cu.cuGraphNodeGetType(n)) == cu.CUgraphNodeType.CU_GRAPH_NODE_TYPE_KERNEL:
            prm = ok(cu.cuGraphKernelNodeGetParams(n))
            name = ok(cu.cuFuncGetName(prm.func)) if int(prm.func) else ok(cu.cuKernelGetName(prm.kern))
            names[int(n)] = name.decode()
    after = {int(n): set() for n in nodes}
    for a, b in zip(src, dst):
        after[int(a)].add(int(b))
    reach = {}

    def visit(n):
        if n not in reach:
            reach[n] = set()
            for x in after[n]:
                reach[n] |= {x} | visit(x)
        return reach[n]

    for n in after:
        visit(n)
    early = {int(b) for b, x in zip(dst, data) if x[2] == int(cu.CUgraphDependencyType.CU_GRAPH_DEPENDENCY_TYPE_PROGRAMMATIC)}
    return names, reach, early


def kernel_sources():
    """{kernel name: its body} of the library's sources."""
    found = {}
    for path in glob.glob(os.path.join(os.path.dirname(os.path.dirname(__file__)), "paper_2602_03681_b200", "csrc", "*.cu")):
        with open(path) as f:
            text = f.read()
        for m in re.finditer(r"__global__[^;{]*?\b(\w+_kernel)\(", text):
            at = text.index("{", m.end())
            depth, end = 1, at + 1
            while depth:
                depth += {"{": 1, "}": -1}.get(text[end], 0)
                end += 1
            found[m.group(1)] = text[at:end]
    return found


@pytest.mark.parametrize("d,G,norm,block", [(128, 2, True, True), (64, 1, True, True), (128, 1, False, True),
                                            (128, 1, False, False), (64, 1, True, False)])
def test_every_reader_of_the_backward_is_ordered_behind_its_writer(d, G, norm, block):
    from paper_2602_03681_b200 import binding
    B, H, L = 1, 2, 256
    t = {n: torch.randn((B, L, H, d), device="cuda").bfloat16() for n in ("q", "k", "v", "dout", "dq", "dk", "dv")}
    t.update({n: torch.zeros((B, L, H), device="cuda") for n in ("g", "beta", "dg", "dbeta")})
    w, dw = torch.full((B, L, H, 2), 0.5, device="cuda"), torch.empty((B, L, H, 2), device="cuda")
    route = torch.zeros((B, L, H), dtype=torch.uint8, device="cuda")
    route[:, :64] = 1
    p = binding.make_params(B, H, L, d, binding.NATSL_BF16, d ** -0.5, 1.0, w=w, G=G, norm_eps=1e-6,
                            flags=(binding.BLOCK_ROUTING if block else 0) | (binding.QK_NORM if norm else 0))
    if block:
        dscore = torch.empty((B, L // 64, H, 2), device="cuda")
        p.dscore = dscore.data_ptr()
    ws = binding.alloc_workspace(p, binding.OP_BWD)

    def step():
        binding.natsl_hybrid_bwd(t["q"], t["k"], t["v"], t["g"], t["beta"], route, t["dout"], t["dq"], t["dk"], t["dv"],
                                 t["dg"], t["dbeta"], dw, p, ws)

    step()                                     # (first use: streams, events, kernels)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph):
        step()
    names, reach, _ = kernels_and_paths(graph)
    pairs = ALWAYS + (NORMED if norm else []) + (BLOCK if block else TOKEN_NORMED if norm else TOKEN)
    for a, b in pairs:
        at, to = ([n for n, name in names.items() if x in name] for x in (a, b))
        assert at and to, (a, b, sorted(names.values()))
        for x in at:
            for y in to:
                assert y in reach[x], f"{names[y]} is not ordered behind {names[x]}"


@pytest.mark.parametrize("dtype,B,H,L,d", [("bf16", 1, 2, 128, 128), ("bf16", 1, 2, 2048, 64), ("bf16", 4, 16, 1024, 64),
                                           ("f32", 1, 2, 128, 64)])
def test_a_programmatic_dependent_waits_for_its_predecessor(dtype, B, H, L, d):
    """A forward and two decode steps: a kernel that may start before its predecessor has ended must wait for it before
    it ends itself.  Otherwise whoever waits for that kernel -- the first decode step reads the forward's final state --
    does not wait for the one ahead of it."""
    from paper_2602_03681_b200 import binding
    dt, code = (torch.bfloat16, binding.NATSL_BF16) if dtype == "bf16" else (torch.float32, binding.NATSL_F32)
    t = {n: torch.randn((B, L, H, d), device="cuda").to(dt) for n in ("q", "k", "v", "out")}
    g, beta = torch.zeros((B, L, H), device="cuda"), torch.zeros((B, L, H), device="cuda")
    route = torch.zeros((B, L, H), dtype=torch.uint8, device="cuda")
    route[:, ::7] = 1
    kc, vc = (torch.zeros((B, H, L + 2, d), dtype=dt, device="cuda") for _ in range(2))
    n, state = torch.zeros((B, H), dtype=torch.int32, device="cuda"), torch.zeros((B, H, d, d), device="cuda")
    p = binding.make_params(B, H, L, d, code, d ** -0.5, 1.0, state_out=state, k_sm=kc, v_sm=vc, sm_len=n, sm_cap=L + 2)
    pd = binding.make_params(B, H, 0, d, code, d ** -0.5, 1.0)
    ws, wd = binding.alloc_workspace(p, binding.OP_FWD), binding.alloc_workspace(pd, binding.OP_DECODE)

    def step():
        binding.natsl_hybrid_fwd(t["q"], t["k"], t["v"], g, beta, route, t["out"], p, ws)
        for i in range(2):
            binding.natsl_decode_step(t["q"][:, i].contiguous(), t["k"][:, i].contiguous(), t["v"][:, i].contiguous(),
                                      g[:, i].contiguous(), beta[:, i].contiguous(), route[:, i].contiguous(), state, kc,
                                      vc, n, t["out"][:, i].contiguous(), pd, wd)

    step()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph):
        step()
    names, _, early = kernels_and_paths(graph)
    sources = kernel_sources()
    seen = set()
    for x in early:
        own = [k for k in sources if f"{len(k)}{k}" in names[x]]
        assert len(own) == 1, names[x]
        assert "grid_dependency_wait()" in sources[own[0]], f"{own[0]} does not wait for the kernel before it"
        seen.add(own[0])
    assert seen >= ({"softmax_combine_tc_kernel", "route_gather_kernel"} if dtype == "bf16" else {"softmax_combine_simt_kernel"})


@pytest.mark.parametrize("d,G,norm,block", [(128, 2, True, True), (128, 1, False, False), (64, 1, False, False)])
def test_a_training_step_starts_behind_the_one_before(d, G, norm, block):
    """Two training steps in one graph.  The second one's first kernel is a programmatic dependent of what the first one ends
    with, where two streams have been joined: every kernel of the first step lies ahead of it, and the graph gives the bits
    of the same steps launched one by one."""
    from paper_2602_03681_b200 import binding
    B, H, L = 1, 2, 512
    gen = torch.Generator(device="cuda").manual_seed(3)

    def rand(*s):
        return torch.randn(s, generator=gen, device="cuda")

    t = {n: (torch.nn.functional.normalize(rand(B, L, H, d), dim=-1) if n in "qk" else rand(B, L, H, d)).bfloat16()
         for n in ("q", "k", "v", "dout")}
    g, beta = -torch.nn.functional.softplus(rand(B, L, H)), torch.sigmoid(rand(B, L, H))
    w = torch.softmax(rand(B, L, H, 2), -1).contiguous()
    route = (torch.rand((B, L // 64 if block else L, H), generator=gen, device="cuda") < 0.3).to(torch.uint8)
    if block:
        route = route.repeat_interleave(64, dim=1).contiguous()
    dscore = torch.zeros((B, L // 64, H, 2), device="cuda")
    # out and the gradients of each step; the second works on other values
    results = [[torch.zeros_like(x) for x in (t["q"], t["q"], t["k"], t["v"], g, beta, w)] for _ in range(2)]
    values = [t["v"], t["v"].flip(1).contiguous()]
    flags = (binding.BLOCK_ROUTING if block else 0) | (binding.QK_NORM if norm else 0)
    pf, pb = (binding.make_params(B, H, L, d, binding.NATSL_BF16, d ** -0.5, 1.0, w=w, G=G, norm_eps=1e-6, flags=flags | f)
              for f in (binding.SAVE_FOR_BWD, binding.SAVED_FWD))
    if block:
        pf.dscore = pb.dscore = dscore.data_ptr()
    ws = binding.alloc_workspace(pf, binding.OP_BWD)

    def step(i):
        out, *grads = results[i]
        binding.natsl_hybrid_fwd(t["q"], t["k"], values[i], g, beta, route, out, pf, ws)
        binding.natsl_hybrid_bwd(t["q"], t["k"], values[i], g, beta, route, t["dout"], *grads, pb, ws)

    for i in range(2):
        step(i)
        torch.cuda.synchronize()
        assert binding.natsl_device_status(ws) == 0
    expected = [[x.clone() for x in r] for r in results]
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph):
        step(0)
        step(1)
    names, reach, early = kernels_and_paths(graph)
    first, second = sorted((n for n, name in names.items() if "gdn_prepare" in name), key=lambda n: -len(reach[n]))
    assert second in early
    ahead = [n for n in names if second in reach[n]]
    assert len(ahead) == len(names) // 2 and first in ahead
    assert all(n == second or n in reach[second] for n in names if n not in ahead)
    sources = kernel_sources()
    for x in early:
        own = [k for k in sources if f"{len(k)}{k}" in names[x]]
        assert len(own) == 1 and "grid_dependency_wait()" in sources[own[0]], names[x]
    for r in results:
        for x in r:
            x.zero_()
    graph.instantiate()
    graph.replay()
    torch.cuda.synchronize()
    assert binding.natsl_device_status(ws) == 0
    for got, want in zip(results, expected):
        for x, y in zip(got, want):
            assert torch.equal(x, y)
