"""Which kernels of a captured backward are ordered behind which: the edges of the graph, not the outcome of one run.
(A missing edge between the two streams gives the right bits whenever the reader happens to start late enough.)"""
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
    """{node: kernel name} and {node: every node ordered behind it} of a captured graph."""
    from cuda.bindings import driver as cu

    def ok(res):
        assert res[0] == cu.CUresult.CUDA_SUCCESS, res[0]
        return res[1] if len(res) == 2 else res[1:]

    g = cu.CUgraph(graph.raw_cuda_graph())
    nodes = ok(cu.cuGraphGetNodes(g, ok(cu.cuGraphGetNodes(g, 0))[1]))[0]
    m = ok(cu.cuGraphGetEdges_v2(g, 0))[-1]
    src, dst = ok(cu.cuGraphGetEdges_v2(g, m))[:2]
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
    return names, reach


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
    names, reach = kernels_and_paths(graph)
    pairs = ALWAYS + (NORMED if norm else []) + (BLOCK if block else TOKEN_NORMED if norm else TOKEN)
    for a, b in pairs:
        at, to = ([n for n, name in names.items() if x in name] for x in (a, b))
        assert at and to, (a, b, sorted(names.values()))
        for x in at:
            for y in to:
                assert y in reach[x], f"{names[y]} is not ordered behind {names[x]}"
