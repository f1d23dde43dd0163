"""The forward's compaction + gather kernel at the edges of its slices: chunk counts around one slice per CTA, one chunk
per CTA and the largest slice, with and without entries already in the cache, against numpy."""
import numpy as np
import pytest
import torch

from paper_2602_03681_b200 import inputs
from test_gpu_parity import dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,H,chunks,before", [(1, 1, 1, 0), (1, 2, 33, 0), (1, 1, 512, 0), (3, 5, 31, 70),
                                               (16, 40, 3, 0), (1, 16, 65, 129), (2, 300, 33, 0)])
def test_cache_and_lengths_are_exact(B, H, chunks, before):
    from paper_2602_03681_b200 import binding
    wl = inputs.WORKLOADS["cfg4_bf16_train"]
    L, d = 64 * chunks, wl.d
    rng = np.random.default_rng(chunks)
    route = (rng.random((B, L, H)) < 0.3).astype(np.uint8)
    gen = torch.Generator(device="cuda").manual_seed(chunks)
    q, k, v = (torch.randn((B, L, H, d), generator=gen, device="cuda").bfloat16() for _ in range(3))
    k = torch.nn.functional.normalize(k.float(), dim=-1).bfloat16()
    g = -torch.rand((B, L, H), generator=gen, device="cuda")
    beta = torch.rand((B, L, H), generator=gen, device="cuda")
    cap = before + L
    ks, vs = (torch.zeros((B, H, cap, d), dtype=torch.bfloat16, device="cuda") for _ in range(2))
    n = torch.full((B, H), before, dtype=torch.int32, device="cuda")
    if before:
        ks[:, :, :before] = torch.randn((B, H, before, d), generator=gen, device="cuda")
        vs[:, :, :before] = torch.randn((B, H, before, d), generator=gen, device="cuda")
    k0, v0 = ks.clone(), vs.clone()
    res = binding.hybrid_fwd(q, k, v, g, beta, dev(route), scale_la=wl.scale_la, scale_sm=wl.scale_sm,
                             cache=(ks, vs, n), flags=binding.APPEND_CACHE if before else 0)
    assert binding.natsl_device_status(res["ws"]) == 0
    assert torch.isfinite(res["out"].float()).all()
    for b in range(0, B, max(1, B - 1)):
        for h in range(0, H, max(1, H // 7)):
            at = dev(np.nonzero(route[b, :, h])[0])
            m = before + len(at)
            assert int(n[b, h]) == m
            assert torch.equal(ks[b, h, :m], torch.cat([k0[b, h, :before], k[b, at, h]]))
            assert torch.equal(vs[b, h, :m], torch.cat([v0[b, h, :before], v[b, at, h]]))
            assert torch.equal(ks[b, h, m:], k0[b, h, m:])
