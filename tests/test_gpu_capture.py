"""The walk and the packed step inside a CUDA graph, on every route they take: all segments in one launch per step, the
forward so and the backward segment by segment on library streams, everything segment by segment; replayed on other inputs
in the same buffers, against the same calls made eagerly."""
import numpy as np
import pytest
import torch

from paper_2607_15105_b200 import binding
from paper_2607_15105_b200.workloads import HgaConfig

pytestmark = pytest.mark.gpu
NAMES = ("cs", "gs", "ci", "gi", "ng", "O", "LSE", "dQ", "dK", "dV")
ROUTES = {"one_launch": (dict(), 0), "d64": (dict(head_dim=64), 0),
          "forward_only_in_one_launch": (dict(chunk=128, group=16, q_block=128, topk_chunks=32, topk_groups=8, sink=128, local=128), 0),
          "bf16_gradients": (dict(), binding.HGA_FLAG_BWD_BF16_GRADS), "cuda_cores": (dict(), binding.HGA_FLAG_GENERIC_KERNELS)}


def z(*s, dt=torch.bfloat16):
    return torch.zeros(*s, dtype=dt, device="cuda")


@pytest.mark.parametrize("kind", ["walk", "packed"])
@pytest.mark.parametrize("route", list(ROUTES))
def test_replay_equals_eager(route, kind):
    kw, flags = ROUTES[route]
    base = dict(name="capture", batch=1, n_q_heads=4, n_kv_heads=2, head_dim=128, total_len=1536, seg_len=384, chunk=64, group=8,
                q_block=64, topk_chunks=4, topk_groups=3, sink=64, local=64, topics=0, needles=0, backward=True, seed=5)
    base.update(kw)
    cfg = HgaConfig(**base)
    L, S, Hq, Hkv, d, bq = cfg.total_len, cfg.seg_len, cfg.n_q_heads, cfg.n_kv_heads, cfg.head_dim, cfg.q_block
    n_seg, items = L // S, Hkv * (L // bq)
    gdt = torch.bfloat16 if flags & binding.HGA_FLAG_BWD_BF16_GRADS else torch.float32
    p = binding.make_params(cfg, flags=flags)
    q_shape, k_shape = ((1, Hq, L, d), (1, Hkv, L, d)) if kind == "walk" else ((L, Hq, d), (L, Hkv, d))
    data = {k: z(*(q_shape if k in ("Q", "dO") else k_shape)) for k in ("Q", "K", "V", "dO")}
    i32 = lambda *s: torch.full(s, -7, dtype=torch.int32, device="cuda")
    out = dict(cs=z(Hkv, L // cfg.chunk, d), gs=z(Hkv, L // cfg.group, d), ci=i32(items, cfg.topk_chunks), gi=i32(items, cfg.topk_chunks * cfg.kg_eff),
               ng=i32(items), O=z(*q_shape), LSE=z(Hq * L, dt=torch.float32), dQ=z(*q_shape), dK=z(Hkv * L * d, dt=gdt), dV=z(Hkv * L * d, dt=gdt))
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    cu = np.array([0, S, 2 * S, L], np.int32)            # packed: three sequences without history
    if kind == "walk":
        ws = torch.empty(sum(binding.hga_workspace_bytes(p)) + 512, dtype=torch.uint8, device="cuda")
    else:
        ws = torch.empty(binding.hga_varlen_workspace_bytes(p, cu, cu), dtype=torch.uint8, device="cuda")

    def call():
        args = [data[k] for k in ("Q", "K", "V", "dO")] + [out[k] for k in NAMES] + [ws, status]
        if kind == "walk":
            binding.hga_tbptt_walk(p, *args)
        else:
            binding.hga_varlen_step(p, cu, cu, *args)

    def fill(seed):
        gen = torch.Generator(device="cuda").manual_seed(seed)
        for t in data.values():
            t.copy_(torch.randn(t.shape, generator=gen, device="cuda"))

    fill(1)
    call()                                                # (streams, attributes and tensor maps are set up outside the capture)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        call()
    fill(2)
    for t in out.values():
        t.zero_()
    graph.replay()
    torch.cuda.synchronize()
    got = {k: v.clone() for k, v in out.items()}
    for t in out.values():
        t.zero_()
    call()
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    for k in NAMES:
        if k in ("dK", "dV"):                             # fp32 adds in another order (and one rounding to bf16)
            assert float((got[k].double() - out[k].double()).norm()) <= (1e-5 if gdt == torch.float32 else 2.0 ** -8) * float(out[k].double().norm()), k
        else:
            assert torch.equal(got[k], out[k]), k
