"""hga_varlen_step and hga_tbptt_walk where one launch for all segments does not take every step, against the four calls
made segment by segment: items so wide that they keep the CUDA-core backward's fp32 probabilities (the forward of all segments in one
launch per 64, the backward segment by segment, on library streams), with gradients that are
overwritten or added to; and strides that no tensor map takes (everything segment by segment, as the calls by themselves)."""
import numpy as np
import pytest
import torch

from paper_2607_15105_b200 import binding
from paper_2607_15105_b200.workloads import HgaConfig

pytestmark = pytest.mark.gpu
NAMES = ("cs", "gs", "ci", "gi", "ng", "O", "LSE", "dQ", "dK", "dV")


def cfg_of(L, S, **kw):
    # 32 chunks of 8 groups of 16 tokens: up to 4.5K routed keys
    base = dict(name="mixed", batch=1, n_q_heads=4, n_kv_heads=2, head_dim=128, total_len=L, seg_len=S, chunk=128, group=16,
                q_block=128, topk_chunks=32, topk_groups=8, sink=128, local=128, topics=0, needles=0, backward=True, seed=5)
    base.update(kw)
    return HgaConfig(**base)


def draw(gen, *shape):
    return torch.randn(*shape, generator=gen, device="cuda").to(torch.bfloat16)


def z(*s, dt=torch.bfloat16):
    return torch.zeros(*s, dtype=dt, device="cuda")


def ran(before):
    return [b - a for a, b in zip(before, binding.hga_kernel_launch_counts())]


def check(a, b):
    for k in NAMES:
        if k in ("dK", "dV"):          # up to the order of their fp32 adds
            assert float((a[k].float() - b[k].float()).norm()) <= 1e-5 * float(b[k].float().norm()), k
        else:
            assert torch.equal(a[k], b[k]), k


@pytest.mark.parametrize("accumulate", [0, binding.HGA_FLAG_BWD_ACCUMULATE])
@pytest.mark.parametrize("n_seq", [3, 66])
def test_varlen_with_items_too_wide_for_the_sweep(n_seq, accumulate):
    gen = torch.Generator(device="cuda").manual_seed(n_seq)
    seqs = [(5120 if i == 1 else 128 * (1 + i % 3), 128 * (1 + i % 2) if i % 3 else 128) for i in range(n_seq)]
    seqs = [(max(L, S), S) for L, S in seqs]
    c0 = cfg_of(128, 128)
    cu_q = np.cumsum([0] + [s for _, s in seqs]).astype(np.int32)
    cu_k = np.cumsum([0] + [l for l, _ in seqs]).astype(np.int32)
    Hq, Hkv, d, kc, kge, nq, nk, bq = c0.n_q_heads, c0.n_kv_heads, c0.head_dim, c0.topk_chunks, c0.kg_eff, int(cu_q[-1]), int(cu_k[-1]), c0.q_block
    Q, dO, K, V = draw(gen, nq, Hq, d), draw(gen, nq, Hq, d), draw(gen, nk, Hkv, d), draw(gen, nk, Hkv, d)
    p = binding.make_params(c0, flags=accumulate)
    items = Hkv * nq // bq

    def outputs():
        i32 = lambda *s: torch.full(s, -7, dtype=torch.int32, device="cuda")
        start = torch.ones(Hkv * nq * d, device="cuda") if accumulate else torch.full((Hkv * nq * d,), 7.0, device="cuda")
        return dict(cs=z(Hkv, nk // c0.chunk, d), gs=z(Hkv, nk // c0.group, d), ci=i32(items, kc), gi=i32(items, kc * kge), ng=i32(items),
                    O=z(nq, Hq, d), LSE=z(Hq * nq, dt=torch.float32), dQ=z(nq, Hq, d), dK=start.clone(), dV=start.clone())

    a, b = outputs(), outputs()
    for o in (a, b):
        for (L, S), k0 in zip(seqs, cu_k):
            if L > S:
                ph = binding.make_params(cfg_of(L, S), k_stride=(L * Hkv * d, d, Hkv * d), summary_len=nk)
                binding.hga_build_summaries(ph, K[k0:], 0, L - S, o["cs"][:, k0 // c0.chunk:], o["gs"][:, k0 // c0.group:])
    ws = torch.empty(binding.hga_varlen_workspace_bytes(p, cu_q, cu_k), dtype=torch.uint8, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    before = binding.hga_kernel_launch_counts()
    binding.hga_varlen_step(p, cu_q, cu_k, Q, K, V, dO, *(a[k] for k in NAMES), ws, status)
    n = ran(before)
    assert n[binding.HGA_KERNELS_FWD_TENSOR] == -(-n_seq // 64) and n[binding.HGA_KERNELS_BWD_TENSOR] == 0
    assert n[binding.HGA_KERNELS_BWD_GENERIC] == n_seq * (1 if accumulate else 2)
    for i, (L, S) in enumerate(seqs):
        q0, k0 = int(cu_q[i]), int(cu_k[i])
        ps = binding.make_params(cfg_of(L, S), flags=accumulate, q_stride=(S * Hq * d, d, Hq * d), o_stride=(S * Hq * d, d, Hq * d),
                                 k_stride=(L * Hkv * d, d, Hkv * d), v_stride=(L * Hkv * d, d, Hkv * d), summary_len=nk)
        w1, w2 = (torch.empty(x, dtype=torch.uint8, device="cuda") for x in binding.hga_workspace_bytes(ps))
        it0 = Hkv * q0 // bq
        cs, gs = b["cs"][:, k0 // c0.chunk:], b["gs"][:, k0 // c0.group:]
        ci, gi, ng, lse, blk = b["ci"][it0:], b["gi"][it0:], b["ng"][it0:], b["LSE"][Hq * q0:], slice(Hkv * d * q0, None)
        binding.hga_build_summaries(ps, K[k0:], L - S, L, cs, gs)
        binding.hga_route(ps, Q[q0:], cs, gs, ci, gi, ng, w1)
        binding.hga_attn_fwd(ps, Q[q0:], K[k0:], V[k0:], gi, ng, b["O"][q0:], lse, status)
        binding.hga_attn_bwd(ps, Q[q0:], K[k0:], V[k0:], b["O"][q0:], lse, dO[q0:], gi, ng, b["dQ"][q0:], b["dK"][blk], b["dV"][blk], w2, status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    check(a, b)


def walk_both(cfg, batch, n_seg, flags=0, **strides):
    """The walk (with the given strides) and the four calls (dense)."""
    S, L = cfg.seg_len, cfg.total_len
    gen = torch.Generator(device="cuda").manual_seed(n_seg)
    B, Hq, Hkv, d, kc, kge, nqb = batch, cfg.n_q_heads, cfg.n_kv_heads, cfg.head_dim, cfg.topk_chunks, cfg.kg_eff, S // cfg.q_block
    Q, dO, K, V = draw(gen, B, Hq, L, d), draw(gen, B, Hq, L, d), draw(gen, B, Hkv, L, d), draw(gen, B, Hkv, L, d)
    gdt = torch.bfloat16 if flags & binding.HGA_FLAG_BWD_BF16_GRADS else torch.float32

    def outputs():
        i32 = lambda *s: torch.full(s, -7, dtype=torch.int32, device="cuda")
        return dict(cs=z(B, Hkv, L // cfg.chunk, d), gs=z(B, Hkv, L // cfg.group, d), ci=i32(n_seg, B, Hkv, nqb, kc), gi=i32(n_seg, B, Hkv, nqb, kc * kge),
                    ng=i32(n_seg, B, Hkv, nqb), O=z(B, Hq, L, d), LSE=z(n_seg, B, Hq, S, dt=torch.float32), dQ=z(B, Hq, L, d),
                    dK=z(n_seg, B, Hkv, S, d, dt=gdt), dV=z(n_seg, B, Hkv, S, d, dt=gdt))

    a, b = outputs(), outputs()
    p = binding.make_params(cfg, flags=flags, **strides)
    ws = torch.empty(sum(binding.hga_workspace_bytes(p)) + 512, dtype=torch.uint8, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    before = binding.hga_kernel_launch_counts()
    binding.hga_tbptt_walk(p, Q, K, V, dO, *(a[k] for k in NAMES), ws, status)
    n = ran(before)
    qs, ks = (Hq * L * d, L * d, d), (Hkv * L * d, L * d, d)
    for s in range(n_seg):
        ps = binding.make_params(cfg.scaled(total_len=(s + 1) * S), flags=flags, q_stride=strides.get("q_stride", qs), o_stride=qs, k_stride=ks, v_stride=ks,
                                 summary_len=L)
        w1, w2 = (torch.empty(x, dtype=torch.uint8, device="cuda") for x in binding.hga_workspace_bytes(ps))
        at = lambda t: t[:, :, s * S:]
        binding.hga_build_summaries(ps, K, s * S, (s + 1) * S, b["cs"], b["gs"])
        binding.hga_route(ps, at(Q), b["cs"], b["gs"], b["ci"][s], b["gi"][s], b["ng"][s], w1)
        binding.hga_attn_fwd(ps, at(Q), K, V, b["gi"][s], b["ng"][s], at(b["O"]), b["LSE"][s], status)
        binding.hga_attn_bwd(ps, at(Q), K, V, at(b["O"]), b["LSE"][s], at(dO), b["gi"][s], b["ng"][s], at(b["dQ"]), b["dK"][s], b["dV"][s], w2, status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    return a, b, n


@pytest.mark.parametrize("batch,S,n_seg", [(2, 1280, 4), (1, 128, 66)])
def test_walk_with_items_too_wide_for_the_sweep(batch, S, n_seg):
    a, b, n = walk_both(cfg_of(S * n_seg, S, batch=batch), batch, n_seg)
    assert n[binding.HGA_KERNELS_FWD_TENSOR] == -(-n_seg // 64) and n[binding.HGA_KERNELS_BWD_GENERIC] == 2 * n_seg
    check(a, b)


def test_walk_with_strides_that_no_tensor_map_takes():
    """The batch axis has one entry, so its stride means nothing and may be anything; no tensor map takes 2^50."""
    cfg = cfg_of(1024, 256, chunk=64, group=8, q_block=64, topk_chunks=4, topk_groups=3, sink=64, local=64)
    L, d = cfg.total_len, cfg.head_dim
    a, b, n = walk_both(cfg, 1, 4, q_stride=(1 << 50, L * d, d))
    assert n[binding.HGA_KERNELS_FWD_TENSOR] == 0 and n[binding.HGA_KERNELS_FWD_GENERIC] == 4 and n[binding.HGA_KERNELS_ROUTE_GENERIC] > 0
    check(a, b)


def test_walk_with_bf16_gradients():
    cfg = cfg_of(1024, 256, chunk=64, group=8, q_block=64, topk_chunks=4, topk_groups=3, sink=64, local=64)
    a, b, _ = walk_both(cfg, 1, 4, flags=binding.HGA_FLAG_BWD_BF16_GRADS)
    for k in NAMES:
        if k in ("dK", "dV"):          # fp32 adds in another order, then one rounding to 8 bits: now and then the neighbour
            assert float((a[k].double() - b[k].double()).abs().max()) <= 2.0 ** -7 * float(b[k].double().abs().max()), k
        else:
            assert torch.equal(a[k], b[k]), k


@pytest.mark.parametrize("kc,tensor", [(383, True), (384, False)])
def test_the_widest_items_the_sweep_has_room_for(kc, tensor):
    """Up to 3327 routed keys per item (sink, groups, window, block and a chunk) the sweep; from there on the CUDA cores, with fp32 P and dS."""
    cfg = cfg_of(1024, 256, chunk=64, group=8, q_block=64, topk_chunks=kc, topk_groups=1, sink=64, local=64)
    gen = torch.Generator(device="cuda").manual_seed(kc)
    Q, dO = (draw(gen, 1, cfg.n_q_heads, 256, 128) for _ in range(2))
    K, V = (draw(gen, 1, cfg.n_kv_heads, 1024, 128) for _ in range(2))
    grads = []
    for flags in (0, binding.HGA_FLAG_GENERIC_KERNELS):
        buf = binding.HgaLayerBuffers(cfg, flags=flags)
        buf.build_summaries(K, 0, 1024)
        buf.route(Q)
        buf.attn_fwd(Q, K, V)
        before = binding.hga_kernel_launch_counts()
        buf.attn_bwd(Q, K, V, dO)
        n = ran(before)
        assert n[binding.HGA_KERNELS_BWD_TENSOR] == (2 if tensor and not flags else 0)
        grads.append((buf.dQ.float(), buf.dK, buf.dV))
    torch.cuda.synchronize()
    for a, b in zip(*grads):          # bf16 P and dS against fp32 ones: 2^-9 per term
        assert float((a - b).norm()) <= 1e-2 * float(b.norm())


def test_a_window_that_no_sequence_reaches_is_a_wide_item():
    """A local window near 2^31 (every key is local): its sum with the other parts of an item does not fit 32 bits."""
    cfg = cfg_of(1024, 256, chunk=64, group=8, q_block=64, topk_chunks=4, topk_groups=3, sink=64, local=2 ** 31 - 128)
    gen = torch.Generator(device="cuda").manual_seed(3)
    Q, dO = (draw(gen, 1, cfg.n_q_heads, 256, 128) for _ in range(2))
    K, V = (draw(gen, 1, cfg.n_kv_heads, 1024, 128) for _ in range(2))
    grads = []
    for c, flags in ((cfg, 0), (cfg.scaled(local=1024), binding.HGA_FLAG_GENERIC_KERNELS)):
        buf = binding.HgaLayerBuffers(c, flags=flags)
        buf.build_summaries(K, 0, 1024)
        buf.route(Q)
        buf.attn_fwd(Q, K, V)
        before = binding.hga_kernel_launch_counts()
        buf.attn_bwd(Q, K, V, dO)
        n = ran(before)
        assert n[binding.HGA_KERNELS_BWD_TENSOR] == 0 and n[binding.HGA_KERNELS_BWD_GENERIC] == 2 and int(buf.status.item()) == 0
        grads.append((buf.dQ.float(), buf.dK, buf.dV))
    for a, b in zip(*grads):          # (O, which delta is taken of, comes from two forward kernels: bf16 weights and fp32 ones)
        assert float((a - b).norm()) <= 1e-2 * float(b.norm())
