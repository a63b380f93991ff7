"""Several segments per launch (hga_varlen_step, hga_tbptt_walk) against the four calls made segment by segment, which other
tests hold against the oracle: more segments than one launch's table takes, segments shorter than a key tile, very
unequal lengths, a batch of sequences in the walk, head_dim 64 and partly filled M-tiles; and how many launches it takes."""
import numpy as np
import pytest
import torch

from paper_2607_15105_b200 import binding
from paper_2607_15105_b200.workloads import HgaConfig

pytestmark = pytest.mark.gpu


def cfg_of(L, S, **kw):
    base = dict(name="segments", batch=1, n_q_heads=4, n_kv_heads=2, head_dim=128, total_len=L, seg_len=S, chunk=64, group=8,
                q_block=64, topk_chunks=4, topk_groups=3, sink=64, local=64, topics=0, needles=0, backward=True, seed=5)
    base.update(kw)
    return HgaConfig(**base)


def draw(gen, *shape):
    return torch.randn(*shape, generator=gen, device="cuda").to(torch.bfloat16)


def same(a, b, what):
    """Routing lists, O, LSE and dQ are bit-equal; dK / dV up to the order of their fp32 adds."""
    if what in ("dK", "dV"):
        assert float((a - b).norm()) <= 1e-5 * float(b.norm()), what
    else:
        assert torch.equal(a, b), what


HEADS = {"d128": {}, "d64_rows64": dict(head_dim=64, n_q_heads=2), "d128_rows192": dict(n_q_heads=3, n_kv_heads=1)}


@pytest.mark.parametrize("heads", list(HEADS))
@pytest.mark.parametrize("n_seq", [1, 5, 64, 65, 130])
def test_varlen_equals_the_four_calls(n_seq, heads):
    gen = torch.Generator(device="cuda").manual_seed(n_seq)
    rng = np.random.default_rng(n_seq)
    seqs = []
    for i in range(n_seq):
        S = 64 * int(rng.choice([1, 1, 2, 3, 5]))
        seqs.append((S + 64 * int(rng.choice([0, 0, 1, 7, 20])), S))
    seqs[0] = (4096, 64)
    c0 = cfg_of(64, 64, **HEADS[heads])
    cu_q = np.cumsum([0] + [s for _, s in seqs]).astype(np.int32)
    cu_k = np.cumsum([0] + [l for l, _ in seqs]).astype(np.int32)
    Hq, Hkv, d, kc, kge, nq, nk = c0.n_q_heads, c0.n_kv_heads, c0.head_dim, c0.topk_chunks, c0.kg_eff, int(cu_q[-1]), int(cu_k[-1])
    Q, dO, K, V = draw(gen, nq, Hq, d), draw(gen, nq, Hq, d), draw(gen, nk, Hkv, d), draw(gen, nk, Hkv, d)
    p = binding.make_params(c0)
    items = Hkv * nq // 64

    def outputs():
        i32 = lambda *s: torch.full(s, -7, dtype=torch.int32, device="cuda")
        z = lambda *s, dt=torch.bfloat16: torch.zeros(*s, dtype=dt, device="cuda")
        return dict(cs=z(Hkv, nk // 64, d), gs=z(Hkv, nk // 8, d), ci=i32(items, kc), gi=i32(items, kc * kge), ng=i32(items),
                    O=z(nq, Hq, d), LSE=z(Hq * nq, dt=torch.float32), dQ=z(nq, Hq, d), dK=z(Hkv * nq * d, dt=torch.float32),
                    dV=z(Hkv * nq * d, dt=torch.float32))

    a, b = outputs(), outputs()
    for o in (a, b):
        for (L, S), k0 in zip(seqs, cu_k):
            if L > S:
                ph = binding.make_params(cfg_of(L, S, **HEADS[heads]), k_stride=(L * Hkv * d, d, Hkv * d), summary_len=nk)
                binding.hga_build_summaries(ph, K[k0:], 0, L - S, o["cs"][:, k0 // 64:], o["gs"][:, k0 // 8:])
    ws = torch.empty(binding.hga_varlen_workspace_bytes(p, cu_q, cu_k), dtype=torch.uint8, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    n0 = binding.hga_kernel_launch_count()
    binding.hga_varlen_step(p, cu_q, cu_k, Q, K, V, dO, *(a[k] for k in ("cs", "gs", "ci", "gi", "ng", "O", "LSE", "dQ", "dK", "dV")), ws, status)
    assert binding.hga_kernel_launch_count() - n0 == 5 * -(-n_seq // 64)
    for i, (L, S) in enumerate(seqs):
        q0, k0 = int(cu_q[i]), int(cu_k[i])
        ps = binding.make_params(cfg_of(L, S, **HEADS[heads]), q_stride=(S * Hq * d, d, Hq * d), o_stride=(S * Hq * d, d, Hq * d),
                                 k_stride=(L * Hkv * d, d, Hkv * d), v_stride=(L * Hkv * d, d, Hkv * d), summary_len=nk)
        rb, bb = binding.hga_workspace_bytes(ps)
        w1, w2 = (torch.empty(n, dtype=torch.uint8, device="cuda") for n in (rb, bb))
        it0 = Hkv * q0 // 64
        cs, gs = b["cs"][:, k0 // 64:], b["gs"][:, k0 // 8:]
        ci, gi, ng, lse, blk = b["ci"][it0:], b["gi"][it0:], b["ng"][it0:], b["LSE"][Hq * q0:], slice(Hkv * d * q0, None)
        binding.hga_build_summaries(ps, K[k0:], L - S, L, cs, gs)
        binding.hga_route(ps, Q[q0:], cs, gs, ci, gi, ng, w1)
        binding.hga_attn_fwd(ps, Q[q0:], K[k0:], V[k0:], gi, ng, b["O"][q0:], lse, status)
        binding.hga_attn_bwd(ps, Q[q0:], K[k0:], V[k0:], b["O"][q0:], lse, dO[q0:], gi, ng, b["dQ"][q0:], b["dK"][blk], b["dV"][blk], w2, status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    single_bwd_is_fp32 = c0.head_dim == 64      # (a single short sequence may take the CUDA-core backward)
    for k in a:
        if single_bwd_is_fp32 and k in ("dQ", "dK", "dV"):
            assert float((a[k].float() - b[k].float()).norm()) <= 1e-2 * float(b[k].float().norm()), k
        else:
            same(a[k], b[k], k)


@pytest.mark.parametrize("heads", list(HEADS))
@pytest.mark.parametrize("batch,S,n_seg", [(1, 64, 70), (2, 192, 3), (2, 512, 1)])
def test_walk_equals_the_four_calls(batch, S, n_seg, heads):
    L = S * n_seg
    cfg = cfg_of(L, S, batch=batch, **HEADS[heads])
    gen = torch.Generator(device="cuda").manual_seed(n_seg)
    B, Hq, Hkv, d, kc, kge, nqb = batch, cfg.n_q_heads, cfg.n_kv_heads, cfg.head_dim, cfg.topk_chunks, cfg.kg_eff, S // 64
    Q, dO, K, V = draw(gen, B, Hq, L, d), draw(gen, B, Hq, L, d), draw(gen, B, Hkv, L, d), draw(gen, B, Hkv, L, d)
    p = binding.make_params(cfg)

    def outputs():
        i32 = lambda *s: torch.full(s, -7, dtype=torch.int32, device="cuda")
        z = lambda *s, dt=torch.bfloat16: torch.zeros(*s, dtype=dt, device="cuda")
        return dict(cs=z(B, Hkv, L // 64, d), gs=z(B, Hkv, L // 8, d), ci=i32(n_seg, B, Hkv, nqb, kc), gi=i32(n_seg, B, Hkv, nqb, kc * kge),
                    ng=i32(n_seg, B, Hkv, nqb), O=z(B, Hq, L, d), LSE=z(n_seg, B, Hq, S, dt=torch.float32), dQ=z(B, Hq, L, d),
                    dK=z(n_seg, B, Hkv, S, d, dt=torch.float32), dV=z(n_seg, B, Hkv, S, d, dt=torch.float32))

    a, b = outputs(), outputs()
    ws = torch.empty(sum(binding.hga_workspace_bytes(p)) + 512, dtype=torch.uint8, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    n0 = binding.hga_kernel_launch_count()
    binding.hga_tbptt_walk(p, Q, K, V, dO, *(a[k] for k in ("cs", "gs", "ci", "gi", "ng", "O", "LSE", "dQ", "dK", "dV")), ws, status)
    assert binding.hga_kernel_launch_count() - n0 == 1 + 4 * -(-n_seg // 64)
    qs, ks = (Hq * L * d, L * d, d), (Hkv * L * d, L * d, d)
    for s in range(n_seg):
        ps = binding.make_params(cfg_of((s + 1) * S, S, batch=batch, **HEADS[heads]), q_stride=qs, o_stride=qs, k_stride=ks, v_stride=ks, summary_len=L)
        rb, bb = binding.hga_workspace_bytes(ps)
        w1, w2 = (torch.empty(n, dtype=torch.uint8, device="cuda") for n in (rb, bb))
        at = lambda t: t[:, :, s * S:]
        binding.hga_build_summaries(ps, K, s * S, (s + 1) * S, b["cs"], b["gs"])
        binding.hga_route(ps, at(Q), b["cs"], b["gs"], b["ci"][s], b["gi"][s], b["ng"][s], w1)
        binding.hga_attn_fwd(ps, at(Q), K, V, b["gi"][s], b["ng"][s], at(b["O"]), b["LSE"][s], status)
        binding.hga_attn_bwd(ps, at(Q), K, V, at(b["O"]), b["LSE"][s], at(dO), b["gi"][s], b["ng"][s], at(b["dQ"]), b["dK"][s], b["dV"][s], w2, status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    for k in a:
        if cfg.head_dim == 64 and k in ("dQ", "dK", "dV"):
            assert float((a[k].float() - b[k].float()).norm()) <= 1e-2 * float(b[k].float().norm()), k
        else:
            same(a[k], b[k], k)
