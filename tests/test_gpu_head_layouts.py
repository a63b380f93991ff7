"""Head layouts whose query rows do not fill the 128-row tiles (odd groupings, one query head per kv head) and
head_dim 64, through the tensor-core kernels, against the oracle: padded M-tiles in router, forward and sweep, odd
numbers of half-steps in the band kernel, row counts that the router splits into parts, local windows that end inside
a key tile, and an invalid index list in the head_dim-64 sweep."""
import numpy as np
import pytest
import torch

import oracle
from paper_2607_15105_b200 import binding
from paper_2607_15105_b200.workloads import HgaConfig, make_inputs

from hga_testlib import TOL_LSE, TOL_O, bf16_to_f64, check_grads, check_routing, to_dev

pytestmark = pytest.mark.gpu


def cfg_of(**kw):
    base = dict(name="heads", batch=1, n_q_heads=2, n_kv_heads=2, head_dim=64, total_len=1536, seg_len=512, chunk=64,
                group=8, q_block=64, topk_chunks=5, topk_groups=3, sink=64, local=128, topics=16, needles=0,
                backward=True, seed=71)
    base.update(kw)
    return HgaConfig(**base)


CASES = {
    "d64_rows64": cfg_of(),
    "d64_rows192": cfg_of(n_q_heads=6, seg_len=256),
    "d64_rows320_no_history": cfg_of(n_q_heads=5, n_kv_heads=1, total_len=576, seg_len=576, topk_chunks=3),
    "d64_c128_bq128": cfg_of(n_q_heads=4, chunk=128, group=16, q_block=128, sink=128, local=256, total_len=2048, topk_groups=4),
    "d64_window_inside_a_tile": cfg_of(chunk=32, local=96, sink=32, total_len=1024, seg_len=320, topk_chunks=6, topk_groups=2),
    "d64_one_block": cfg_of(n_q_heads=16, n_kv_heads=8, total_len=704, seg_len=64),
    "d128_rows64": cfg_of(head_dim=128),
    "d128_rows64_one_block": cfg_of(head_dim=128, n_q_heads=1, n_kv_heads=1, total_len=640, seg_len=64),
    "d128_rows192": cfg_of(head_dim=128, n_q_heads=3, n_kv_heads=1, seg_len=320),
    "d128_rows448": cfg_of(head_dim=128, n_q_heads=7, n_kv_heads=1, seg_len=192),
}


@pytest.mark.parametrize("name", list(CASES))
def test_layout_matches_oracle(name):
    cfg = CASES[name]
    x = make_inputs(cfg)
    Q, K, V, dO = (to_dev(x[n]) for n in ("Q", "K", "V", "dO"))
    buf = binding.HgaLayerBuffers(cfg)
    buf.build_summaries(K, 0, cfg.history)
    before = binding.hga_kernel_launch_counts()
    buf.step(Q, K, V, dO)
    torch.cuda.synchronize()
    ran = [b - a for a, b in zip(before, binding.hga_kernel_launch_counts())]
    assert int(buf.status.item()) == 0
    # (chunks of 32 tokens have four groups: those are routed by the CUDA-core router)
    assert ran[binding.HGA_KERNELS_ROUTE_TENSOR] == (1 if cfg.chunk // cfg.group in (8, 16) else 0), ran
    assert ran[binding.HGA_KERNELS_FWD_TENSOR] == 1 and ran[binding.HGA_KERNELS_FWD_GENERIC] == 0, ran
    assert ran[binding.HGA_KERNELS_BWD_TENSOR] == 2 and ran[binding.HGA_KERNELS_BWD_GENERIC] == 0, ran
    cs, gs = oracle.build_summaries(cfg, x["K"])
    ref = oracle.route(cfg, x["Q"], cs, gs, want_scores=True)
    gi, ng = buf.group_idx.cpu().numpy(), buf.n_groups.cpu().numpy()
    n, ec, eg = check_routing(cfg, ref, buf.chunk_idx.cpu().numpy(), gi, ng)
    assert ec <= max(1, n // 10) and eg <= max(1, n // 5), (n, ec, eg)
    O, LSE = oracle.attn_fwd(cfg, x["Q"], x["K"], x["V"], gi, ng)
    assert np.max(np.abs(bf16_to_f64(buf.O) - O)) <= TOL_O
    assert np.max(np.abs(buf.LSE.cpu().numpy().astype(np.float64) - LSE)) <= TOL_LSE
    check_grads((bf16_to_f64(buf.dQ), buf.dK.double().cpu().numpy(), buf.dV.double().cpu().numpy()),
                oracle.attn_bwd(cfg, x["Q"], x["K"], x["V"], x["dO"], gi, ng), name)


def test_invalid_entries_are_skipped_at_head_dim_64():
    """Entries out of range, out of order and inside the local window, in the middle of a list: forward and backward must
    behave as if they were not there."""
    cfg = CASES["d64_rows64"]
    x = make_inputs(cfg)
    Q, K, V, dO = (to_dev(x[n]) for n in ("Q", "K", "V", "dO"))
    ref = oracle.route(cfg, x["Q"], *oracle.build_summaries(cfg, x["K"]))
    gi, ng = ref["group_idx"].copy(), ref["n_groups"]
    clean_gi, clean_ng = gi.copy(), ng.copy()
    for h, qb, at, bad in ((0, 7, 4, 10 ** 6), (1, 5, 0, -3), (0, 3, 9, 0), (1, 7, 6, (cfg.history + 7 * 64) // cfg.group)):
        keep = [int(m) for i, m in enumerate(gi[0, h, qb, :ng[0, h, qb]]) if i != at]
        gi[0, h, qb, at] = bad
        clean_gi[0, h, qb] = -1
        clean_gi[0, h, qb, :len(keep)] = keep
        clean_ng[0, h, qb] = len(keep)
    buf = binding.HgaLayerBuffers(cfg)
    gid, ngd = torch.from_numpy(gi).cuda(), torch.from_numpy(ng).cuda()
    buf.attn_fwd(Q, K, V, gid, ngd)
    buf.attn_bwd(Q, K, V, dO, gid, ngd)
    torch.cuda.synchronize()
    assert int(buf.status.item()) == binding.HGA_STATUS_BAD_INDEX
    O, _ = oracle.attn_fwd(cfg, x["Q"], x["K"], x["V"], clean_gi, clean_ng)
    assert np.max(np.abs(bf16_to_f64(buf.O) - O)) <= TOL_O
    check_grads((bf16_to_f64(buf.dQ), buf.dK.double().cpu().numpy(), buf.dV.double().cpu().numpy()),
                oracle.attn_bwd(cfg, x["Q"], x["K"], x["V"], x["dO"], clean_gi, clean_ng), "invalid entries")
