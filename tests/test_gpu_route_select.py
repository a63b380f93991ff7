"""The router's chunk selection where it changes method: rank counting for few candidates, bit-by-bit search for many;
ties that straddle the k-th place on both sides of that line (lowest index wins); and query-row counts that need more
accumulators than a CTA has (several passes over a summary tile)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2607_15105_b200 import binding
from paper_2607_15105_b200.workloads import HgaConfig, make_inputs

from hga_testlib import check_routing, to_dev

pytestmark = pytest.mark.gpu


def cfg_of(**kw):
    base = dict(name="select", batch=1, n_q_heads=1, n_kv_heads=1, head_dim=64, total_len=0, seg_len=64, chunk=64, group=8,
                q_block=64, topk_chunks=7, topk_groups=3, sink=0, local=0, topics=32, needles=0, backward=False, seed=91)
    base.update(kw)
    return HgaConfig(**base)


def routed(cfg, x, cs, gs, flags=0):
    buf = binding.HgaLayerBuffers(cfg, backward=False, flags=flags)
    buf.chunk_sum.copy_(to_dev(cs))
    buf.group_sum.copy_(to_dev(gs))
    before = binding.hga_kernel_launch_counts()
    buf.route(to_dev(x["Q"]))
    torch.cuda.synchronize()
    ran = [b - a for a, b in zip(before, binding.hga_kernel_launch_counts())]
    assert ran[binding.HGA_KERNELS_ROUTE_TENSOR] == 1
    return buf.chunk_idx.cpu().numpy(), buf.group_idx.cpu().numpy(), buf.n_groups.cpu().numpy()


@pytest.mark.parametrize("ties", [False, True])
@pytest.mark.parametrize("n_cand", [1, 127, 129, 639, 640, 641, 1300])
def test_candidate_counts(n_cand, ties):
    cfg = cfg_of(total_len=(n_cand + 1) * 64)
    x = make_inputs(cfg)
    cs, gs = oracle.build_summaries(cfg, x["K"])
    if ties:
        # blocks of identical chunk summaries: whole runs of equal scores, so that some tie straddles the k-th place
        cs = cs.copy()
        for j in range(0, n_cand, 5):
            cs[0, 0, j:j + 5] = cs[0, 0, j]
    ref = oracle.route(cfg, x["Q"], cs, gs, want_scores=True)
    ci, gi, ng = routed(cfg, x, cs, gs)
    if ties:      # equal bits give equal scores on both sides, so even tied selections agree exactly
        assert np.array_equal(ci, ref["chunk_idx"])
    check_routing(cfg, ref, ci, gi, ng)


@pytest.mark.parametrize("n_cand,k", [(255, 7), (256, 64), (257, 7), (257, 64), (512, 32), (513, 40), (2048, 16), (2049, 33), (257, 65), (300, 200)])
def test_selection_by_shares(n_cand, k):
    """A thread per candidate up to 256, each warp's share first beyond (2, 8 or any number of keys per lane), one warp where
    more than 64 chunks are opened; ties inside a share and across shares."""
    cfg = cfg_of(total_len=(n_cand + 1) * 64, topk_chunks=k)
    x = make_inputs(cfg)
    cs, gs = oracle.build_summaries(cfg, x["K"])
    cs = cs.copy()
    for j in range(0, n_cand, 9):
        cs[0, 0, j:j + 9] = cs[0, 0, j % 63]
    ref = oracle.route(cfg, x["Q"], cs, gs, want_scores=True)
    ci, gi, ng = routed(cfg, x, cs, gs)
    assert np.array_equal(ci, ref["chunk_idx"])
    check_routing(cfg, ref, ci, gi, ng)


@pytest.mark.parametrize("agg", [0, binding.HGA_FLAG_SCORE_MEAN, binding.HGA_FLAG_SCORE_LSE])
@pytest.mark.parametrize("rows", ["384", "512", "1024"])
def test_row_counts(rows, agg):
    kw = {"384": dict(n_q_heads=3, q_block=128, seg_len=256, head_dim=128),                # 3 parts, a whole SM
          "512": dict(n_q_heads=4, q_block=128, seg_len=128, head_dim=128),                # 4 parts, four accumulators
          "1024": dict(n_q_heads=8, q_block=128, seg_len=128, head_dim=64)}[rows]          # 8 parts: two passes
    cfg = cfg_of(total_len=4096, topk_chunks=20, **kw)
    x = make_inputs(cfg)
    cs, gs = oracle.build_summaries(cfg, x["K"])
    name = {0: "max", binding.HGA_FLAG_SCORE_MEAN: "mean", binding.HGA_FLAG_SCORE_LSE: "lse"}[agg]
    ref = oracle.route(cfg, x["Q"], cs, gs, want_scores=True, score_agg=name)
    ci, gi, ng = routed(cfg, x, cs, gs, agg)
    check_routing(cfg, ref, ci, gi, ng)
