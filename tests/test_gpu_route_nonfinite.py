"""Routing of scores that are not finite (a diverged step's queries or keys): a mean or a log-sum-exp over the rows can be
NaN, which no comparison of floats orders.  The lists must still be lists: as many groups per opened chunk as the budget says,
ascending, inside the opened chunks, and nothing written behind an item's list or the whole output."""
import numpy as np
import pytest
import torch

from paper_2607_15105_b200 import binding
from paper_2607_15105_b200.workloads import HgaConfig, make_inputs

from hga_testlib import to_dev

pytestmark = pytest.mark.gpu

VARIANTS = {"max": 0, "mean": binding.HGA_FLAG_SCORE_MEAN, "lse": binding.HGA_FLAG_SCORE_LSE}
CASES = {"per8": dict(), "per16": dict(chunk=128, group=8, q_block=128, topk_groups=5), "many_slots": dict(topk_chunks=24, topk_groups=8),
         "d64": dict(head_dim=64)}


@pytest.mark.parametrize("generic", [0, binding.HGA_FLAG_GENERIC_KERNELS])
@pytest.mark.parametrize("budget", [0, binding.HGA_FLAG_GLOBAL_GROUP_BUDGET])
@pytest.mark.parametrize("variant", list(VARIANTS))
@pytest.mark.parametrize("name", list(CASES))
@pytest.mark.parametrize("where", ["query", "one_group", "all_groups", "infinite_key"])
def test_lists_stay_lists(where, name, variant, budget, generic):
    base = dict(name="nonfinite", batch=1, n_q_heads=4, n_kv_heads=2, head_dim=128, total_len=4096, seg_len=512, chunk=64, group=8,
                q_block=64, topk_chunks=6, topk_groups=3, sink=0, local=128, topics=16, needles=0, backward=False, seed=3)
    base.update(CASES[name])
    cfg = HgaConfig(**base)
    x = make_inputs(cfg)
    buf = binding.HgaLayerBuffers(cfg, backward=False, want_scores=True, flags=VARIANTS[variant] | budget | generic)
    Q, K = to_dev(x["Q"]), to_dev(x["K"])
    buf.build_summaries(K, 0, cfg.total_len)
    nan = float("nan")
    if where == "query":
        Q[0, 1, 70, 5] = nan                              # one row: the mean of every score of its block
    elif where == "one_group":
        buf.group_sum[0, 0, 5::8, 3] = nan
    elif where == "all_groups":
        buf.group_sum[0, 1, :, 3] = nan
        buf.chunk_sum[0, 1, ::3, 3] = nan
    else:
        buf.group_sum[0, :, 2::4, 7] = float("inf")
        buf.chunk_sum[0, :, 1::2, 7] = float("inf")
    kc, kge, per = cfg.topk_chunks, cfg.kg_eff, cfg.chunk // cfg.group
    # the outputs inside larger buffers, so that what is written behind them shows
    n = cfg.n_items
    guard_c = torch.full((n * kc + 4096,), -77, dtype=torch.int32, device="cuda")
    guard_g = torch.full((n * kc * kge + 4096,), -77, dtype=torch.int32, device="cuda")
    buf.chunk_idx = guard_c[:n * kc].view(1, cfg.n_kv_heads, cfg.n_q_blocks, kc)
    buf.group_idx = guard_g[:n * kc * kge].view(1, cfg.n_kv_heads, cfg.n_q_blocks, kc * kge)
    buf.route(Q)
    torch.cuda.synchronize()
    assert bool((guard_c[n * kc:] == -77).all()) and bool((guard_g[n * kc * kge:] == -77).all())
    ci, gi, ng = (t.cpu().numpy() for t in (buf.chunk_idx, buf.group_idx, buf.n_groups))
    for h in range(cfg.n_kv_heads):
        for qb in range(cfg.n_q_blocks):
            p0 = cfg.history + qb * cfg.q_block
            cand = (p0 - cfg.local) // cfg.chunk
            c = ci[0, h, qb]
            sel = c[c >= 0]
            assert len(sel) == min(kc, cand) and np.all(np.diff(sel) > 0) and sel[-1] < cand, (h, qb, c)
            g = gi[0, h, qb]
            assert ng[0, h, qb] == len(sel) * kge
            real = g[:ng[0, h, qb]]
            assert np.all(np.diff(real) > 0) and np.all(g[ng[0, h, qb]:] == -1), (h, qb, g)
            assert np.all(np.isin(real // per, sel)), (h, qb, g, sel)
            if not budget:
                assert np.all(np.bincount(np.searchsorted(sel, real // per), minlength=len(sel)) == kge)
