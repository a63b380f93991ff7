"""The warp-level forward of the smallest generation shapes where it can go wrong: row counts on both sides of a matrix
instruction's eight, cluster sizes from one CTA per item to eight, units that do not divide over the warps, few or no
routed keys, more than sixteen units per warp, an odd last octet; and the shapes just past its limits."""
import numpy as np
import pytest
import torch

import oracle
from paper_2607_15105_b200 import binding
from paper_2607_15105_b200.workloads import HgaConfig, make_inputs

from hga_testlib import TOL_LSE, TOL_O, bf16_to_f64, to_dev

pytestmark = pytest.mark.gpu


def cfg_of(hist, n, **kw):
    base = dict(name="split", batch=1, n_q_heads=8, n_kv_heads=2, head_dim=128, total_len=hist + n, seg_len=n, chunk=64,
                group=8, q_block=n, topk_chunks=6, topk_groups=3, sink=64, local=128, topics=16, needles=0,
                backward=False, seed=57, decode=True)
    base.update(kw)
    return HgaConfig(**base)


CASES = {
    "8_rows": cfg_of(1500, 2),
    "9_rows": cfg_of(1500, 3, n_q_heads=6),
    "16_rows": cfg_of(1500, 4),
    "17_rows": cfg_of(1499, 17, n_q_heads=2),                       # past the limit
    "one_row": cfg_of(1517, 1, n_q_heads=2),
    "d64": cfg_of(1517, 3, head_dim=64),
    "nothing_but_the_block": cfg_of(0, 5, local=0, sink=0),
    "wide_budget": cfg_of(6000, 1, topk_chunks=80, topk_groups=8),    # 330 units over at most 64 warps
    "wide_budget_one_cta": cfg_of(6000, 1, batch=2, n_q_heads=148, n_kv_heads=74, topk_chunks=40, topk_groups=8),   # 148 items, 20 units a warp
    "149_items": cfg_of(700, 1, n_q_heads=149, n_kv_heads=149, topk_chunks=2),                                      # past the limit
    "g16": cfg_of(3000, 2, chunk=128, group=16, sink=128, topk_groups=5),
}


@pytest.mark.parametrize("name", list(CASES))
def test_decode_forward(name):
    cfg = CASES[name]
    x = make_inputs(cfg)
    closed = (cfg.total_len // cfg.chunk) * cfg.chunk
    cs, gs = oracle.build_summaries(cfg, x["K"]) if closed else (None, None)
    if closed:
        ref = oracle.route(cfg, x["Q"], cs, gs)
        gi, ng = ref["group_idx"], ref["n_groups"]
    else:
        gi = np.full((cfg.batch, cfg.n_kv_heads, 1, cfg.topk_chunks * cfg.kg_eff), -1, np.int32)
        ng = np.zeros((cfg.batch, cfg.n_kv_heads, 1), np.int32)
    items = None if cfg.n_items <= 16 else [0, 1, cfg.n_items // 2, cfg.n_items - 1]
    O, LSE = oracle.attn_fwd(cfg, x["Q"], x["K"], x["V"], gi, ng, items=items)
    Od, L = torch.zeros(x["Q"].shape, dtype=torch.bfloat16, device="cuda"), torch.zeros(x["Q"].shape[:3], device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    p = binding.make_params(cfg)
    binding.hga_attn_fwd(p, to_dev(x["Q"]), to_dev(x["K"]), to_dev(x["V"]), torch.from_numpy(gi).cuda(),
                         torch.from_numpy(ng).cuda(), Od, L, status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    got, lse = bf16_to_f64(Od), L.cpu().numpy().astype(np.float64)
    for item in (range(cfg.n_items) if items is None else items):
        h, b = item % cfg.n_kv_heads, item // cfg.n_kv_heads
        sl = (b, slice(h * cfg.gqa, (h + 1) * cfg.gqa))
        assert np.max(np.abs(got[sl] - O[sl])) <= TOL_O, item
        assert np.max(np.abs(lse[sl] - LSE[sl])) <= TOL_LSE, item
