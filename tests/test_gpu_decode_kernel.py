"""The forward of the smallest generation shapes beyond single blocks and clean lists: several query blocks per call (the last
octet of a block's window then holds real keys of the next block, which masking alone hides), K and V as views of larger
caches with a batch, lists with entries to be skipped; and which kernel the dispatch takes on both sides of its limits."""
import json
import os
import subprocess
import sys

import numpy as np
import pytest
import torch

import oracle
from paper_2607_15105_b200 import binding
from paper_2607_15105_b200.workloads import make_inputs

from hga_testlib import TOL_LSE, TOL_O, bf16_to_f64, to_dev
from test_gpu_decode_split import CASES, cfg_of

pytestmark = pytest.mark.gpu

BLOCKS = {"3_blocks_of_3": cfg_of(1500, 3, total_len=1509, seg_len=9), "3_blocks_of_5_d64": cfg_of(1333, 5, total_len=1348, seg_len=15, head_dim=64, n_q_heads=6),
          "5_blocks_of_1": cfg_of(1499, 1, total_len=1504, seg_len=5, batch=2), "3_blocks_of_11_rows": cfg_of(700, 11, total_len=733, seg_len=33, n_q_heads=2)}


def routed(cfg, x):
    cs, gs = oracle.build_summaries(cfg, x["K"])
    ref = oracle.route(cfg, x["Q"], cs, gs)
    return ref["group_idx"], ref["n_groups"]


def forward(cfg, Q, K, V, gi, ng, p=None):
    O = torch.zeros(tuple(Q.shape), dtype=torch.bfloat16, device="cuda")
    L = torch.zeros(tuple(Q.shape[:3]), device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    binding.hga_attn_fwd(p or binding.make_params(cfg), Q, K, V, torch.from_numpy(gi).cuda(), torch.from_numpy(ng).cuda(), O, L, status)
    torch.cuda.synchronize()
    return bf16_to_f64(O), L.cpu().numpy().astype(np.float64), int(status.item())


@pytest.mark.parametrize("name", list(BLOCKS))
def test_several_blocks(name):
    cfg = BLOCKS[name]
    x = make_inputs(cfg)
    gi, ng = routed(cfg, x)
    O, LSE = oracle.attn_fwd(cfg, x["Q"], x["K"], x["V"], gi, ng)
    got, lse, status = forward(cfg, to_dev(x["Q"]), to_dev(x["K"]), to_dev(x["V"]), gi, ng)
    assert status == 0 and np.max(np.abs(got - O)) <= TOL_O and np.max(np.abs(lse - LSE)) <= TOL_LSE


@pytest.mark.parametrize("name", ["3_blocks_of_3", "5_blocks_of_1"])
def test_views_of_larger_caches(name):
    """Token-major caches with room behind the sequence, which holds non-finite values that must not be read."""
    cfg = BLOCKS[name].scaled(batch=3)
    x = make_inputs(cfg)
    gi, ng = routed(cfg, x)
    O, LSE = oracle.attn_fwd(cfg, x["Q"], x["K"], x["V"], gi, ng)
    views = []
    for t, fill in ((to_dev(x["K"]), float("nan")), (to_dev(x["V"]), float("inf"))):
        cache = torch.full((3, cfg.total_len + 40, cfg.n_kv_heads + 1, cfg.head_dim), fill, dtype=torch.bfloat16, device="cuda")
        view = cache.transpose(1, 2)[:, :cfg.n_kv_heads, :cfg.total_len]
        view.copy_(t)
        views.append(view)
    K, V = views
    got, lse, status = forward(cfg, to_dev(x["Q"]), K, V, gi, ng, binding.params_for(cfg, K=K, V=V))
    assert status == 0 and np.max(np.abs(got - O)) <= TOL_O and np.max(np.abs(lse - LSE)) <= TOL_LSE


@pytest.mark.parametrize("name", ["8_rows", "16_rows", "3_blocks_of_3"])
def test_entries_to_be_skipped(name):
    """Out of range, inside the local window, not ascending: reported, and the rest of the list is used."""
    cfg = {**CASES, **BLOCKS}[name]
    x = make_inputs(cfg)
    gi, ng = routed(cfg, x)
    bad, good, good_ng = gi.copy(), gi.copy(), ng.copy()
    for item in np.ndindex(*ng.shape):
        n = int(ng[item])
        assert n >= 6
        bad[item][1] = 10 ** 6                                # ascending, but behind the window
        bad[item][2:] = gi[item][2:]                          # ... so these still ascend from entry 0
        bad[item][4] = bad[item][3]                           # repeated
        keep = [g for i, g in enumerate(gi[item][:n]) if i not in (1, 4)]
        good[item] = -1
        good[item][:len(keep)] = keep
        good_ng[item] = len(keep)
    O, LSE = oracle.attn_fwd(cfg, x["Q"], x["K"], x["V"], good, good_ng)
    got, lse, status = forward(cfg, to_dev(x["Q"]), to_dev(x["K"]), to_dev(x["V"]), bad, ng)
    assert status == binding.HGA_STATUS_BAD_INDEX
    assert np.max(np.abs(got - O)) <= TOL_O and np.max(np.abs(lse - LSE)) <= TOL_LSE


# (in a process of its own: the profiler stays attached to the one it has run in)
SCRIPT = """
import json, sys
import torch
from torch.profiler import ProfilerActivity, profile
from paper_2607_15105_b200 import binding
from paper_2607_15105_b200.workloads import HgaConfig
names = {}
for name, kw in json.loads(sys.stdin.read()).items():
    cfg = HgaConfig(**kw)
    buf = binding.HgaLayerBuffers(cfg, backward=False)
    z = lambda heads, n: torch.zeros(cfg.batch, heads, n, cfg.head_dim, dtype=torch.bfloat16, device="cuda")
    Q, K = z(cfg.n_q_heads, cfg.seg_len), z(cfg.n_kv_heads, cfg.total_len)
    torch.cuda.synchronize()
    with profile(activities=[ProfilerActivity.CUDA]) as p:
        buf.attn_fwd(Q, K, K)
        torch.cuda.synchronize()
    names[name] = [e.name for e in p.events() if "hga::" in e.name]
print(json.dumps(names))
"""


def test_which_kernel_runs():
    cases = {**CASES, **BLOCKS}
    text = json.dumps({n: {f: getattr(c, f) for f in c.__dataclass_fields__} for n, c in cases.items()})
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    run = subprocess.run([sys.executable, "-c", SCRIPT], input=text, capture_output=True, text=True, timeout=300, cwd=root)
    assert run.returncode == 0, run.stderr[-2000:]
    ran = json.loads(run.stdout.strip().splitlines()[-1])
    for name, c in cases.items():
        rows, items = c.gqa * c.q_block, c.n_items
        want = "k_attn_decode" if rows <= 16 and items <= 148 else "k_attn_fwd_sm100"
        assert len(ran[name]) == 1 and want in ran[name][0], (name, rows, items, ran[name])
