"""The persistent backward sweep (head_dim 128, whole 128-row M-tiles) where a unit's octets change how its pairs are made up:
none, some or nearly all of them in the active segment, in numbers around multiples of eight, lists of every length and
lists with entries to skip, against the oracle on the same lists."""
import numpy as np
import pytest
import torch

import oracle
from paper_2607_15105_b200 import binding
from paper_2607_15105_b200.workloads import HgaConfig, make_inputs

from hga_testlib import bf16_to_f64, check_grads, to_dev

pytestmark = pytest.mark.gpu


def cfg_of(**kw):
    base = dict(name="sweep", batch=2, n_q_heads=4, n_kv_heads=2, head_dim=128, total_len=1536, seg_len=1024, chunk=64, group=8,
                q_block=64, topk_chunks=8, topk_groups=4, sink=64, local=64, topics=0, needles=0, backward=True, seed=71)
    base.update(kw)
    return HgaConfig(**base)


CASES = {
    "history": (cfg_of(), "any"), "no_history": (cfg_of(total_len=1024), "any"), "most_recent": (cfg_of(), "recent"),
    "groups_of_16": (cfg_of(chunk=128, group=16, q_block=128, sink=128, local=128), "any"),
    "four_tiles": (cfg_of(n_q_heads=8, n_kv_heads=1, batch=1), "any"), "three_tiles_of_192": (cfg_of(q_block=192, seg_len=768, n_q_heads=4), "any"),
    "no_window": (cfg_of(sink=0, local=0), "recent"), "with_entries_to_skip": (cfg_of(), "invalid"),
    "one_unit": (cfg_of(batch=1, n_q_heads=2, n_kv_heads=1, seg_len=64), "any"),
}


@pytest.mark.parametrize("name", list(CASES))
def test_sweep_on_lists_of_every_length(name):
    cfg, kind = CASES[name]
    rng = np.random.default_rng(7)
    x = make_inputs(cfg)
    B, Hkv, nqb, width = cfg.batch, cfg.n_kv_heads, cfg.n_q_blocks, cfg.topk_chunks * cfg.kg_eff
    gi = np.full((B, Hkv, nqb, width), -1, dtype=np.int32)
    ng = np.zeros((B, Hkv, nqb), dtype=np.int32)
    gi_ref, ng_ref = gi.copy(), ng.copy()       # without the entries to skip
    for item in range(B * Hkv * nqb):
        b, h, qb = item // (Hkv * nqb), item // nqb % Hkv, item % nqb
        ls, se = oracle.window(cfg, qb)
        pool = np.arange(-(-se // cfg.group), ls // cfg.group)
        n = min(len(pool), item % (width + 1))
        pick = pool[-n:] if kind == "recent" and n else np.sort(rng.choice(pool, n, replace=False)) if n else pool[:0]
        pick = pick.astype(np.int32)
        valid = pick
        if kind == "invalid" and n > 2:
            valid = np.delete(pick, n // 2)
            pick[n // 2] = pick[n // 2 - 1] if item % 2 else 10 ** 6      # repeated, or past the window
        gi[b, h, qb, :n], ng[b, h, qb] = pick, n
        gi_ref[b, h, qb, :len(valid)], ng_ref[b, h, qb] = valid, len(valid)
    O, LSE = oracle.attn_fwd(cfg, x["Q"], x["K"], x["V"], gi_ref, ng_ref)
    ref = oracle.attn_bwd(cfg, x["Q"], x["K"], x["V"], x["dO"], gi_ref, ng_ref)
    buf = binding.HgaLayerBuffers(cfg)
    dev = {k: to_dev(x[k]) for k in ("Q", "K", "V", "dO")}
    gid, ngd = torch.from_numpy(gi).cuda(), torch.from_numpy(ng).cuda()
    buf.attn_fwd(dev["Q"], dev["K"], dev["V"], gid, ngd)
    torch.cuda.synchronize()
    buf.status.zero_()                          # (the forward reports entries to skip)
    before = binding.hga_kernel_launch_counts()
    buf.attn_bwd(dev["Q"], dev["K"], dev["V"], dev["dO"], gid, ngd)
    torch.cuda.synchronize()
    ran = [b - a for a, b in zip(before, binding.hga_kernel_launch_counts())]
    assert ran[binding.HGA_KERNELS_BWD_TENSOR] == 2 and int(buf.status.item()) == 0
    got = (bf16_to_f64(buf.dQ), buf.dK.cpu().numpy().astype(np.float64), buf.dV.cpu().numpy().astype(np.float64))
    check_grads(got, ref, name)
