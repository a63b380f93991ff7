"""The persistent backward sweep (head_dim 128, whole 128-row M-tiles) where a unit's octets change how its pairs are made up:
none, some or nearly all of them in the active segment, in numbers around multiples of eight, lists of every length and
lists with entries to skip, against the oracle on the same lists: with few units, one to a CTA, and with several times as many as
the device has SMs, where a CTA takes over units of another make-up."""
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


def many(**kw):
    return cfg_of(**{**dict(batch=1, n_q_heads=16, n_kv_heads=8, total_len=4096, seg_len=3840, topk_chunks=8, topk_groups=4, sink=0, local=0), **kw})


MANY = {
    # windows of nothing but the block itself: units whose pairs all get dK/dV, among others none of whose do
    "short_history": (many(), False), "entries_to_skip": (many(), True), "windows": (many(sink=64, local=128), False),
    "groups_of_16": (many(n_q_heads=8, total_len=7424, seg_len=7168, chunk=128, group=16, q_block=128), False),
    "four_tiles": (many(n_q_heads=32, n_kv_heads=4, total_len=2176, seg_len=1920), False),
}


@pytest.mark.parametrize("name", list(MANY))
def test_units_of_every_make_up_follow_one_another(name):
    cfg, skip = MANY[name]
    B, Hkv, nqb, width, g = cfg.batch, cfg.n_kv_heads, cfg.n_q_blocks, cfg.topk_chunks * cfg.kg_eff, cfg.group
    assert B * Hkv * nqb * (cfg.gqa * cfg.q_block // 128) >= 3 * torch.cuda.get_device_properties(0).multi_processor_count
    rng = np.random.default_rng(11)
    x = make_inputs(cfg)
    gi = np.full((B, Hkv, nqb, width), -1, dtype=np.int32)
    ng = np.zeros((B, Hkv, nqb), dtype=np.int32)
    gi_ref, ng_ref = gi.copy(), ng.copy()
    for item in range(Hkv * nqb):
        h, qb = item // nqb, item % nqb
        ls, se = oracle.window(cfg, qb)
        pool = np.arange(-(-se // g), ls // g)
        hist, act = pool[pool * g < cfg.history], pool[pool * g >= cfg.history]
        # eight octets of the active segment to a pair with dK/dV: numbers around that, with and without history before them
        n_act = min(len(act), int(rng.choice([0, 0, 0, 1, 7, 8, 9, 15, 16, 17, 31, 32]) * 8 // g), width)
        n_hist = min(len(hist), int(rng.choice([0, 0, 5, 16])), width - n_act)
        pick = np.concatenate([np.sort(rng.choice(hist, n_hist, replace=False)), np.sort(rng.choice(act, n_act, replace=False))]).astype(np.int32)
        valid, n = pick, len(pick)
        if skip and n > 2 and item % 3 == 0:
            valid = np.delete(pick, n // 2)
            pick[n // 2] = pick[n // 2 - 1]
        gi[0, h, qb, :n], ng[0, h, qb] = pick, n
        gi_ref[0, h, qb, :len(valid)], ng_ref[0, h, qb] = valid, len(valid)
    O, LSE = oracle.attn_fwd(cfg, x["Q"], x["K"], x["V"], gi_ref, ng_ref)
    ref = oracle.attn_bwd(cfg, x["Q"], x["K"], x["V"], x["dO"], gi_ref, ng_ref)
    buf = binding.HgaLayerBuffers(cfg)
    dev = {k: to_dev(x[k]) for k in ("Q", "K", "V", "dO")}
    gid, ngd = torch.from_numpy(gi).cuda(), torch.from_numpy(ng).cuda()
    buf.attn_fwd(dev["Q"], dev["K"], dev["V"], gid, ngd)
    torch.cuda.synchronize()
    buf.status.zero_()
    for rep in range(3):
        for t in (buf.dQ, buf.dK, buf.dV):
            t.fill_(7.0)
        before = binding.hga_kernel_launch_counts()
        buf.attn_bwd(dev["Q"], dev["K"], dev["V"], dev["dO"], gid, ngd)
        torch.cuda.synchronize()
        ran = [b - a for a, b in zip(before, binding.hga_kernel_launch_counts())]
        assert ran[binding.HGA_KERNELS_BWD_TENSOR] == 2 and int(buf.status.item()) == 0
        got = (bf16_to_f64(buf.dQ), buf.dK.cpu().numpy().astype(np.float64), buf.dV.cpu().numpy().astype(np.float64))
        check_grads(got, ref, (name, rep))


def test_units_of_packed_documents_follow_one_another():
    """Documents without history, long before short: units all of whose pairs get dK/dV (a long one's late blocks) are followed in
    the same CTA by units without any (the next one's first blocks)."""
    lens = [1024, 192, 704, 1024, 704, 192, 320, 1024]
    cfgs = [cfg_of(batch=1, n_q_heads=16, n_kv_heads=8, total_len=n, seg_len=n, topk_chunks=16, local=128, seed=80 + i) for i, n in enumerate(lens)]
    c0, total = cfgs[0], sum(lens)
    Hq, Hkv, d, bq, kc, width = c0.n_q_heads, c0.n_kv_heads, c0.head_dim, c0.q_block, c0.topk_chunks, c0.topk_chunks * c0.kg_eff
    assert total // bq * Hkv >= 3 * torch.cuda.get_device_properties(0).multi_processor_count
    xs = [make_inputs(c) for c in cfgs]
    cu = np.cumsum([0] + lens).astype(np.int32)
    Q, K, V, dO = (to_dev(np.ascontiguousarray(np.concatenate([x[k][0].transpose(1, 0, 2) for x in xs]))) for k in ("Q", "K", "V", "dO"))
    z = lambda *s, dt=torch.bfloat16: torch.zeros(*s, dtype=dt, device="cuda")
    items = Hkv * total // bq
    cs, gs, O, dQ, LSE = z(Hkv, total // c0.chunk, d), z(Hkv, total // c0.group, d), z(total, Hq, d), z(total, Hq, d), z(Hq * total, dt=torch.float32)
    ci, gi, ng, status = (z(*s, dt=torch.int32) for s in ((items, kc), (items, width), (items,), (1,)))
    dK, dV = z(Hkv * total * d, dt=torch.float32), z(Hkv * total * d, dt=torch.float32)
    p = binding.make_params(c0)
    ws = torch.empty(binding.hga_varlen_workspace_bytes(p, cu, cu), dtype=torch.uint8, device="cuda")
    for rep in range(5):
        before = binding.hga_kernel_launch_counts()
        binding.hga_varlen_step(p, cu, cu, Q, K, V, dO, cs, gs, ci, gi, ng, O, LSE, dQ, dK, dV, ws, status)
        torch.cuda.synchronize()
        ran = [b - a for a, b in zip(before, binding.hga_kernel_launch_counts())]
        assert ran[binding.HGA_KERNELS_BWD_TENSOR] == 2 and int(status.item()) == 0
        first = rep == 0
        if first:
            refs = []
        for i, (c, x) in enumerate(zip(cfgs, xs)):
            q0, q1, n = int(cu[i]), int(cu[i + 1]), lens[i]
            it = slice(Hkv * q0 // bq, Hkv * q1 // bq)
            if first:
                shape = (1, Hkv, n // bq)
                refs.append(oracle.attn_bwd(c, x["Q"], x["K"], x["V"], x["dO"], gi[it].cpu().numpy().reshape(*shape, width), ng[it].cpu().numpy().reshape(shape)))
            blk = slice(Hkv * d * q0, Hkv * d * q1)
            got = (bf16_to_f64(dQ[q0:q1]).transpose(1, 0, 2)[None], *(t[blk].double().cpu().numpy().reshape(1, Hkv, n, d) for t in (dK, dV)))
            check_grads(got, refs[i], (rep, i))
