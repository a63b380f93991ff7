"""What a program that uses this library has it do, as cases that can be timed and compared.

Five kinds of work, each through the public entry points of `paper_2607_15105_b200.binding`:

  step     one layer step on resident device tensors, as a training or evaluation loop calls it: summaries of
           the active segment, routing, attention forward and, when training, backward (HgaLayerBuffers.step)
  decode   one generation step: routing and attention forward of the newest tokens of every sequence
  walk     one layer over a whole sequence, segment by segment (hga_tbptt_walk)
  varlen   one layer step over packed sequences of different lengths (hga_varlen_step)
  host     one layer step from pinned host buffers (hga_step_host)

The inputs are drawn on the GPU with the structure the method meets in use and `workloads.py` describes: chunks
share a topic, a query block follows the topics of two earlier chunks, and a few groups match one block's queries
("needles").  The resident state a program keeps from earlier segments (history K/V and its summaries) is built
in prepare().
"""
import math

import torch

from paper_2607_15105_b200 import binding
from paper_2607_15105_b200.workloads import CONFIGS, HgaConfig

# ----------------------------------------------------------------------------- cases


def _from_config(n, name, kind="step", **kw):
    """A case in the shape of one of the repository's configurations."""
    c = CONFIGS[n]
    case = dict(name=name, kind=kind, batch=c.batch, n_q=c.n_q_heads, n_kv=c.n_kv_heads, d=c.head_dim,
                total=c.total_len, seg=c.seg_len, chunk=c.chunk, group=c.group, q_block=c.q_block,
                kc=c.topk_chunks, kg=c.topk_groups, sink=c.sink, local=c.local, topics=c.topics,
                needles=c.needles, backward=c.backward, flags=0)
    case.update(kw)
    return case


# (new tokens : resident tokens) of twelve documents of a packed batch
_PACKED = "512:2048,64:64,320:1344,1024:1024,128:4096,704:704,256:2816,896:1920,448:3584,192:192,640:1280,384:2432"


def listed():
    return [
        # the smallest training step: a tiny layer with head_dim 64, four query blocks; launches and latency count
        _from_config(1, "tiny_1k"),
        # a 2K sequence trained in one segment: every key is differentiable
        _from_config(2, "train_2k"),
        # one segment of a long-context fine-tuning run: 2048 new tokens behind 14336 detached ones
        _from_config(3, "train_16k"),
        # the same with the paper's default budget (selected chunks opened whole) and bf16 gradients, as an
        # autograd node returns them
        _from_config(6, "train_16k_whole_chunks", flags=binding.HGA_FLAG_BWD_BF16_GRADS),
        # a small model with head_dim 64 and one query head per kv head (multi-head attention)
        _from_config(3, "train_mha_d64_16k", n_q=16, n_kv=16, d=64, needles=0),
        # prefill / evaluation of the last 2048 tokens of a 128K document, forward only
        _from_config(4, "eval_128k"),
        # the largest: four sequences of 64K, no topic structure, a wide budget
        _from_config(5, "train_b4_64k"),
        # one user, one new token behind an odd number of resident ones: the smallest generation step
        _from_config(7, "decode_b1", kind="decode", batch=1, total=5003, topics=64),
        # batched generation over long documents
        _from_config(7, "decode_b32", kind="decode"),
        # a whole 16K sequence trained in eight segments
        _from_config(3, "walk_16k", kind="walk", needles=0),
        # a packed batch of documents of different lengths, with and without history
        _from_config(3, "packed_12", kind="varlen", seqs=_PACKED, total=0, seg=0, topics=64, needles=0),
        # a step whose tensors live in (pinned) host memory
        _from_config(3, "host_16k", kind="host"),
    ]


def _log_int(rng, lo, hi):
    """An integer between lo and hi, spread over the logarithm."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _budget(rng, case):
    """Chunk, group, query block, budget and windows."""
    c, g = rng.choice([(64, 8), (64, 8), (64, 8), (128, 16), (128, 8)])
    case.update(chunk=c, group=g, q_block=c, kc=_log_int(rng, 4, 32), kg=rng.choice([2, 3, 4, 4, 8]),
                sink=c * rng.choice([0, 1, 1, 2]), local=c * rng.choice([0, 1, 2, 2, 4]))
    case["kg"] = min(case["kg"], c // g)


def _keys(case):
    """Routed keys of a query block with a full budget behind it."""
    return case["sink"] + case["kc"] * case["kg"] * case["group"] + case["local"] + case["q_block"]


def _score_flags(rng):
    """The routing variants, now and then."""
    return rng.choice([0] * 9 + [binding.HGA_FLAG_GLOBAL_GROUP_BUDGET, binding.HGA_FLAG_SCORE_MEAN, binding.HGA_FLAG_SCORE_LSE])


def draw(rng):
    kind = rng.choice(["step"] * 6 + ["small"] * 3 + ["decode"] * 4 + ["walk", "walk", "varlen", "varlen", "varlen", "host"])
    while True:
        case = dict(kind="step" if kind == "small" else kind, batch=1, n_q=32, n_kv=8, d=128, flags=_score_flags(rng),
                    topics=rng.choice([0, 64, 256, 1024]), needles=0, backward=rng.random() < 0.75)
        _budget(rng, case)
        bq = case["q_block"]
        if kind == "step":           # the layer shape of the repository's configurations, any length
            case["batch"] = rng.choice([1, 1, 1, 2, 4])
            case["total"] = _log_int(rng, 1024 // bq, 131072 // bq) * bq
            case["seg"] = min(case["total"], _log_int(rng, 256 // bq, 4096 // bq) * bq)
            case["needles"] = rng.choice([0, 32]) if case["topics"] else 0
            if case["backward"] and rng.random() < 0.4:
                case["flags"] |= binding.HGA_FLAG_BWD_BF16_GRADS
            # within the largest listed case, in resident tokens and in (query row, key) pairs
            if case["batch"] * case["total"] <= 4 * 65536 and case["batch"] * case["seg"] * _keys(case) <= 4 * 4096 * 2400:
                return case
        elif kind == "small":        # other head layouts: few heads, head_dim 64 or 128, every grouping
            case["d"] = rng.choice([64, 64, 128])
            case["n_kv"] = rng.choice([1, 2, 4, 8])
            case["n_q"] = case["n_kv"] * rng.choice([1, 1, 2, 2, 3, 4, 4, 5, 6, 7, 8])
            case["batch"] = rng.choice([1, 1, 2])
            case["total"] = _log_int(rng, 512 // bq, 16384 // bq) * bq
            case["seg"] = min(case["total"], _log_int(rng, 1, 1024 // bq) * bq)
            # within the listed head_dim-64 case, and query blocks of a small layer (rows * keys of one block)
            if (case["n_q"] <= 16 and case["batch"] * case["n_q"] * case["seg"] * _keys(case) * case["d"] <= 16 * 2048 * 768 * 64
                    and case["n_q"] // case["n_kv"] * bq * _keys(case) <= 64 * 1024):
                return case
        elif kind == "decode":
            n = rng.choice([1, 1, 1, 1, 2, 4, 5, 8])
            case.update(batch=_log_int(rng, 1, 64), total=_log_int(rng, 300, 65536) + n, seg=n, q_block=n, backward=False)
            if case["batch"] * case["total"] <= 4 * 65536 * 2:
                return case
        elif kind == "walk":
            s = rng.choice([512, 1024, 2048, 2048, 4096])
            case.update(seg=s, total=s * rng.randint(2, 8))
            if case["total"] * _keys(case) <= 4 * 4096 * 1600:
                return case
        elif kind == "varlen":
            n = _log_int(rng, 2, 48)
            seqs = []
            for _ in range(n):
                new = _log_int(rng, 1, 1024 // bq) * bq
                seqs.append("%d:%d" % (new, new + rng.choice([0, 1]) * _log_int(rng, 1, 4096 // bq) * bq))
            case.update(seqs=",".join(seqs), total=0, seg=0)
            if sum(s for s, _ in _seqs(case)) * _keys(case) <= 4 * 4096 * 1600:
                return case
        else:
            case.update(total=_log_int(rng, 2048 // bq, 16384 // bq) * bq, backward=True)
            case["seg"] = min(case["total"], _log_int(rng, 512 // bq, 2048 // bq) * bq)
            return case


# ----------------------------------------------------------------------------- inputs


def _seqs(case):
    """[(new tokens, resident tokens)] of a packed batch."""
    return [tuple(int(x) for x in s.split(":")) for s in case["seqs"].split(",")]


def _config(case, total=None, seg=None):
    return HgaConfig(case["kind"], case["batch"], case["n_q"], case["n_kv"], case["d"],
                     case["total"] if total is None else total, case["seg"] if seg is None else seg,
                     case["chunk"], case["group"], case["q_block"], case["kc"], case["kg"], case["sink"],
                     case["local"], topics=case["topics"], needles=case["needles"], backward=case["backward"],
                     seed=0, decode=case["kind"] == "decode")


def _inputs(cfg, gen, with_dO):
    """Q, K, V (and dO) of one layer step on the GPU, structured as workloads.make_inputs describes."""
    B, Hq, Hkv, d, L, S = cfg.batch, cfg.n_q_heads, cfg.n_kv_heads, cfg.head_dim, cfg.total_len, cfg.seg_len
    G, c, H, nqb = cfg.gqa, cfg.chunk, cfg.history, cfg.n_q_blocks

    def normal(*shape):
        return torch.randn(*shape, generator=gen, device="cuda")

    def uniform(*shape):
        return torch.rand(*shape, generator=gen, device="cuda")

    K = torch.empty(B, Hkv, L, d, dtype=torch.bfloat16, device="cuda")
    Q = torch.empty(B, Hq, S, d, dtype=torch.bfloat16, device="cuda")
    for b in range(B):
        k = normal(Hkv, L, d)
        q = normal(Hkv, G, nqb, cfg.q_block, d)
        if cfg.topics:
            nch = -(-L // c)
            U = torch.nn.functional.normalize(normal(Hkv, cfg.topics, d), dim=-1)
            tau = (uniform(Hkv, nch) * cfg.topics).long()                          # topic of every chunk
            topic = torch.gather(U, 1, tau[..., None].expand(-1, -1, d))           # [Hkv, nch, d]
            k += 1.5 * topic.repeat_interleave(c, 1)[:, :L]
            prev = ((H + torch.arange(nqb, device="cuda") * cfg.q_block) // c).clamp(min=1)
            pick = (uniform(2, Hkv, nqb) * prev).long()                            # two earlier chunks per block
            for a in pick:
                q += 3.0 * torch.gather(topic, 1, a[..., None].expand(-1, -1, d))[:, None, :, None, :]
        for n in range(cfg.needles):
            h, qb = n % Hkv, n % nqb
            lo, hi = cfg.sink // cfg.group, (H + qb * cfg.q_block - cfg.local - c) // cfg.group
            if hi > lo:
                m = lo + (n * 7919 + 13) % (hi - lo)
                w = 8.0 * torch.nn.functional.normalize(normal(d), dim=0)
                k[h, m * cfg.group:(m + 1) * cfg.group] = normal(cfg.group, d) + w
                q[h, :, qb] += w
        K[b] = k
        Q[b] = q.reshape(Hq, S, d)
    V = torch.empty_like(K)
    for b in range(B):
        V[b] = normal(Hkv, L, d)
    dO = normal(B, Hq, S, d).to(torch.bfloat16) if with_dO else None
    return Q, K, V, dO


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    return {"step": _prepare_step, "decode": _prepare_step, "host": _prepare_host, "walk": _prepare_walk,
            "varlen": _prepare_varlen}[case["kind"]](case, gen)


def _prepare_step(case, gen):
    cfg = _config(case)
    Q, K, V, dO = _inputs(cfg, gen, case["backward"])
    buf = binding.HgaLayerBuffers(cfg, backward=case["backward"], flags=case["flags"])
    done = (cfg.total_len // cfg.chunk) * cfg.chunk if cfg.decode else cfg.history
    buf.build_summaries(K, 0, done)                 # summaries of everything that is already resident
    return {"kind": case["kind"], "buf": buf, "Q": Q, "K": K, "V": V, "dO": dO}


def _prepare_host(case, gen):
    cfg = _config(case)
    Q, K, V, dO = _inputs(cfg, gen, True)
    buf = binding.HgaLayerBuffers(cfg, flags=case["flags"])
    buf.build_summaries(K, 0, cfg.history)
    H = cfg.history
    pin = lambda t: t.cpu().pin_memory()
    host = dict(Q=pin(Q), Kseg=pin(K[:, :, H:].contiguous()), Vseg=pin(V[:, :, H:].contiguous()), dO=pin(dO))
    out = dict(O=torch.empty_like(host["Q"]).pin_memory(), dQ=torch.empty_like(host["Q"]).pin_memory(),
               dK=torch.empty(cfg.batch, cfg.n_kv_heads, cfg.seg_len, cfg.head_dim).pin_memory(),
               dV=torch.empty(cfg.batch, cfg.n_kv_heads, cfg.seg_len, cfg.head_dim).pin_memory())
    arena = torch.empty(binding.hga_step_arena_bytes(buf.p), dtype=torch.uint8, device="cuda")
    return {"kind": "host", "buf": buf, "K": K, "V": V, "host": host, "out": out, "arena": arena}


def _lists(cfg, *lead):
    """Routing outputs: chunk_idx, group_idx, n_groups with the given leading sizes."""
    kc, w = cfg.topk_chunks, cfg.topk_chunks * cfg.kg_eff
    mk = lambda *s: torch.full(s, -1, dtype=torch.int32, device="cuda")
    return mk(*lead, kc), mk(*lead, w), mk(*lead)


def _prepare_walk(case, gen):
    cfg = _config(case)
    L, S, B, Hq, Hkv, d = cfg.total_len, cfg.seg_len, cfg.batch, cfg.n_q_heads, cfg.n_kv_heads, cfg.head_dim
    Q, K, V, dO = _inputs(cfg.scaled(seg_len=L), gen, case["backward"])     # every token of the sequence is a query
    ci, gi, ng = _lists(cfg, L // S, B, Hkv, S // cfg.q_block)
    p = binding.make_params(cfg, flags=case["flags"])
    zeros = lambda *s, dt=torch.bfloat16: torch.zeros(*s, dtype=dt, device="cuda")
    st = dict(kind="walk", p=p, Q=Q, K=K, V=V, dO=dO, cs=zeros(B, Hkv, L // cfg.chunk, d), gs=zeros(B, Hkv, L // cfg.group, d),
              ci=ci, gi=gi, ng=ng, O=torch.zeros_like(Q), LSE=zeros(L // S, B, Hq, S, dt=torch.float32),
              ws=torch.empty(sum(binding.hga_workspace_bytes(p)) + 512, dtype=torch.uint8, device="cuda"),
              status=torch.zeros(1, dtype=torch.int32, device="cuda"), dQ=None, dK=None, dV=None)
    if case["backward"]:
        st.update(dQ=torch.zeros_like(Q), dK=zeros(L // S, B, Hkv, S, d, dt=torch.float32),
                  dV=zeros(L // S, B, Hkv, S, d, dt=torch.float32))
    return st


def _prepare_varlen(case, gen):
    seqs = _seqs(case)
    cu_q, cu_k = [0], [0]
    parts = []
    for new, resident in seqs:
        parts.append(_inputs(_config(case, resident, new), gen, case["backward"]))
        cu_q.append(cu_q[-1] + new)
        cu_k.append(cu_k[-1] + resident)
    pack = lambda i: torch.cat([p[i][0].transpose(0, 1) for p in parts]).contiguous()      # token-major
    Q, K, V = pack(0), pack(1), pack(2)
    dO = pack(3) if case["backward"] else None
    del parts
    cfg = _config(case, cu_k[-1], cu_q[-1])
    Hq, Hkv, d, n_q, n_k = cfg.n_q_heads, cfg.n_kv_heads, cfg.head_dim, cu_q[-1], cu_k[-1]
    ci, gi, ng = _lists(cfg, Hkv * n_q // cfg.q_block)
    p = binding.make_params(cfg, flags=case["flags"])
    zeros = lambda *s, dt=torch.bfloat16: torch.zeros(*s, dtype=dt, device="cuda")
    cs, gs = zeros(Hkv, n_k // cfg.chunk, d), zeros(Hkv, n_k // cfg.group, d)
    for (new, resident), k0 in zip(seqs, cu_k):     # summaries of the resident history of every sequence
        if resident > new:
            ph = binding.make_params(_config(case, resident, new), k_stride=(resident * Hkv * d, d, Hkv * d), summary_len=n_k)
            binding.hga_build_summaries(ph, K[k0:], 0, resident - new, cs[:, k0 // cfg.chunk:], gs[:, k0 // cfg.group:])
    st = dict(kind="varlen", p=p, cu_q=cu_q, cu_k=cu_k, Q=Q, K=K, V=V, dO=dO, cs=cs, gs=gs, ci=ci, gi=gi, ng=ng,
              O=zeros(n_q, Hq, d), LSE=zeros(Hq * n_q, dt=torch.float32), dQ=None, dK=None, dV=None,
              ws=torch.empty(binding.hga_varlen_workspace_bytes(p, cu_q, cu_k) + 256, dtype=torch.uint8, device="cuda"),
              status=torch.zeros(1, dtype=torch.int32, device="cuda"))
    if case["backward"]:
        st.update(dQ=zeros(n_q, Hq, d), dK=zeros(Hkv * n_q * d, dt=torch.float32), dV=zeros(Hkv * n_q * d, dt=torch.float32))
    return st


# ----------------------------------------------------------------------------- one pass


def run(st):
    kind = st["kind"]
    if kind == "step":
        b = st["buf"]
        b.step(st["Q"], st["K"], st["V"], st["dO"])
        out = {"O": b.O, "LSE": b.LSE, "chunk_idx": b.chunk_idx, "group_idx": b.group_idx, "n_groups": b.n_groups,
               "chunk_sum": b.chunk_sum, "group_sum": b.group_sum}
        if b.backward:
            out.update(dQ=b.dQ, dK=b.dK, dV=b.dV)
        return out
    if kind == "decode":
        b = st["buf"]
        b.route(st["Q"])
        b.attn_fwd(st["Q"], st["K"], st["V"])
        return {"O": b.O, "LSE": b.LSE, "chunk_idx": b.chunk_idx, "group_idx": b.group_idx, "n_groups": b.n_groups}
    if kind == "host":
        b, h, o = st["buf"], st["host"], st["out"]
        binding.hga_step_host(b.p, h["Q"], h["Kseg"], h["Vseg"], h["dO"], st["K"], st["V"], b.chunk_sum, b.group_sum,
                              o["O"], o["dQ"], o["dK"], o["dV"], st["arena"], b.status)
        return dict(o, chunk_sum=b.chunk_sum, group_sum=b.group_sum)
    args = [st[k] for k in ("Q", "K", "V", "dO", "cs", "gs", "ci", "gi", "ng", "O", "LSE", "dQ", "dK", "dV", "ws", "status")]
    if kind == "walk":
        binding.hga_tbptt_walk(st["p"], *args)
    else:
        binding.hga_varlen_step(st["p"], st["cu_q"], st["cu_k"], *args)
    return {k: st[k] for k in ("O", "LSE", "ci", "gi", "ng", "cs", "gs", "dQ", "dK", "dV")}


# ----------------------------------------------------------------------------- work and tolerance


def _problem_work(case, total, seg, summaries=True):
    """Bytes and operations of one (batch, layer) step, history = total - seg."""
    B, Hq, Hkv, d, c, g, bq = (case[k] for k in ("batch", "n_q", "n_kv", "d", "chunk", "group", "q_block"))
    decode, bwd = case["kind"] == "decode", case["backward"]
    H, G, per = total - seg, Hq // Hkv, c // g
    kge = min(case["kg"], per)
    route_flops = pairs = active = 0.0
    touched = sums = 0.0             # K/V rows and summary rows that some block reads, at most every one once
    for qb in range(seg // bq):
        p0 = H + qb * bq
        ls = max(0, ((p0 - case["local"]) // c) * c)
        se = min(case["sink"], ls)
        cand = (ls - se) // c
        sel = min(case["kc"], cand)
        far = se + sel * kge * g
        local = G * (bq * (p0 - ls) + bq * (bq + 1) / 2.0)
        pairs += local + G * bq * far
        routed_active = sel * kge * g * (max(0, ls - max(H, se)) / max(1.0, ls - se))       # in expectation
        active += G * (bq * (p0 - max(ls, H)) + bq * (bq + 1) / 2.0 + bq * (routed_active + max(0, se - H)))
        route_flops += 2.0 * d * G * bq * (cand + sel * per)
        touched += far + p0 + bq - ls
        sums += cand + sel * per
    touched, sums = min(touched, total), min(sums, total // c + total // g)
    n = B * Hkv
    flops = n * (route_flops + 4.0 * d * pairs + ((6.0 * pairs + 4.0 * active) * d if bwd else 0.0))
    rows, kv = B * Hq * seg, n * seg
    nbytes = n * (2.0 * touched + sums) * d * 2 + rows * d * 2 * 2 + rows * 4
    nbytes += n * (seg // bq) * (case["kc"] * (1 + kge) + 1) * 4
    if summaries and not decode:
        nbytes += kv * d * 2 * (1.0 / c + 1.0 / g)          # summaries of the active segment, written
    if bwd:
        grad = 2 if case["flags"] & binding.HGA_FLAG_BWD_BF16_GRADS else 4
        nbytes += rows * d * 2 * 2 + 2.0 * kv * d * grad    # dO read, dQ, dK, dV written
    return nbytes, flops


def work(case):
    if case["kind"] == "varlen":
        parts = [_problem_work(case, resident, new) for new, resident in _seqs(case)]
    elif case["kind"] == "walk":
        s = case["seg"]
        parts = [_problem_work(case, (i + 1) * s, s) for i in range(case["total"] // s)]
        # a later segment reads history rows that earlier segments have brought in already
        B, Hkv, d = case["batch"], case["n_kv"], case["d"]
        again = sum(_problem_work(case, (i + 1) * s, s)[0] - _problem_work(case, s, s)[0] for i in range(case["total"] // s))
        parts.append((-max(0.0, again), 0.0))
    else:
        parts = [_problem_work(case, case["total"], case["seg"])]
    return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}


def tolerance(case):
    # O and the gradients go through bf16 probabilities: against the 64-bit oracle O and dQ are off by up to 3.8e-3
    # (relative 2-norm), dK and dV by 2.3e-3.  Routing is exact up to near ties (scores closer than the fp32
    # accumulation error): a tie that falls the other way changes single list entries.  A dominant element of O
    # or of a gradient row may be off by a few bf16 steps of the values it is summed from.
    return {"rel": 1e-2, "max": 0.5, "differ": 5e-3}
