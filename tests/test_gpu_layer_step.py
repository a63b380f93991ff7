"""hga_layer_step (HgaLayerBuffers.step) against its four calls made one by one: the same lists and outputs, on every kernel family,
and the status codes of the four; with inputs that the kernel ahead of it in the stream is still writing when it lets its
successor start, and with buffers that are input and output at once (these also for hga_tbptt_walk and hga_varlen_step)."""
import pytest
import torch

from paper_2607_15105_b200 import binding
from paper_2607_15105_b200.workloads import HgaConfig, make_inputs

import oracle
from hga_testlib import bf16_to_f64, check_grads, to_dev

pytestmark = pytest.mark.gpu


def cfg_of(**kw):
    base = dict(name="step", batch=1, n_q_heads=8, n_kv_heads=2, head_dim=128, total_len=4096, seg_len=1024, chunk=64, group=8,
                q_block=64, topk_chunks=8, topk_groups=4, sink=64, local=128, topics=16, needles=0, backward=True, seed=91)
    base.update(kw)
    return HgaConfig(**base)


CASES = {"d128": (cfg_of(), 0), "no_history": (cfg_of(total_len=1024), 0), "d64_rows64": (cfg_of(head_dim=64, n_q_heads=2), 0),
         "bf16_grads": (cfg_of(), binding.HGA_FLAG_BWD_BF16_GRADS), "cuda_cores": (cfg_of(seg_len=256), binding.HGA_FLAG_GENERIC_KERNELS),
         "small_d64": (cfg_of(head_dim=64, n_q_heads=2, n_kv_heads=1, total_len=1024, seg_len=256, topk_chunks=4, local=64), 0),
         "forward": (cfg_of(), "forward")}


@pytest.mark.parametrize("name", list(CASES))
def test_step_is_its_four_calls(name):
    cfg, flags = CASES[name]
    bwd = flags != "forward"
    flags = flags if bwd else 0
    x = {k: to_dev(v) for k, v in make_inputs(cfg).items() if k in ("Q", "K", "V", "dO")}
    one, four = (binding.HgaLayerBuffers(cfg, backward=bwd, flags=flags) for _ in range(2))
    for buf in (one, four):
        buf.build_summaries(x["K"], 0, cfg.history)
    four.build_summaries(x["K"])
    four.route(x["Q"])
    four.attn_fwd(x["Q"], x["K"], x["V"])
    if bwd:
        four.attn_bwd(x["Q"], x["K"], x["V"], x["dO"])
    torch.cuda.synchronize()
    late = {k: torch.empty_like(v) for k, v in x.items()}
    for rep in range(3):
        for k in late:                       # written by the kernels right before the step
            late[k].fill_(float(rep))
            late[k].copy_(x[k])
        one.step(late["Q"], late["K"], late["V"], late["dO"] if bwd else None)
    torch.cuda.synchronize()
    assert int(one.status.item()) == 0
    for k in ("chunk_idx", "group_idx", "n_groups", "chunk_sum", "group_sum", "O", "LSE"):
        assert torch.equal(getattr(one, k), getattr(four, k)), k
    if bwd:
        # (up to the order of fp32 additions, and one rounding where the outputs are bf16)
        assert torch.equal(one.dQ, four.dQ)
        for k in ("dQ", "dK", "dV"):
            a, b = getattr(one, k).float(), getattr(four, k).float()
            assert float((a - b).norm()) <= (2.0 ** -9 if getattr(one, k).dtype == torch.bfloat16 else 1e-5) * float(b.norm()), k


def test_step_refuses_what_its_calls_refuse():
    cfg = cfg_of()
    x = {k: to_dev(v) for k, v in make_inputs(cfg).items() if k in ("Q", "K", "V", "dO")}
    buf = binding.HgaLayerBuffers(cfg)
    before = binding.hga_kernel_launch_count()
    for bit in (1 << 29, 1 << 30, 128):
        buf.p.flags = bit
        with pytest.raises(binding.HgaError):
            buf.step(x["Q"], x["K"], x["V"], x["dO"])
    assert binding.hga_kernel_launch_count() == before
    buf.p.flags = 0
    buf.route_ws = buf.route_ws[:8]
    with pytest.raises(binding.HgaError):
        buf.step(x["Q"], x["K"], x["V"], x["dO"])


HEADS = {"d128": dict(n_q_heads=32, n_kv_heads=8), "d64_rows64": dict(head_dim=64, n_q_heads=16, n_kv_heads=16)}


def outputs(cfg):
    """Tensors of a whole sequence of one row (walk, or step where it is one segment) or of packed documents."""
    Hq, Hkv, d, n = cfg.n_q_heads, cfg.n_kv_heads, cfg.head_dim, cfg.total_len
    z = lambda *s, dt=torch.bfloat16: torch.zeros(*s, dtype=dt, device="cuda")
    items = Hkv * n // cfg.q_block
    return dict(cs=z(Hkv, n // cfg.chunk, d), gs=z(Hkv, n // cfg.group, d), ci=z(items, cfg.topk_chunks, dt=torch.int32),
                gi=z(items, cfg.topk_chunks * cfg.kg_eff, dt=torch.int32), ng=z(items, dt=torch.int32), O=z(Hq * n * d).fill_(3.0),
                LSE=z(Hq * n, dt=torch.float32), dQ=z(Hq * n * d), dK=z(Hkv * n * d, dt=torch.float32), dV=z(Hkv * n * d, dt=torch.float32))


def one_call(kind, cfg, x, o, dO, status, flags=0):
    """The step (with and without summaries to build first), the walk in segments of a third, or three packed documents of a third
    each: no history, dO may be None."""
    n, third = cfg.total_len, cfg.total_len // 3
    args = [x["Q"], x["K"], x["V"], dO] + [o[k] for k in ("cs", "gs", "ci", "gi", "ng", "O", "LSE", "dQ", "dK", "dV")]
    if kind in ("step", "step_without_summaries"):
        p = binding.make_params(cfg, flags=flags)
        w1, w2 = (torch.empty(b, dtype=torch.uint8, device="cuda") for b in binding.hga_workspace_bytes(p))
        binding.hga_layer_step(p, *args[:4], 0 if kind == "step" else n, n, *args[4:9], None, None, *args[9:], w1, w2, status)
    elif kind == "walk":
        p = binding.make_params(cfg.scaled(seg_len=third), flags=flags)
        binding.hga_tbptt_walk(p, *args, torch.empty(sum(binding.hga_workspace_bytes(p)) + 512, dtype=torch.uint8, device="cuda"), status)
    else:
        cu = [0, third, 2 * third, n]
        p = binding.make_params(cfg, flags=flags)
        binding.hga_varlen_step(p, cu, cu, *args, torch.empty(binding.hga_varlen_workspace_bytes(p, cu, cu), dtype=torch.uint8, device="cuda"), status)


def random_inputs(cfg, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    draw = lambda h: torch.randn(h * cfg.total_len * cfg.head_dim, generator=gen, device="cuda").to(torch.bfloat16)
    return dict(Q=draw(cfg.n_q_heads), K=draw(cfg.n_kv_heads), V=draw(cfg.n_kv_heads), dO=draw(cfg.n_q_heads))


def check_equal(a, b, keys):
    for k in keys:
        if k in ("dK", "dV"):                # up to the order of their fp32 adds
            assert float((a[k] - b[k]).norm()) <= 1e-5 * float(b[k].norm()), k
        else:
            assert torch.equal(a[k], b[k]), k


@pytest.mark.parametrize("heads", list(HEADS))
@pytest.mark.parametrize("kind", ["step", "walk", "packed"])
def test_the_gradient_may_be_the_output(kind, heads):
    """dO is O (the gradient of |O|^2 / 2), against a call with a copy of that O as dO."""
    cfg = cfg_of(total_len=3072, seg_len=3072, **HEADS[heads])
    x, status = random_inputs(cfg, 5), torch.zeros(1, dtype=torch.int32, device="cuda")
    ref, got = outputs(cfg), outputs(cfg)
    one_call(kind, cfg, x, ref, None, status)
    torch.cuda.synchronize()
    one_call(kind, cfg, x, ref, ref["O"].clone(), status)
    for _ in range(3):
        got["O"].fill_(3.0)
        one_call(kind, cfg, x, got, got["O"], status)
        torch.cuda.synchronize()
        assert int(status.item()) == 0
        check_equal(got, ref, ("gi", "ng", "O", "LSE", "dQ", "dK", "dV"))


@pytest.mark.parametrize("heads", list(HEADS))
@pytest.mark.parametrize("over", ["Q", "dO", "O"])
@pytest.mark.parametrize("kind", ["bwd", "step", "walk", "packed"])
def test_dq_may_take_the_place_of_an_input(kind, over, heads):
    """dQ in the buffer of Q, dO or O, by hga_attn_bwd itself and by the calls that make it, against buffers of its own."""
    cfg = cfg_of(total_len=3072, seg_len=3072, **HEADS[heads])
    x, status = random_inputs(cfg, 6), torch.zeros(1, dtype=torch.int32, device="cuda")
    ref = outputs(cfg)
    one_call("step" if kind == "bwd" else kind, cfg, x, ref, x["dO"], status)
    torch.cuda.synchronize()
    for _ in range(3):
        got, y = outputs(cfg), {k: v.clone() for k, v in x.items()}
        if kind == "bwd":
            one_call("step", cfg, y, got, None, status)
        got["dQ"] = got["O"] if over == "O" else y[over]
        if kind == "bwd":
            p = binding.make_params(cfg)
            ws = torch.empty(binding.hga_workspace_bytes(p)[1], dtype=torch.uint8, device="cuda")
            binding.hga_attn_bwd(p, y["Q"], y["K"], y["V"], got["O"], got["LSE"], y["dO"], got["gi"], got["ng"], got["dQ"], got["dK"], got["dV"], ws, status)
        else:
            one_call(kind, cfg, y, got, y["dO"], status)
        torch.cuda.synchronize()
        assert int(status.item()) == 0
        check_equal(got, ref, ("gi", "ng", "LSE", "dQ", "dK", "dV"))


@pytest.mark.parametrize("heads", list(HEADS))
@pytest.mark.parametrize("kind", ["step", "step_without_summaries", "walk", "packed"])
def test_inputs_that_are_being_written(kind, heads):
    """Q and dO are dQ of the step right before: its last kernel lets its successor start long before it has stored them."""
    cfg = cfg_of(total_len=3072, seg_len=3072, **HEADS[heads])
    x, status = random_inputs(cfg, 7), torch.zeros(1, dtype=torch.int32, device="cuda")
    before = outputs(cfg)
    ref, got = outputs(cfg), outputs(cfg)
    for o in (ref, got):
        binding.hga_build_summaries(binding.make_params(cfg), x["K"], 0, cfg.total_len, o["cs"], o["gs"])

    def both(o, wait):
        before["dQ"].fill_(0.5)
        torch.cuda.synchronize()
        one_call("step", cfg, x, before, x["dO"], status)
        if wait:
            torch.cuda.synchronize()
        one_call(kind, cfg, dict(x, Q=before["dQ"]), o, before["dQ"], status)
        torch.cuda.synchronize()

    both(ref, True)
    for _ in range(3):
        both(got, False)
        assert int(status.item()) == 0
        check_equal(got, ref, ("gi", "ng", "O", "LSE", "dQ", "dK", "dV"))


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("rows", ["60_of_an_item", "one_key_round"])
def test_cuda_core_backward_with_two_ctas_per_eight_rows(rows, d):
    """Few rows: every eight of them have a cluster of two CTAs.  A last eight that is not full, keys of odd numbers of rounds, and so few
    keys that the second CTA may have none."""
    kw = dict(n_q_heads=3, q_block=20, chunk=20, group=4, seg_len=100, total_len=400, sink=20, local=40) if rows == "60_of_an_item" else \
        dict(n_q_heads=1, q_block=12, chunk=12, group=4, seg_len=60, total_len=60, sink=12, local=12, topk_chunks=3)
    cfg = cfg_of(**{**dict(n_kv_heads=1, head_dim=d, topk_chunks=4, topics=0), **kw})
    slices = cfg.n_items * -(-cfg.gqa * cfg.q_block // 8)
    assert 2 * slices <= torch.cuda.get_device_properties(0).multi_processor_count
    assert cfg.sink + cfg.topk_chunks * cfg.kg_eff * cfg.group + cfg.local + cfg.q_block + cfg.chunk > 64      # (the rule's bound of an item's keys)
    x = make_inputs(cfg)
    dev = {k: to_dev(x[k]) for k in ("Q", "K", "V", "dO")}
    buf = binding.HgaLayerBuffers(cfg)
    buf.build_summaries(dev["K"], 0, cfg.total_len)
    before = binding.hga_kernel_launch_counts()
    buf.step(dev["Q"], dev["K"], dev["V"], dev["dO"])
    torch.cuda.synchronize()
    ran = [b - a for a, b in zip(before, binding.hga_kernel_launch_counts())]
    assert ran[binding.HGA_KERNELS_BWD_GENERIC] == 2 and int(buf.status.item()) == 0
    ref = oracle.attn_bwd(cfg, x["Q"], x["K"], x["V"], x["dO"], buf.group_idx.cpu().numpy(), buf.n_groups.cpu().numpy())
    got = (bf16_to_f64(buf.dQ), buf.dK.cpu().numpy().astype("f8"), buf.dV.cpu().numpy().astype("f8"))
    check_grads(got, ref, rows)
    # no rounded tensor enters dV: fp32 weights (__expf: some ulp, fp32 logits and LSE: 1e-6) times bf16 inputs, summed in fp32
    assert float(((got[2] - ref[2]) ** 2).sum() ** 0.5) <= 1e-5 * float((ref[2] ** 2).sum() ** 0.5)
