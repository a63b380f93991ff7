"""hga_layer_step (HgaLayerBuffers.step) against its four calls made one by one: the same lists and outputs, with inputs that a
kernel ahead of it in the stream has just written, on every kernel family, and the status codes of the four."""
import pytest
import torch

from paper_2607_15105_b200 import binding
from paper_2607_15105_b200.workloads import HgaConfig, make_inputs

from hga_testlib import to_dev

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
        assert torch.equal(one.dQ, four.dQ) or name == "cuda_cores"
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
