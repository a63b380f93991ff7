"""The forward kernel takes a row's exponentials against its maximum over the first tile (the start of the local
window).  A sink key whose logit lies tens of binary orders above that -- inside and beyond the fp32 exponent range --
must still come out right: such rows are recomputed with a running maximum."""
import numpy as np
import pytest
import torch

import oracle
from paper_2607_15105_b200 import binding
from paper_2607_15105_b200.workloads import HgaConfig, f32_to_bf16_bits, make_inputs

from hga_testlib import TOL_LSE, TOL_O, bf16_to_f64, to_dev

pytestmark = pytest.mark.gpu


def cfg_of(**kw):
    base = dict(name="reference", batch=1, n_q_heads=4, n_kv_heads=2, head_dim=128, total_len=1536, seg_len=512,
                chunk=64, group=8, q_block=64, topk_chunks=5, topk_groups=3, sink=64, local=128, topics=16, needles=0,
                backward=False, seed=83)
    base.update(kw)
    return HgaConfig(**base)


CASES = {"d128": cfg_of(), "d64_rows64": cfg_of(head_dim=64, n_q_heads=2),
         "decode": cfg_of(total_len=1503, seg_len=3, q_block=3, decode=True)}


@pytest.mark.parametrize("orders", [70, 98, 150])
@pytest.mark.parametrize("name", list(CASES))
def test_dominant_sink_key(name, orders):
    cfg = CASES[name]
    x = make_inputs(cfg)
    K, Q = x["K"].copy(), x["Q"].copy()
    K[..., 0] = 0                                           # component 0 belongs to the planted pair alone
    Q[..., 0] = 0
    k = 48.0
    q = orders * np.log(2.0) * np.sqrt(cfg.head_dim) / k    # q * k / sqrt(d) = `orders` binary orders
    K[0, :, 3, 0] = f32_to_bf16_bits(np.array([k], np.float32))[0]
    t0 = cfg.seg_len - cfg.q_block                          # a few rows of the last block, one head per kv head
    Q[0, ::cfg.gqa, t0:t0 + 2, 0] = f32_to_bf16_bits(np.array([q], np.float32))[0]
    cs, gs = oracle.build_summaries(cfg, K)
    ref = oracle.route(cfg, Q, cs, gs)
    gi, ng = ref["group_idx"], ref["n_groups"]
    O, LSE = oracle.attn_fwd(cfg, Q, K, x["V"], gi, ng)
    assert float(LSE.max()) > 0.6 * orders                  # the planted logit is really there
    buf = binding.HgaLayerBuffers(cfg, backward=False)
    buf.attn_fwd(to_dev(Q), to_dev(K), to_dev(x["V"]), torch.from_numpy(gi).cuda(), torch.from_numpy(ng).cuda())
    torch.cuda.synchronize()
    assert int(buf.status.item()) == 0
    assert np.max(np.abs(bf16_to_f64(buf.O) - O)) <= TOL_O
    # the logit itself is a bf16 product of up to 104 nats: exact in fp32 up to 2^-24 of it
    assert np.max(np.abs(buf.LSE.cpu().numpy().astype(np.float64) - LSE)) <= TOL_LSE
