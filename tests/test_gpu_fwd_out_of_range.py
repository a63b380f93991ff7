"""Rows of the forward kernel whose exponentials leave the range of the first tile's reference: every row of every item at
once, infinities and NaN in the inputs, values that only such a reference takes out of the fp32 range, a first tile without
a finite logit; and that none of it costs more than a small multiple of an ordinary call."""
import numpy as np
import pytest
import torch

import oracle
from paper_2607_15105_b200 import binding
from paper_2607_15105_b200.workloads import HgaConfig, f32_to_bf16_bits, make_inputs

from hga_testlib import TOL_LSE, TOL_O, bf16_to_f64, to_dev

pytestmark = pytest.mark.gpu


def cfg_of(**kw):
    base = dict(name="range", batch=1, n_q_heads=8, n_kv_heads=2, head_dim=128, total_len=3072, seg_len=1024,
                chunk=64, group=8, q_block=64, topk_chunks=12, topk_groups=4, sink=64, local=128, topics=16, needles=0,
                backward=False, seed=29)
    base.update(kw)
    return HgaConfig(**base)


CASES = {"d128": cfg_of(), "d64_rows64": cfg_of(head_dim=64, n_q_heads=2), "d128_rows192": cfg_of(n_q_heads=6),
         "decode_20_rows": cfg_of(total_len=3005, seg_len=5, q_block=5, decode=True)}
# (an ordinary pass, one for the maxima and one against them, the last two with nothing overlapped: 3 to 7 times)
MOST = 15.0
bits = lambda v: f32_to_bf16_bits(np.array([v], np.float32))[0]


class Problem:
    def __init__(self, name):
        self.cfg = cfg = CASES[name]
        x = make_inputs(cfg)
        self.Q, self.K, self.V = x["Q"].copy(), x["K"].copy(), x["V"].copy()
        cs, gs = oracle.build_summaries(cfg, self.K)
        ref = oracle.route(cfg, self.Q, cs, gs)
        self.gi, self.ng = ref["group_idx"], ref["n_groups"]

    def time(self, Q, K, V):
        """O, LSE and the fastest of a few calls (us)"""
        buf = binding.HgaLayerBuffers(self.cfg, backward=False)
        dev = [to_dev(a) for a in (Q, K, V)]
        gid, ngd = torch.from_numpy(self.gi).cuda(), torch.from_numpy(self.ng).cuda()
        best = np.inf
        for _ in range(6):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            buf.attn_fwd(*dev, gid, ngd)
            b.record()
            torch.cuda.synchronize()
            best = min(best, 1e3 * a.elapsed_time(b))
        assert int(buf.status.item()) == 0
        return bf16_to_f64(buf.O), buf.LSE.cpu().numpy().astype(np.float64), best

    def plant(self, orders):
        """A sink key whose logit lies `orders` binary orders above every other for all rows; component 0 belongs to it."""
        Q, K = self.Q.copy(), self.K.copy()
        K[..., 0] = 0
        K[:, :, 3, 0] = bits(48.0)
        Q[..., 0] = bits(orders * np.log(2.0) * np.sqrt(self.cfg.head_dim) / 48.0)
        return Q, K


@pytest.mark.parametrize("name", list(CASES))
def test_every_row_past_the_range(name):
    pr = Problem(name)
    plain = pr.time(pr.Q, pr.K, pr.V)[2]
    Q, K = pr.plant(110)
    O, LSE, us = pr.time(Q, K, pr.V)
    O_ref, LSE_ref = oracle.attn_fwd(pr.cfg, Q, K, pr.V, pr.gi, pr.ng)
    assert np.max(np.abs(O - O_ref)) <= TOL_O
    assert np.max(np.abs(LSE - LSE_ref)) <= TOL_LSE
    print(name, "%.1f us, ordinary %.1f" % (us, plain))
    assert us <= MOST * plain


@pytest.mark.parametrize("name", list(CASES))
def test_nan_key(name):
    pr = Problem(name)
    plain = pr.time(pr.Q, pr.K, pr.V)[2]
    K = pr.K.copy()
    K[:, :, 5, 7] = 0x7fc0
    O, LSE, us = pr.time(pr.Q, K, pr.V)
    assert np.all(np.isnan(O)) and np.all(np.isnan(LSE))
    print(name, "%.1f us, ordinary %.1f" % (us, plain))
    assert us <= MOST * plain


@pytest.mark.parametrize("name", list(CASES))
def test_infinite_key(name):
    """Rows whose product with it is -inf do not see the key; where it is +inf there is no finite answer."""
    pr = Problem(name)
    plain = pr.time(pr.Q, pr.K, pr.V)[2]
    K = pr.K.copy()
    K[:, :, 5, 7] = 0x7f80
    O, LSE, us = pr.time(pr.Q, K, pr.V)
    sees_minus = (pr.Q[..., 7] & 0x8000) != 0
    K[:, :, 5, 7] = bits(3e38)
    Q = pr.Q.copy()
    Q[..., 7] = np.where(sees_minus, Q[..., 7], 0)
    O_ref, LSE_ref = oracle.attn_fwd(pr.cfg, Q, K, pr.V, pr.gi, pr.ng)      # (-1e35 and the like weigh nothing either)
    nonzero = (pr.Q[..., 7] & 0x7fff) != 0
    ok = sees_minus & nonzero
    assert np.all(np.isnan(O[~ok])) and np.max(np.abs(O[ok] - O_ref[ok])) <= TOL_O
    assert np.max(np.abs(LSE[ok] - LSE_ref[ok])) <= TOL_LSE
    print(name, "%.1f us, ordinary %.1f" % (us, plain))
    assert us <= MOST * plain


@pytest.mark.parametrize("name", list(CASES))
def test_values_that_only_the_reference_takes_out_of_range(name):
    """A weight of 2^60 against the first tile's reference times values of 2^100: O itself is of the values' size."""
    pr = Problem(name)
    Q, K = pr.plant(60)
    V = f32_to_bf16_bits((pr.V.astype(np.uint32) << 16).view(np.float32) * np.float32(2.0 ** 100))
    O, LSE, _ = pr.time(Q, K, V)
    O_ref, LSE_ref = oracle.attn_fwd(pr.cfg, Q, K, V, pr.gi, pr.ng)
    assert np.max(np.abs(O - O_ref)) <= TOL_O * 2.0 ** 100
    assert np.max(np.abs(LSE - LSE_ref)) <= TOL_LSE


def test_first_tile_without_a_finite_logit():
    cfg = cfg_of(local=0, seg_len=128)
    x = make_inputs(cfg)
    cs, gs = oracle.build_summaries(cfg, x["K"])
    ref = oracle.route(cfg, x["Q"], cs, gs)
    K, Q = x["K"].copy(), x["Q"].copy()
    Q[..., 0] = bits(1.0)
    K[:, :, :cfg.sink, 0] = 0xff80                      # -inf: the sink and the active segment weigh nothing,
    K[:, :, cfg.history:, 0] = 0xff80                   # which leaves the routed groups behind the first tile
    Kf = K.copy()
    Kf[..., 0] = np.where(K[..., 0] == 0xff80, bits(-1e30), K[..., 0])
    gid, ngd = torch.from_numpy(ref["group_idx"]).cuda(), torch.from_numpy(ref["n_groups"]).cuda()
    O_ref, LSE_ref = oracle.attn_fwd(cfg, Q, Kf, x["V"], ref["group_idx"], ref["n_groups"])
    buf = binding.HgaLayerBuffers(cfg, backward=False)
    buf.attn_fwd(to_dev(Q), to_dev(K), to_dev(x["V"]), gid, ngd)
    torch.cuda.synchronize()
    assert int(buf.status.item()) == 0
    assert np.max(np.abs(bf16_to_f64(buf.O) - O_ref)) <= TOL_O
    assert np.max(np.abs(buf.LSE.cpu().numpy().astype(np.float64) - LSE_ref)) <= TOL_LSE
