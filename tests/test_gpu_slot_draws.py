"""Byte draws of the few-position draft at the edges of its builds: vocabularies of an odd, an even and a four-fold number of symbols
per lane, padded ones, more and fewer draws than half the units (the units' weights are kept in shared memory only with more),
static transitions as running sums, windows beyond one per warp. Bytes the oracle's except within 1e-6 of a boundary (fp32 running
sums of at most 512 weights), log-marginals to 2e-3."""
import numpy as np
import pytest

from oracle import mtpc_oracle as orc
from paper_2511_11346_b200 import inputs as I
from paper_2511_11346_b200.runner import DeviceHead

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("family,n,r,v,vv,P,wpp", [
    (I.CP, 4, 16, 272, 260, 5, 8),          # nine symbols per lane
    (I.CP, 2, 64, 320, 0, 3, 40),           # a mixture wider than a warp, three rounds of windows
    (I.HMM, 9, 32, 512, 0, 2, 16),          # static tables and weights together beyond one CTA's share
    (I.HMM, 5, 4, 16, 0, 7, 1),
    (I.HMM, 1, 8, 48, 44, 3, 4),            # no transition at all
    (I.HMM_CTX, 4, 16, 128, 0, 6, 9),
    (I.BTREE, 8, 32, 256, 249, 4, 2),       # few draws on many units
    (I.BTREE, 8, 8, 192, 0, 33, 64),
])
def test_draws_against_the_oracle(family, n, r, v, vv, P, wpp):
    wl = I.make_workload("slots", I.HeadShape(family, n, r, v, 64, v_valid=vv), P, seed=7700 + n + r + v, wpp=wpp, weight_std=0.25)
    dh = DeviceHead(wl)
    b, pre = dh.draft_sample_prefix(wpp)
    assert dh.head.mtpc_get_status() == 0
    ref = orc.draft_sample(family, wl.hidden_q, wl.W_emit_q, wl.W_sum_q, wl.T_static, wpp, wl.uniforms)
    gb = b.cpu().numpy()
    differ = (gb != ref["bytes"]).any(axis=1)
    assert not (differ & (ref["margin"] >= 1e-6)).any()
    assert differ.mean() < 0.05
    logphi = orc.emission_logphi(wl.hidden_q, wl.W_emit_q)
    logw = orc.head_logw(family, wl.hidden_q, wl.W_sum_q, wl.T_static, r)
    want = orc.prefix_logprob(family, logw, logphi, wl.T_static, gb, np.repeat(np.arange(P), wpp))
    assert np.abs(pre.cpu().numpy() - want).max() <= 2e-3
    dh.close()
