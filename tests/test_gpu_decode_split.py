"""The few-position weight pass where K is split over a cluster of CTAs: heads of few weight rows, with long and short K, one
and many positions (a full 128-position batch needs the largest exchange), sum units alone in a tile, wide mixtures whose
logits stay unnormalised. Bytes as the oracle's except within 1e-6 of a boundary, log-probabilities to 2e-3, as everywhere."""
import numpy as np
import pytest

from oracle import mtpc_oracle as orc
from paper_2511_11346_b200 import inputs as I
from paper_2511_11346_b200.runner import DeviceHead

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("family,n,r,v,d,P,wpp", [
    (I.CP, 1, 1, 16, 2048, 1, 1),           # one tile and a sum tile: clusters of eight
    (I.CP, 2, 4, 48, 1088, 128, 2),         # 17 K blocks split unevenly, 128 positions
    (I.CP, 2, 64, 16, 512, 17, 3),          # 64 components: unnormalised mixture logits
    (I.HMM, 4, 8, 112, 4096, 33, 2),        # 3584 rows: clusters of two to four
    (I.HMM_CTX, 3, 16, 80, 1024, 70, 1),    # 528 sum rows with their bias
    (I.BTREE, 8, 8, 64, 256, 5, 4),         # four K blocks: no split
])
def test_drafts_of_heads_with_few_weight_rows(family, n, r, v, d, P, wpp):
    wl = I.make_workload("ksplit", I.HeadShape(family, n, r, v, d), P, seed=8200 + n + r + P, wpp=wpp, weight_std=0.1)
    dh = DeviceHead(wl)
    for _ in range(2):                       # the second draft follows the first with its launches overlapped
        out_bytes, out_lp = dh.draft_sample()
    assert dh.head.mtpc_get_status() == 0
    ref = orc.draft_sample(family, wl.hidden_q, wl.W_emit_q, wl.W_sum_q, wl.T_static, wpp, wl.uniforms)
    differ = (out_bytes.cpu().numpy() != ref["bytes"]).any(axis=1)
    assert not (differ & (ref["margin"] >= 1e-6)).any()
    assert np.abs(out_lp.cpu().numpy()[~differ] - ref["logprob"][~differ]).max() <= 2e-3
    dh.close()


@pytest.mark.parametrize("family,n,r,v,P", [
    (I.BTREE, 8, 32, 256, 40),               # four tiles a CTA in two passes of two, sum tiles between them
    (I.HMM_CTX, 6, 32, 256, 100),            # 128 positions' accumulators: passes of two
])
def test_drafts_of_heads_with_several_tiles_per_cta(family, n, r, v, P):
    wl = I.make_workload("passes", I.HeadShape(family, n, r, v, 64), P, seed=8300 + n, wpp=1, weight_std=0.2)
    dh = DeviceHead(wl)
    out_bytes, out_lp = dh.draft_sample()
    assert dh.head.mtpc_get_status() == 0
    ref = orc.draft_sample(family, wl.hidden_q, wl.W_emit_q, wl.W_sum_q, wl.T_static, 1, wl.uniforms)
    differ = (out_bytes.cpu().numpy() != ref["bytes"]).any(axis=1)
    assert not (differ & (ref["margin"] >= 1e-6)).any()
    assert np.abs(out_lp.cpu().numpy()[~differ] - ref["logprob"][~differ]).max() <= 2e-3
    dh.close()
