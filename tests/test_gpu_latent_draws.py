"""Latent draws of a long draft (Algorithm 1 at the sum units), one warp per window: every latent's row of its table is chosen by
values other draws of the window have just produced. Trees of one, three, fifteen and sixty-three latents (the last ones in a lane's
second register), chains of up to sixty-four, mixtures wider than a warp, refused windows between good ones, a last CTA that is not
full. The peaked tables make a wrong parent show in the bytes. Bytes the oracle's except within 1e-6 of a boundary, as everywhere."""
import numpy as np
import pytest
import torch

from oracle import mtpc_oracle as orc
from paper_2511_11346_b200 import binding as B
from paper_2511_11346_b200 import inputs as I
from paper_2511_11346_b200.runner import DeviceHead

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("family,n,r,P,wpp", [
    (I.BTREE, 2, 32, 130, 1), (I.BTREE, 4, 32, 301, 1), (I.BTREE, 16, 8, 129, 3), (I.BTREE, 64, 4, 150, 1),
    (I.HMM, 64, 4, 150, 1), (I.HMM, 33, 8, 131, 1), (I.HMM_CTX, 5, 16, 130, 2), (I.CP, 2, 128, 140, 1),
])
def test_latents_of_long_drafts_against_the_oracle(family, n, r, P, wpp):
    wl = I.make_workload("latents", I.HeadShape(family, n, r, 16, 64), P, seed=9900 + n + r, wpp=wpp, weight_std=0.5)
    dh = DeviceHead(wl)
    u = wl.uniforms.copy()
    refused = [1, 6]
    u[refused, 0] = (1.0, -0.5)
    got, lp = dh.draft_sample(uniforms=torch.from_numpy(u).cuda())
    assert dh.head.mtpc_get_status(with_code=True) == (B.MTPC_OK, B.STATUS_BAD_UNIFORM)
    ref = orc.draft_sample(family, wl.hidden_q, wl.W_emit_q, wl.W_sum_q, wl.T_static, wpp, wl.uniforms)
    gb, gl = got.cpu().numpy(), lp.cpu().numpy()
    assert (gb[refused] == -1).all() and np.isnan(gl[refused]).all()
    ok = np.ones(len(gb), dtype=bool)
    ok[refused] = False
    differ = (gb != ref["bytes"]).any(axis=1) & ok
    assert not (differ & (ref["margin"] >= 1e-6)).any()
    same = ok & ~differ
    assert np.abs(gl[same] - ref["logprob"][same]).max() <= 2e-3
    dh.close()
