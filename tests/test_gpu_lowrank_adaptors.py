"""Factored projection with small and with very large adaptors (corrections of more than a hundred, where any fixed reference
would leave the exponents' range), and at the edges of its column blocks: one block of sixteen columns, a last block of 16 or of
96 columns, a padded vocabulary, more components than one round of its staging holds. A large adaptor in between leaves nothing
behind. Bar: 2e-3 absolute per log-probability against the fp64 oracle on the exactly composed tensor, plus 2e-6 per slot of
the largest logit's size for the large adaptors (fp32 sums of terms that size)."""
import numpy as np
import pytest
import torch

from oracle import mtpc_oracle as orc
from paper_2511_11346_b200 import inputs as I
from paper_2511_11346_b200.runner import DeviceHead

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("family,n,r,v,vv,d,k,T", [
    (I.CP, 2, 4, 320, 0, 128, 16, 140),
    (I.HMM, 3, 8, 272, 268, 64, 32, 70),     # last block of 16 columns, padded, rank 32
    (I.BTREE, 4, 2, 16, 0, 64, 16, 9),
    (I.CP, 1, 1, 1792, 0, 64, 16, 130),
    (I.CP, 2, 128, 96, 90, 64, 16, 129),     # four rounds of components
    (I.CP, 2, 64, 224, 0, 64, 32, 20),
])
def test_small_and_large_adaptors(family, n, r, v, vv, d, k, T):
    shape = I.HeadShape(family, n, r, v, d, v_valid=vv)
    wl = I.make_workload("bound", shape, T, seed=9100 + v + r, weight_std=0.2)
    Wb, A, Bm = I.lowrank_parameters(n, r, v, d, k, seed=9200 + v, weight_std=0.2, adaptor_std=0.1)
    sym = vv or v
    dh = DeviceHead(wl, lowrank=(Wb, A, Bm))
    hidden, targets = dh.hidden_device(), torch.from_numpy(wl.targets).cuda()
    logw = orc.head_logw(family, wl.hidden_q, wl.W_sum_q, wl.T_static, r)
    for scale in (1.0, 128.0, 1.0):
        dh.lowrank[1].copy_(torch.from_numpy(A * np.float32(scale)).to(torch.bfloat16))
        U = orc.lowrank_unembedding(Wb, A * np.float32(scale), Bm)[:, :, :sym, :]
        logphi = orc.emission_logphi(wl.hidden_q, U)
        ref = orc.prefix_logprob(family, logw, logphi, wl.T_static, wl.targets)
        got = dh.window_prefix_logprob(hidden=hidden, targets=targets).cpu().numpy()
        assert dh.head.mtpc_get_status() == 0
        largest = np.abs(np.einsum("td,nrvd->tnrv", wl.hidden_q.astype(np.float64), U)).max()
        assert (largest > 100.0) == (scale > 1.0), largest
        assert np.abs(got - ref).max() <= 2e-3 + 2e-6 * n * largest, scale
    dh.close()
