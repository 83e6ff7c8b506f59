"""The tree's sweeps run on probabilities; where a step's sum is tiny against its maximum (states that only their evidence makes likely) they
take it again with logarithms. Prefix marginals and the Eq. 6 training call on such windows beside ordinary ones, at every build of the
kernels (r = 32, 16, 8 and any other) and where the tables do not fit (n = 64), against the fp64 oracle: log-marginals 2e-3 as
everywhere, gradients relative L2 5e-3 (their factors are rounded to bf16)."""
import numpy as np
import pytest
import torch

from oracle import mtpc_oracle as orc
from oracle import mtpc_oracle_grad as og
from paper_2511_11346_b200 import inputs as I
from paper_2511_11346_b200.runner import DeviceHead

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,r,T,rare", [(8, 32, 36, True), (8, 32, 500, False), (4, 16, 24, True), (16, 8, 20, True), (8, 4, 20, True), (4, 2, 10, False),
                                        (64, 32, 6, False)])
def test_prefixes_and_gradients(n, r, T, rare):
    wl = I.make_workload("tree", I.HeadShape(I.BTREE, n, r, 16, 64), T, seed=9300 + n + r, weight_std=0.05 if rare else 0.2)
    t = wl.targets.copy()
    if rare:                                             # value 0 of every latent but the root: probability about e^-80 ...
        wl.hidden_q[:, :32] = 1.0
        tables = wl.W_sum_q[r:].reshape(n - 2, r, r, 64)
        tables[:, :, 0, :32] = -2.5
        wl.W_emit_q[:, :, 5, :32] = -4.0                 # ... but it alone emits symbol 5 with more than e^-120
        wl.W_emit_q[:, 0, 5, :32] = 0.0
        t[::2, 1] = 5
        t[1::4, n - 2] = 5
    t[1, n // 2:] = -1
    dh = DeviceHead(wl)
    td = torch.from_numpy(t).cuda()
    got = dh.window_prefix_logprob(targets=td).cpu().numpy()
    ref = orc.window_prefix_logprob(I.BTREE, wl.hidden_q, wl.W_emit_q, wl.W_sum_q, None, t)
    assert np.abs(got - ref).max() <= 2e-3
    out = dh.window_loss_backward(1, T, 0.9, targets=td)
    assert dh.head.mtpc_get_status() == 0
    want = og.composite_loss_grad(I.BTREE, wl.hidden_q, wl.W_emit_q, wl.W_sum_q, None, t, 1, 0.9)
    for key in ("dh", "dW_emit", "dW_sum"):
        g = out[key].cpu().numpy().astype(np.float64)
        assert np.linalg.norm(g - want[key]) <= 5e-3 * np.linalg.norm(want[key]) + 1e-6, key
    dh.close()
