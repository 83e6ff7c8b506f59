"""The plain GEMMs of the training calls where their last round of tiles is cut along K: few tiles against long contractions,
single CTAs (one row of tiles) and pairs, odd numbers of row tiles, ragged K, two K segments. Gradients against the fp64 oracle
with the bars of test_gpu_backward.py (the operands' bf16 rounding: relative L2 5e-3, largest error 1e-2 of the largest
magnitude), and the same bits on every run: the parts are added in K order whoever finishes last."""
import numpy as np
import pytest
import torch

from oracle import mtpc_oracle_grad as og
from paper_2511_11346_b200 import inputs as I
from paper_2511_11346_b200.runner import DeviceHead

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("family,n,r,v,d,T", [
    (I.CP, 8, 8, 320, 64, 100),       # d hidden: one tile, K = 20480; dW: 160 row tiles, K = 100
    (I.CP, 4, 8, 320, 320, 300),      # d hidden: 3 row tiles (an odd pair), K = 10240 + 8
    (I.CP, 2, 2, 48, 512, 2000),      # dW_emit: 2 row tiles x 2, K = 2000 (ragged); dW_sum: 2 rows
    (I.HMM_CTX, 4, 16, 64, 128, 770), # dW_sum: 784 rows; d hidden: two long K segments
    (I.BTREE, 8, 8, 272, 192, 257),
])
def test_gradients_where_the_last_round_is_cut(family, n, r, v, d, T):
    wl = I.make_workload("split", I.HeadShape(family, n, r, v, d), T, seed=7100 + n + r + v + T, weight_std=0.2)
    dh = DeviceHead(wl)
    weight = np.random.default_rng(T).normal(size=T).astype(np.float32)
    wd = torch.from_numpy(weight).cuda()
    a = dh.window_logprob_backward(wd)
    b = dh.window_logprob_backward(wd)
    assert dh.head.mtpc_get_status() == 0
    want = og.window_logprob_grad(wl.shape.family, wl.hidden_q, wl.W_emit_q, wl.W_sum_q, wl.T_static, wl.targets, weight)
    for key in ("dh", "dW_emit", "dW_sum"):
        assert torch.equal(a[key], b[key]), key
        got, ref = a[key].cpu().numpy().astype(np.float64), want[key]
        assert np.linalg.norm(got - ref) <= 5e-3 * np.linalg.norm(ref), key
        assert np.abs(got - ref).max() <= 1e-2 * np.abs(ref).max(), key
    dh.close()
