"""Plain GEMMs of fewer tiles than SMs and long K, which CTA pairs take: an odd number of row tiles, ragged rows and K. Gradients against the
fp64 oracle with the bars of test_gpu_backward.py (relative L2 5e-3, largest error 1e-2 of the largest magnitude), the same bits on every run."""
import numpy as np
import pytest
import torch

from oracle import mtpc_oracle_grad as og
from paper_2511_11346_b200 import inputs as I
from paper_2511_11346_b200.runner import DeviceHead

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("family,n,r,v,d,T", [
    (I.CP, 4, 4, 272, 1024, 1300),    # d hidden: 11 x 4 tiles, 69 K blocks and 4 sum rows
    (I.HMM, 2, 8, 256, 1280, 1000),   # 8 x 5 tiles, 64 K blocks
])
def test_gradients(family, n, r, v, d, T):
    wl = I.make_workload("pairs", I.HeadShape(family, n, r, v, d), T, seed=7700 + T, weight_std=0.1)
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
