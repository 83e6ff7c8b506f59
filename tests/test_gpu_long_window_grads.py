"""Training calls of a static HMM at the window lengths where the transition gradients fill a CTA's shared memory: r = 32 with
n = 33 and 44, where one more float per step would halve the warps, and n = 54, the longest that fits at all (one warp, exactly the
limit); n = 55 is refused. Gradients against the fp64 oracle with the bars of tests/test_gpu_backward.py: an entry's product has two
factors rounded to bf16, so relative L2 5e-3 and largest error 1e-2 of the largest magnitude."""
import numpy as np
import pytest
import torch

from oracle import mtpc_oracle_grad as og
from paper_2511_11346_b200 import binding as B
from paper_2511_11346_b200 import inputs as I
from paper_2511_11346_b200.runner import DeviceHead

pytestmark = pytest.mark.gpu


def held(name, got, ref):
    got = got.cpu().numpy().astype(np.float64)
    assert np.linalg.norm(got - ref) <= 5e-3 * np.linalg.norm(ref), name
    assert np.abs(got - ref).max() <= 1e-2 * np.abs(ref).max(), name


@pytest.mark.parametrize("n", [33, 44, 54])
def test_gradients_of_long_windows(n):
    T, gamma = 6, 0.9
    wl = I.make_workload("long_window", I.HeadShape(I.HMM, n, 32, 16, 64), T, seed=5400 + n, weight_std=0.2)
    dh = DeviceHead(wl)
    t = wl.targets.copy()
    t[2, n - 5:] = -1
    td = torch.from_numpy(t).cuda()
    weight = np.linspace(-0.5, 1.0, T).astype(np.float32)
    for call, ref in ((lambda: dh.window_logprob_backward(torch.from_numpy(weight).cuda(), targets=td),
                       og.window_logprob_grad(I.HMM, wl.hidden_q, wl.W_emit_q, wl.W_sum_q, wl.T_static, t, weight)),
                      (lambda: dh.window_loss_backward(2, T // 2, gamma, targets=td),
                       og.composite_loss_grad(I.HMM, wl.hidden_q, wl.W_emit_q, wl.W_sum_q, wl.T_static, t, 2, gamma))):
        got = call()
        assert dh.head.mtpc_get_status() == 0
        for key in ("dh", "dW_emit", "dW_sum", "dT_static"):
            held(key, got[key], ref[key])
        if "loss" in ref:
            assert np.abs(got["slot_loss"].cpu().numpy() - ref["slot_loss"]).max() <= 2e-3
    dh.close()


def test_a_longer_window_is_refused():
    wl = I.make_workload("long_window", I.HeadShape(I.HMM, 55, 32, 16, 64), 2, seed=5455, weight_std=0.2)
    dh = DeviceHead(wl)
    for call in (lambda: dh.window_logprob_backward(torch.ones(2, device="cuda")), lambda: dh.window_loss_backward(1, 2, 0.9)):
        with pytest.raises(B.MtpcError) as e:
            call()
        assert e.value.code == -3
    dh.close()
