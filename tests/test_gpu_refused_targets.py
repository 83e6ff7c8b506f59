"""Training calls on a batch with one refused target (past the vocabulary): the status bit, NaN for that window's log-probability (not
-inf: its evidence is not zero, it is undefined) or for the loss, and every other window as without it."""
import pytest
import torch

from paper_2511_11346_b200 import binding as B
from paper_2511_11346_b200 import inputs as I
from paper_2511_11346_b200.runner import DeviceHead

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("family,n,r", [(I.CP, 3, 8), (I.CP, 2, 64), (I.HMM, 3, 8), (I.HMM_CTX, 3, 4), (I.BTREE, 4, 8)])
def test_training_calls_with_a_refused_target(family, n, r):
    v, T, bad = 48, 40, 11
    wl = I.make_workload("refused", I.HeadShape(family, n, r, v, 64), T, seed=640 + n + r, weight_std=0.2)
    dh = DeviceHead(wl)
    weight = torch.full((T,), -1.0 / T, device="cuda")
    good = torch.from_numpy(wl.targets).cuda()
    t = good.clone()
    t[bad, n - 1] = v + 3
    want = dh.window_logprob_backward(weight, targets=good)["logprob"]
    got = dh.window_logprob_backward(weight, targets=t)["logprob"]
    assert dh.head.mtpc_get_status() == B.STATUS_BAD_TARGET
    keep = torch.arange(T, device="cuda") != bad
    assert torch.isnan(got[bad]) and torch.equal(got[keep], want[keep])
    loss = dh.window_loss_backward(2, T // 2, 0.9, targets=t)
    assert dh.head.mtpc_get_status() == B.STATUS_BAD_TARGET
    assert torch.isnan(loss["slot_loss"][n - 1]) and torch.isnan(loss["loss"]).all()
    assert torch.isfinite(loss["slot_loss"][:n - 1]).all()
    dh.close()
