"""Prefix marginals and slot messages of the circuit kernels at the sizes where their branches change: tables that do not fit
shared memory (n = 64 at r = 32), widths below a warp, several slot tiles of the mixture kernel, several windows per position;
and the acceptance stage after a draft that returned the joint log-probability only (it then forms the messages itself).

Bar: 2e-3 absolute against the fp64 oracle per prefix log-marginal, as everywhere (the kernels sum the same fp32 terms)."""
import numpy as np
import pytest
import torch

from oracle import mtpc_oracle as orc
from paper_2511_11346_b200 import inputs as I
from paper_2511_11346_b200.runner import DeviceHead

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("family,n,r,T", [
    (I.CP, 40, 64, 9), (I.CP, 33, 1, 5), (I.CP, 64, 128, 3),
    (I.HMM, 64, 32, 11), (I.HMM, 9, 16, 40), (I.HMM, 5, 2, 17), (I.HMM, 3, 1, 9),
    (I.HMM_CTX, 64, 32, 3), (I.HMM_CTX, 9, 16, 13), (I.HMM_CTX, 5, 2, 17),
    (I.BTREE, 64, 32, 3), (I.BTREE, 32, 32, 5), (I.BTREE, 16, 2, 19), (I.BTREE, 8, 1, 7), (I.BTREE, 2, 32, 33),
])
def test_prefix_marginals_at_the_edges_of_the_sweeps(family, n, r, T):
    wl = I.make_workload("sweep", I.HeadShape(family, n, r, 16, 64), T, seed=6100 + n + r + T, weight_std=0.25)
    t = wl.targets.copy()
    t[T // 2:, n - n // 3:] = -1                     # masked tails, as at the end of a sequence
    dh = DeviceHead(wl)
    tt = torch.from_numpy(t).cuda()
    got = dh.window_prefix_logprob(targets=tt).cpu().numpy()
    joint = dh.window_logprob(targets=tt).cpu().numpy()
    assert dh.head.mtpc_get_status() == 0
    logphi = orc.emission_logphi(wl.hidden_q, wl.W_emit_q)
    logw = orc.head_logw(family, wl.hidden_q, wl.W_sum_q, wl.T_static, r)
    ref = orc.prefix_logprob(family, logw, logphi, wl.T_static, t)
    assert np.abs(got - ref).max() <= 2e-3
    assert np.abs(joint - ref[:, -1]).max() <= 2e-3
    dh.close()


@pytest.mark.parametrize("family,n,r,v,P,wpp", [
    (I.CP, 4, 64, 48, 5, 8), (I.HMM, 6, 16, 48, 7, 8), (I.HMM_CTX, 4, 8, 48, 5, 12), (I.BTREE, 8, 8, 48, 6, 8),
    (I.BTREE, 4, 16, 32, 150, 1), (I.HMM, 3, 32, 320, 140, 1),       # more than 128 positions
])
def test_acceptance_after_a_draft_of_joints_is_that_after_a_draft_of_prefixes(family, n, r, v, P, wpp):
    wl = I.make_workload("sweep_acc", I.HeadShape(family, n, r, v, 64), P, seed=6300 + n + r, wpp=wpp, weight_std=0.25)
    dh = DeviceHead(wl)
    W = P * wpp
    h = dh.hidden_device()
    # target rows flat enough that every accepted length occurs
    tp = torch.softmax(torch.from_numpy(0.4 * I._normal(31, 2, (W, n + 1, v), 1.0)).cuda(), dim=-1)
    ua = torch.from_numpy(I.uniforms(31, 3, (W, n + 1))).cuda()
    b1, pre = dh.draft_sample_prefix(wpp, hidden=h)
    first = dh.speculative_accept(P, wpp, b1, pre, tp, ua)
    b2, joint = dh.draft_sample(wpp, hidden=h)
    second = dh.speculative_accept(P, wpp, b2, pre, tp, ua)
    assert dh.head.mtpc_get_status() == 0
    assert torch.equal(b1, b2) and (joint - pre[:, -1]).abs().max() <= 1e-4
    assert torch.equal(first[0], second[0]) and torch.equal(first[1], second[1])
    acc = first[0].cpu().numpy()
    assert len(np.unique(acc)) >= 3
    dh.close()
