"""Training call (Eq. 6) of a static HMM where its kernel can go wrong: CTAs with several batches of windows and a short last one, the
window lengths where 16, 8 and 4 warps fit beside the tables (r = 32: n = 16, 17, 24) and the first that takes the streaming kernel (25), every width
r, and states that only their evidence makes likely, whose steps are redone with logarithms. Gradients against the fp64 oracle with
the bars of tests/test_gpu_backward.py (bf16-rounded factors: relative L2 5e-3); the transition gradients never pass through bf16:
fp32 sums of at most T terms, 1e-5 of the largest entry."""
import numpy as np
import pytest
import torch

from oracle import mtpc_oracle_grad as og
from paper_2511_11346_b200 import inputs as I
from paper_2511_11346_b200.runner import DeviceHead

pytestmark = pytest.mark.gpu


def compare(wl, targets, N, gamma=0.9):
    dh = DeviceHead(wl)
    out = dh.window_loss_backward(N, wl.T // N, gamma, targets=torch.from_numpy(targets).cuda())
    assert dh.head.mtpc_get_status() == 0
    ref = og.composite_loss_grad(I.HMM, wl.hidden_q, wl.W_emit_q, wl.W_sum_q, wl.T_static, targets, N, gamma)
    assert np.abs(out["slot_loss"].cpu().numpy() - ref["slot_loss"]).max() <= 2e-3
    slot, _ = dh.window_loss(N, wl.T // N, gamma, targets=torch.from_numpy(targets).cuda())
    assert torch.equal(slot, out["slot_loss"])
    for key in ("dh", "dW_emit", "dW_sum"):
        got = out[key].cpu().numpy().astype(np.float64)
        assert np.linalg.norm(got - ref[key]) <= 5e-3 * np.linalg.norm(ref[key]) + 1e-6, key
    if wl.shape.n > 1:
        got = out["dT_static"].cpu().numpy()[: wl.shape.n - 1]
        assert np.abs(got - ref["dT_static"]).max() <= 1e-5 * np.abs(ref["dT_static"]).max() + 1e-9
    dh.close()


@pytest.mark.parametrize("n,r,N,L", [(8, 32, 3, 1667), (16, 32, 2, 90), (17, 32, 1, 77), (24, 32, 1, 40), (25, 32, 1, 40), (6, 16, 2, 1201),
                                     (5, 8, 1, 333), (4, 4, 3, 50), (7, 2, 1, 45), (4, 1, 2, 20), (1, 8, 2, 20), (40, 8, 1, 60)])
def test_gradients_match_the_oracle(n, r, N, L):
    wl = I.make_workload(f"static_{n}_{r}", I.HeadShape(I.HMM, n, r, 16, 64), N * L, seed=9100 + n + r, weight_std=0.2)
    t = wl.targets.copy().reshape(N, L, n)
    for j in range(1, n):
        t[:, max(L - j, 0):, j] = -1
    compare(wl, t.reshape(N * L, n), N)


def test_states_that_only_their_evidence_makes_likely():
    n, r, T = 5, 32, 40
    wl = I.make_workload("static_rare", I.HeadShape(I.HMM, n, r, 16, 64), T, seed=9200, weight_std=0.05)
    wl.hidden_q[:, :32] = 1.0                            # state 0: reached with probability e^-80, but the only one that emits symbol 5
    wl.W_emit_q[:, :, 5, :32] = -4.0                     # with more than e^-120
    wl.W_emit_q[:, 0, 5, :32] = 0.0
    wl.T_static[:, :, 0] = -80.0
    t = wl.targets.copy()
    t[::2, 2] = 5
    compare(wl, t, 1)


@pytest.mark.parametrize("r,logp,N", [(32, -83.0, 1), (8, -83.0, 2), (32, -76.0, 2)])
def test_columns_taken_with_logarithms(r, logp, N):
    """As above, with sums below the floor of the products (e^-83 = 2^-119.7, itself good to 2^-30) or quotients above their limit, in windows
    of both kinds, and tails in which the same state has no gradient."""
    n, L = 6, 30
    wl = I.make_workload("static_lost", I.HeadShape(I.HMM, n, r, 16, 64), N * L, seed=9230 + r, weight_std=0.05)
    wl.hidden_q[:, :32] = 1.0
    wl.W_emit_q[:, :, 5, :32] = -4.0
    wl.W_emit_q[:, 0, 5, :32] = 0.0
    wl.T_static[:, :, 0] = logp
    t = wl.targets.copy().reshape(N, L, n)
    t[:, ::2, 2] = 5
    t[:, 1::4, 3] = 5
    for j in range(1, n):
        t[:, max(L - j, 0):, j] = -1
    compare(wl, t.reshape(N * L, n), N)


@pytest.mark.parametrize("r", [32, 8])
def test_sums_below_the_normal_numbers_in_marginalised_tails(r):
    """State 0 is reached (e^-50) from state 1 alone, which the last byte before the tail makes unlikely (e^-50): the step's sum for state 0
    is subnormal, and its gradient, exactly 0 there, is not to be divided by it."""
    n, N, L = 6, 2, 30
    wl = I.make_workload("static_tail", I.HeadShape(I.HMM, n, r, 16, 64), N * L, seed=9210 + r, weight_std=0.05)
    wl.hidden_q[:, :32] = 1.0
    wl.W_emit_q[:, 1, 5, :32] = -1.5625
    wl.T_static[:, :, 0] = -200.0
    wl.T_static[:, 1, 0] = -50.0
    t = wl.targets.copy().reshape(N, L, n)
    for j in range(1, n):
        t[:, max(L - j, 0):, j] = -1
        t[:, L - j, j - 1] = 5
    compare(wl, t.reshape(N * L, n), N)
