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


def compare(wl, t):
    dh = DeviceHead(wl)
    td = torch.from_numpy(t).cuda()
    got = dh.window_prefix_logprob(targets=td).cpu().numpy()
    ref = orc.window_prefix_logprob(I.BTREE, wl.hidden_q, wl.W_emit_q, wl.W_sum_q, None, t)
    assert np.abs(got - ref).max() <= 2e-3
    out = dh.window_loss_backward(1, wl.T, 0.9, targets=td)
    assert dh.head.mtpc_get_status() == 0
    want = og.composite_loss_grad(I.BTREE, wl.hidden_q, wl.W_emit_q, wl.W_sum_q, None, t, 1, 0.9)
    for key in ("dh", "dW_emit", "dW_sum"):
        g = out[key].cpu().numpy().astype(np.float64)
        assert np.linalg.norm(g - want[key]) <= 5e-3 * np.linalg.norm(want[key]) + 1e-6, key
    dh.close()


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
    compare(wl, t)


@pytest.mark.parametrize("n,r,T,steps", [(8, 32, 36, 2.625), (8, 32, 36, 3.25), (4, 16, 24, 2.625), (16, 8, 20, 3.25), (8, 4, 20, 2.625), (64, 32, 6, 3.25)])
def test_values_taken_with_logarithms(n, r, T, steps):
    """Value 0 of every latent but the root has probability about e^(-32 steps), below the floor of the sums, and for some windows the only
    evidence; in the others it is a column that goes by itself, and in the tails one without a gradient."""
    wl = I.make_workload("tree_lost", I.HeadShape(I.BTREE, n, r, 16, 64), T, seed=9500 + n + r, weight_std=0.05)
    wl.hidden_q[:, :32] = 1.0
    wl.W_sum_q[r:].reshape(n - 2, r, r, 64)[:, :, 0, :32] = -steps
    wl.W_emit_q[:, :, 5, :32] = -4.0
    wl.W_emit_q[:, 0, 5, :32] = 0.0
    t = wl.targets.copy()
    t[::3, 1] = 5
    t[::6, n - 2] = 5
    for j in range(1, min(n, T)):
        t[T - j:, j] = -1
    compare(wl, t)


@pytest.mark.parametrize("r", [32, 16, 8])
def test_sums_below_the_normal_numbers_in_marginalised_tails(r):
    """Node 2 of four slots covers the tail, node 1 the bytes before it. Value 1 begets value 1, emits the byte 5 with e^-50 and is the
    only one to beget value 0 (e^-50): in front of a tail the sum over node 2's table for value 0 is subnormal. Value 2 begets value 1 with
    e^-50 and otherwise value 4, which hardly emits that byte: so is its sum over node 1's table. Neither reaches a gradient (exactly 0),
    which is not to be divided by them."""
    T = 40
    wl = I.make_workload("tree_tail", I.HeadShape(I.BTREE, 4, r, 16, 64), T, seed=9400 + r, weight_std=0.05)
    wl.hidden_q[:, :32] = 1.0
    wl.W_emit_q[:, 1, 5, :32] = -1.5625
    wl.W_emit_q[:, 4, 5, :32] = -6.25
    tables = wl.W_sum_q[r:].reshape(2, r, r, 64)
    tables[:, :, 0, :32] = -6.25
    tables[:, 1:3, :, :32] = -6.25
    tables[:, 1, 0, :32] = -1.5625
    tables[:, 1, 1, :32] = 0.0
    tables[:, 2, 1, :32] = -1.5625
    tables[:, 2, 4, :32] = 0.0
    t = wl.targets.copy()
    t[::2, 1] = 5
    t[::2, 2:] = -1
    compare(wl, t)


@pytest.mark.parametrize("n,r,T", [(16, 32, 300), (8, 32, 600), (8, 16, 1000)])
def test_marginals_are_as_precise_as_the_joint(n, r, T):
    """The last prefix marginal is the joint, which its own kernel forms with logarithms throughout: the sweeps may be no further from the oracle.
    Bar: 1.1 times the joint's rms error (measured 0.97 to 1.0; with the fast logarithm behind the sums 1.2 to 1.3)."""
    wl = I.make_workload("tree_prec", I.HeadShape(I.BTREE, n, r, 64, 64), T, seed=9600, weight_std=0.15)
    dh = DeviceHead(wl)
    td = torch.from_numpy(wl.targets).cuda()
    ref = orc.window_prefix_logprob(I.BTREE, wl.hidden_q, wl.W_emit_q, wl.W_sum_q, None, wl.targets)[:, -1]
    last = dh.window_prefix_logprob(targets=td)[:, -1].cpu().numpy().astype(np.float64)
    joint = dh.window_logprob(targets=td).cpu().numpy().astype(np.float64)
    assert np.sqrt(np.mean((last - ref) ** 2)) <= 1.1 * np.sqrt(np.mean((joint - ref) ** 2))
    dh.close()
