"""Weights that mask a run of symbols: a constant feature of the hidden states and weights on it far below any logit, or -inf. The projection's
epilogue keeps two running maxima of a unit's columns, so that a run may be all that one of them has seen when it starts.

Tolerance against fp64: a logit is a sum of d products in fp32, off by at most d 2^-24 of the sum of their magnitudes (the mask's own
only where it is the target's), and 4e-6 for the sum of exponentials and its logarithm."""
import pytest
import torch

from paper_2511_11346_b200 import binding as B

pytestmark = pytest.mark.gpu

N, D = 2, 64


def _inputs(v, run, value, T):
    g = torch.Generator(device="cuda")
    g.manual_seed(v + run[0] + run[1])
    W = (0.3 * torch.randn(N, 1, v, D, device="cuda", generator=g)).bfloat16()
    hidden = torch.randn(T, D, device="cuda", generator=g).bfloat16()
    W[..., 0] = 0.0
    W[0, :, run[0]:run[1], 0] = value
    hidden[:, 0] = 1.0
    targets = torch.empty(T, N, dtype=torch.int32, device="cuda")
    free = [b for b in range(v) if value > -1e5 or not run[0] <= b < run[1]]
    targets[:, 0] = torch.tensor([free[t % len(free)] for t in range(T)], device="cuda")
    targets[:, 1] = torch.arange(T, device="cuda") % v
    return W, hidden, targets


def _reference(W, hidden, targets):
    """[T] log-likelihoods in fp64 and their slack."""
    want, slack = 0.0, 0.0
    for i in range(N):
        U = W[i, 0].double()
        mask, U[:, 0] = U[:, 0].clone(), 0.0
        logits = hidden.double() @ U.T + mask
        want = want + torch.log_softmax(logits, -1).gather(1, targets[:, i].long()[:, None])[:, 0]
        slack = slack + 2 * D * 2.0 ** -24 * (hidden.double().abs() @ U.abs().T).max(-1).values + 4e-6
    return want, slack


RUNS = [(0, 16), (16, 32), (32, 64), (0, 64), (64, 256)]


@pytest.mark.parametrize("value", [-1e4, -1e9, -1e10, -1e30, -3e38, float("-inf")])
@pytest.mark.parametrize("run", RUNS)
@pytest.mark.parametrize("v", [272, 320])
def test_log_likelihood(v, run, value):
    T = 400
    W, hidden, targets = _inputs(v, run, value, T)
    head = B.MtpcHead(B.MTPC_CP, N, 1, v, D, B.MTPC_BF16, T, 1, W, torch.zeros(1, D, device="cuda", dtype=torch.bfloat16), None)
    want, slack = _reference(W, hidden, targets)
    if value > -1e5:        # masked targets too, whose logits have the mask among their products
        slack = slack + 2 * D * 2.0 ** -24 * abs(value)
    got = []
    for variant in (1, 2):
        out = torch.empty(T, device="cuda")
        head.mtpc_debug_set_projection_variant(variant)
        head.mtpc_window_logprob(hidden, targets, out)
        assert ((out.double() - want).abs() <= slack).all()
        got.append(out)
    assert torch.equal(*got)
    assert head.mtpc_get_status() == 0
    head.mtpc_destroy()


def test_a_whole_unit_far_below():
    """Every symbol of a unit at -1e10 and below: to fp32 the largest logit is the log-sum-exp, and a target's log-probability its distance from it."""
    v, T = 272, 200
    W, hidden, targets = _inputs(v, (100, 272), -1e30, T)
    W[0, :, :100, 0] = -1e10
    head = B.MtpcHead(B.MTPC_CP, N, 1, v, D, B.MTPC_BF16, T, 1, W, torch.zeros(1, D, device="cuda", dtype=torch.bfloat16), None)
    out = torch.empty(T, device="cuda")
    head.mtpc_window_logprob(hidden, targets, out)
    want, slack = _reference(W, hidden, targets)
    assert ((out.double() - want).abs() <= slack + 2 * D * 2.0 ** -24 * 1e10).all()
    head.mtpc_destroy()


@pytest.mark.parametrize("run", RUNS)
@pytest.mark.parametrize("v", [272, 320])
def test_gradients(v, run):
    """The training call keeps the logits and their log-sum-exps: dW_emit of a masked symbol is 0, the rest that of the same head with the run
    at -1e4, where no symbol has mass either: bit for bit, since neither run contributes to any sum."""
    T = 300
    grads = []
    for value in (-1e4, -1e30):
        W, hidden, targets = _inputs(v, run, value, T)
        targets[:, 0] = torch.tensor([b for b in range(v) if not run[0] <= b < run[1]], device="cuda").repeat(T)[:T]
        head = B.MtpcHead(B.MTPC_CP, N, 1, v, D, B.MTPC_BF16, T, 1, W, torch.zeros(1, D, device="cuda", dtype=torch.bfloat16), None)
        out, dh, dW, dS = (torch.empty(*s, device="cuda") for s in ((T,), (T, D), (N, 1, v, D), (1, D)))
        head.mtpc_window_logprob_backward(hidden, targets, torch.full((T,), -1.0 / T, device="cuda"), out, dh, dW, dS)
        assert head.mtpc_get_status() == 0
        assert torch.isfinite(out).all() and torch.isfinite(dh).all() and torch.isfinite(dW).all()
        assert (dW[0, 0, run[0]:run[1]] == 0).all()
        grads.append((out, dh, dW))
        head.mtpc_destroy()
    for a, b in zip(*grads):
        assert torch.equal(a, b)
