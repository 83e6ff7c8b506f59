"""Contextual HMMs at more positions than a round of CTAs holds, where each window's tables are streamed by one warp. The recursion is
that of the CTA-per-position kernel, so a call equals the same call made in pieces that take that kernel, bit for bit: log-marginals,
and (its messages) the acceptance stage after a draft. Widths below a warp, one-state chains, no transition at all, windows whose
tables never fit a CTA (n = 64 at r = 32); marginalised bytes, a refused target. A few rows of each against the fp64 oracle, 2e-3."""
import numpy as np
import pytest
import torch

from oracle import mtpc_oracle as orc
from paper_2511_11346_b200 import binding as B
from paper_2511_11346_b200 import inputs as I
from paper_2511_11346_b200.runner import DeviceHead

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,r,T,piece", [
    (5, 8, 1650, 400), (9, 16, 1701, 600), (8, 32, 1333, 700), (4, 2, 1603, 500), (3, 1, 1500, 300), (1, 4, 1501, 300), (64, 32, 203, 100),
])
def test_a_long_call_equals_its_pieces(n, r, T, piece):
    wl = I.make_workload("ctx_stream", I.HeadShape(I.HMM_CTX, n, r, 16, 64), T, seed=7300 + n + r, weight_std=0.25)
    dh = DeviceHead(wl)
    t = wl.targets.copy()
    t[T // 2:, n - n // 3:] = -1
    t[7, 0] = 16                                           # refused
    td, h = torch.from_numpy(t).cuda(), dh.hidden_device()
    joint, pre = dh.window_logprob(hidden=h, targets=td), dh.window_prefix_logprob(hidden=h, targets=td)
    cut = [slice(i, min(i + piece, T)) for i in range(0, T, piece)]
    pieces = [(dh.window_logprob(hidden=h[c], targets=td[c]), dh.window_prefix_logprob(hidden=h[c], targets=td[c])) for c in cut]
    assert dh.head.mtpc_get_status() == B.STATUS_BAD_TARGET
    for whole, k in ((joint, 0), (pre, 1)):
        assert torch.equal(torch.nan_to_num(whole, nan=7.0), torch.nan_to_num(torch.cat([p[k] for p in pieces]), nan=7.0))
        assert torch.isnan(whole[7]).all() and torch.isfinite(whole).sum() == whole.numel() - whole[7].numel()
    rows = np.array([0, 1, T // 2 - 1, T // 2, T - 2, T - 1])
    logphi = orc.emission_logphi(wl.hidden_q[rows], wl.W_emit_q)
    logw = orc.head_logw(I.HMM_CTX, wl.hidden_q[rows], wl.W_sum_q, wl.T_static, r)
    ref = orc.prefix_logprob(I.HMM_CTX, logw, logphi, wl.T_static, t[rows])
    assert np.abs(pre.cpu().numpy()[rows] - ref).max() <= 2e-3
    assert np.abs(joint.cpu().numpy()[rows] - ref[:, -1]).max() <= 2e-3
    dh.close()


@pytest.mark.parametrize("n,r,P,wpp,piece", [    # (every piece longer than 128 positions: the same draws)
    (6, 8, 1600, 1, 400), (4, 16, 1500, 2, 300)])
def test_acceptance_after_a_long_draft_equals_that_of_its_pieces(n, r, P, wpp, piece):
    v = 48
    wl = I.make_workload("ctx_draft", I.HeadShape(I.HMM_CTX, n, r, v, 64), P, seed=7400 + n, wpp=wpp, weight_std=0.25)
    dh = DeviceHead(wl)
    h, u = dh.hidden_device(), torch.from_numpy(wl.uniforms).cuda()
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    tp = torch.softmax(0.4 * torch.randn(P * wpp, n + 1, v, device="cuda", generator=g), dim=-1)
    ua = torch.rand(P * wpp, n + 1, device="cuda", generator=g)

    def step(p):
        w = slice(p.start * wpp, p.stop * wpp)
        b, pre = dh.draft_sample_prefix(wpp, hidden=h[p], uniforms=u[w])
        return (b, pre) + dh.speculative_accept(p.stop - p.start, wpp, b, pre, tp[w], ua[w])

    whole = step(slice(0, P))
    pieces = [step(slice(i, min(i + piece, P))) for i in range(0, P, piece)]
    assert dh.head.mtpc_get_status() == 0
    for a, b in zip(whole, zip(*pieces)):
        assert torch.equal(a, torch.cat(b))
    assert len(torch.unique(whole[2])) >= 4
    dh.close()
