"""Drafts of many positions on a composed head (Algorithm 1 and 3): one projection keeps its logits and everything else gathers
from them. Vocabularies that are no multiple of the accumulator tile, several windows per position, wide mixtures, and a draft
whose logits do not fit the workspace's share at once (it runs in two chunks; the acceptance stage then sorts the rejected
windows by slot and recomputes that slot's logits). Bars as everywhere: bytes the oracle's except within 1e-6 of a boundary,
log-marginals to 2e-3. The chunked draft is too large for the oracle and is held against the few-position path of the same head,
which has its own parity tests: the two differ in the order of fp32 sums only, so a byte may differ where a uniform lies within
about 1e-6 of one of 512 boundaries, less than one in a thousand."""
import numpy as np
import pytest
import torch

from oracle import mtpc_oracle as orc
from paper_2511_11346_b200 import inputs as I
from paper_2511_11346_b200.runner import DeviceHead

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("family,n,r,v,vv,P,wpp", [
    (I.CP, 3, 64, 48, 0, 129, 3),           # 64 components: normalised mixture weights on this path
    (I.HMM, 5, 8, 272, 268, 140, 2),        # padded, not a whole number of accumulator tiles
    (I.BTREE, 16, 4, 16, 0, 200, 1),
    (I.HMM_CTX, 3, 4, 1024, 0, 130, 1),     # units of more than 512 symbols
])
def test_long_drafts_against_the_oracle(family, n, r, v, vv, P, wpp):
    shape = I.HeadShape(family, n, r, v, 64, v_valid=vv)
    wl = I.make_workload("long", shape, P, seed=9500 + n + r + v, wpp=wpp, weight_std=0.25)
    dh = DeviceHead(wl)
    b, pre = dh.draft_sample_prefix(wpp)
    assert dh.head.mtpc_get_status() == 0
    ref = orc.draft_sample(family, wl.hidden_q, wl.W_emit_q, wl.W_sum_q, wl.T_static, wpp, wl.uniforms)
    gb = b.cpu().numpy()
    differ = (gb != ref["bytes"]).any(axis=1)
    assert not (differ & (ref["margin"] >= 1e-6)).any()
    logphi = orc.emission_logphi(wl.hidden_q, wl.W_emit_q)
    logw = orc.head_logw(family, wl.hidden_q, wl.W_sum_q, wl.T_static, r)
    want = orc.prefix_logprob(family, logw, logphi, wl.T_static, gb, np.repeat(np.arange(P), wpp))
    assert np.abs(pre.cpu().numpy() - want).max() <= 2e-3
    dh.close()


def test_a_draft_whose_logits_do_not_fit_at_once():
    n, r, v, d, P = 16, 32, 512, 64, 4200                   # 1 MiB of logits per position against 4 GiB kept
    wl = I.make_workload("chunks", I.HeadShape(I.BTREE, n, r, v, d), P, seed=9700, wpp=1, weight_std=0.25)
    dh = DeviceHead(wl)
    h, u = dh.hidden_device(), torch.from_numpy(wl.uniforms).cuda()
    g = torch.Generator(device="cuda")
    g.manual_seed(5)
    tp = torch.softmax(0.5 * torch.randn(P, n + 1, v, device="cuda", generator=g), dim=-1)
    ua = torch.rand(P, n + 1, device="cuda", generator=g)
    b, pre = dh.draft_sample_prefix(1, hidden=h, uniforms=u)
    acc, nxt = dh.speculative_accept(P, 1, b, pre, tp, ua)
    assert dh.head.mtpc_get_status() == 0
    few = []
    for p0 in range(0, P, 128):
        q = slice(p0, min(P, p0 + 128))
        m = q.stop - q.start
        b1, p1 = dh.draft_sample_prefix(1, hidden=h[q].contiguous(), uniforms=u[q].contiguous())
        a1, n1 = dh.speculative_accept(m, 1, b1, p1, tp[q].contiguous(), ua[q].contiguous())
        few.append((b1, p1, a1, n1))
    b1, p1, a1, n1 = (torch.cat(x) for x in zip(*few))
    assert (b != b1).float().mean() < 1e-3
    same = (b == b1).all(dim=1)
    assert same.float().mean() > 0.98
    assert (pre[same] - p1[same]).abs().max() <= 1e-3
    assert (acc[same] != a1[same]).float().mean() < 2e-3 and (nxt[same] != n1[same]).float().mean() < 5e-3
    assert acc.min() >= 0 and len(torch.unique(acc)) >= 4 and (acc < n).any()
    dh.close()
