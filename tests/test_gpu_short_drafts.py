"""A head created with MTPC_FLAG_SHORT_DRAFTS: the same results as without it in every call on up to max_positions positions, drafts of
up to 128 of them (acceptance included), longer drafts refused. Composed and factored heads."""
import pytest
import torch

from paper_2511_11346_b200 import binding as B
from paper_2511_11346_b200 import inputs as I
from paper_2511_11346_b200.runner import DeviceHead

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("family,n,r,v,d,T,wpp,rank", [
    (I.CP, 3, 8, 64, 128, 700, 16, 0), (I.HMM_CTX, 4, 8, 48, 64, 300, 1, 0), (I.BTREE, 8, 8, 64, 64, 129, 64, 0), (I.HMM, 4, 8, 64, 64, 300, 2, 16),
])
def test_short_drafts_only(family, n, r, v, d, T, wpp, rank):
    wl = I.make_workload("short", I.HeadShape(family, n, r, v, d), T, seed=8100 + n + r, wpp=wpp, weight_std=0.25)
    dh = DeviceHead(wl, lowrank=I.lowrank_parameters(n, r, v, d, rank, seed=8200, weight_std=0.25, adaptor_std=0.2) if rank else None)
    ctx = family == I.HMM_CTX
    head = B.MtpcHead(B.MTPC_HMM if ctx else family, n, r, v, d, B.MTPC_BF16, T, wpp, dh.W_emit, dh.W_sum, dh.T_static,
                      flags=B.MTPC_FLAG_SHORT_DRAFTS | (B.MTPC_FLAG_HMM_CONTEXTUAL if ctx else 0), lowrank=dh.lowrank)
    assert head.workspace.numel() < dh.head.workspace.numel()
    h, t = dh.hidden_device(), torch.from_numpy(wl.targets).cuda()
    P = 128
    u = torch.from_numpy(wl.uniforms).cuda()
    tp = torch.softmax(torch.from_numpy(0.4 * I._normal(41, 2, (P * wpp, n + 1, v), 1.0)).cuda(), dim=-1)
    ua = torch.from_numpy(I.uniforms(41, 3, (P * wpp, n + 1))).cuda()

    def calls(x):
        joint, prefix, host = torch.empty(T, device="cuda"), torch.empty(T, n, device="cuda"), torch.empty(T)
        x.mtpc_window_logprob(h, t, joint)
        x.mtpc_window_prefix_logprob(h, t, prefix)
        x.mtpc_window_logprob_host(dh.hidden_host(), torch.from_numpy(wl.targets).pin_memory(), host)
        W = P * wpp
        draft, pre = torch.empty(W, n, dtype=torch.int32, device="cuda"), torch.empty(W, n, device="cuda")
        acc, nxt = (torch.empty(W, dtype=torch.int32, device="cuda") for _ in range(2))
        x.mtpc_draft_sample_prefix(h[:P].contiguous(), wpp, u[:W].contiguous(), draft, pre)
        x.mtpc_speculative_accept(P, wpp, draft, pre, tp, ua, acc, nxt)
        return joint, prefix, host, draft, pre, acc, nxt

    for a, b in zip(calls(dh.head), calls(head)):
        assert torch.equal(a, b)
    assert head.mtpc_get_status() == 0
    W = (P + 1) * wpp
    draft, lp, pre = torch.empty(W, n, dtype=torch.int32, device="cuda"), torch.empty(W, device="cuda"), torch.empty(W, n, device="cuda")
    few = h[:P + 1].contiguous()
    for call in (lambda: head.mtpc_draft_sample(few, wpp, u[:W].contiguous(), draft, lp),
                 lambda: head.mtpc_draft_sample_prefix(few, wpp, u[:W].contiguous(), draft, pre)):
        with pytest.raises(B.MtpcError) as e:
            call()
        assert e.value.code == -3
    head.mtpc_destroy()
    dh.close()
