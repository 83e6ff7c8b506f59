"""What a draft leaves for the acceptance stage depends on P and wpp alone: not on whether it returned joints or prefix marginals, and
not on what the calls before it were. So an acceptance call recorded into a CUDA graph after one draft serves every later draft of the
same size, of either kind: the replay returns what a plain call returns."""
import pytest
import torch

from paper_2511_11346_b200 import inputs as I
from paper_2511_11346_b200.runner import DeviceHead

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("recorded_after", ["joints", "prefixes"])
@pytest.mark.parametrize("family,n,r,v,P,wpp,rank", [
    (I.CP, 6, 16, 64, 9, 16, 0), (I.CP, 4, 64, 48, 5, 16, 0), (I.HMM, 6, 16, 64, 9, 16, 0), (I.HMM_CTX, 4, 8, 48, 9, 16, 0),
    (I.BTREE, 8, 8, 64, 9, 16, 0), (I.BTREE, 8, 8, 64, 150, 2, 0), (I.BTREE, 4, 8, 48, 9, 16, 16), (I.HMM, 5, 8, 48, 150, 1, 16),
])
def test_a_recorded_acceptance_call_serves_every_later_draft(family, n, r, v, P, wpp, rank, recorded_after):
    wl = I.make_workload("state", I.HeadShape(family, n, r, v, 64), P, seed=2500 + n + r, wpp=wpp, weight_std=0.25)
    lowrank = I.lowrank_parameters(n, r, v, 64, rank, seed=2600, weight_std=0.25, adaptor_std=0.2) if rank else None
    dh = DeviceHead(wl, lowrank=lowrank)
    W = P * wpp
    hidden = dh.hidden_device()
    tp = torch.softmax(torch.from_numpy(0.4 * I._normal(33, 2, (W, n + 1, v), 1.0)).cuda(), dim=-1)
    ua = torch.from_numpy(I.uniforms(33, 3, (W, n + 1))).cuda()
    u = [torch.from_numpy(I.uniforms(34 + i, 3, (W, 2 * n))).cuda() for i in range(2)]
    draft, prefix, joint = (torch.zeros(s, dtype=t, device="cuda") for s, t in
                            (((W, n), torch.int32), ((W, n), torch.float32), ((W,), torch.float32)))
    accepted, nxt = (torch.zeros(W, dtype=torch.int32, device="cuda") for _ in range(2))

    def accept():
        dh.head.mtpc_speculative_accept(P, wpp, draft, prefix, tp, ua, accepted, nxt)

    want = []
    for ui in u:
        dh.head.mtpc_draft_sample_prefix(hidden, wpp, ui, draft, prefix)
        accept()
        want.append((draft.clone(), prefix.clone(), accepted.clone(), nxt.clone()))
    assert ((want[0][2] > 0) & (want[0][2] < n)).any()                  # rejections whose posterior depends on the bytes before them
    if recorded_after == "joints":
        dh.head.mtpc_draft_sample(hidden, wpp, u[0], draft, joint)
    else:
        dh.head.mtpc_draft_sample_prefix(hidden, wpp, u[0], draft, prefix)
    accept()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        accept()
    for i in (1, 0):
        prefix.copy_(want[i][1])
        dh.head.mtpc_draft_sample(hidden, wpp, u[i], draft, joint)
        accepted.zero_()
        nxt.zero_()
        graph.replay()
        assert torch.equal(draft, want[i][0]) and torch.equal(accepted, want[i][2]) and torch.equal(nxt, want[i][3])
        assert (joint - want[i][1][:, -1]).abs().max() <= 1e-4
    assert dh.head.mtpc_get_status() == 0
    del graph
    dh.close()
