"""The slot messages of the acceptance stage are the last draft's, whichever of the two draft calls made it and whether it, or the
acceptance call, was recorded into a CUDA graph: a recorded acceptance call serves every later draft of the same size, a plain one a
replayed draft. The acceptance call that follows a draft of prefix marginals stays one kernel."""
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


@pytest.mark.parametrize("family,n,r,v,P,wpp", [(I.CP, 6, 16, 64, 9, 16), (I.BTREE, 8, 8, 64, 150, 2)])
def test_a_plain_acceptance_call_after_replayed_drafts(family, n, r, v, P, wpp):
    wl = I.make_workload("state", I.HeadShape(family, n, r, v, 64), P, seed=2700 + n, wpp=wpp, weight_std=0.25)
    dh = DeviceHead(wl)
    W = P * wpp
    hidden = dh.hidden_device()
    tp = torch.softmax(torch.from_numpy(0.4 * I._normal(35, 2, (W, n + 1, v), 1.0)).cuda(), dim=-1)
    ua = torch.from_numpy(I.uniforms(35, 3, (W, n + 1))).cuda()
    u = [torch.from_numpy(I.uniforms(36 + i, 3, (W, 2 * n))).cuda() for i in range(2)]
    draft, prefix, joint = (torch.zeros(s, dtype=t, device="cuda") for s, t in
                            (((W, n), torch.int32), ((W, n), torch.float32), ((W,), torch.float32)))
    accepted, nxt = (torch.zeros(W, dtype=torch.int32, device="cuda") for _ in range(2))

    def accept():
        dh.head.mtpc_speculative_accept(P, wpp, draft, prefix, tp, ua, accepted, nxt)

    want = []
    for ui in u:
        dh.head.mtpc_draft_sample_prefix(hidden, wpp, ui, draft, prefix)
        before = dh.head.mtpc_launch_count()
        accept()
        assert dh.head.mtpc_launch_count() == before + 1
        want.append((prefix.clone(), accepted.clone(), nxt.clone()))

    def same(i):
        return torch.equal(accepted, want[i][1]) and torch.equal(nxt, want[i][2])

    together, alone, joints = torch.cuda.CUDAGraph(), torch.cuda.CUDAGraph(), torch.cuda.CUDAGraph()
    with torch.cuda.graph(together):                   # draft and acceptance in one graph: two calls, the messages formed once
        dh.head.mtpc_draft_sample_prefix(hidden, wpp, u[1], draft, prefix)
        before = dh.head.mtpc_launch_count()
        accept()
        assert dh.head.mtpc_launch_count() == before + 1
    with torch.cuda.graph(alone):
        dh.head.mtpc_draft_sample_prefix(hidden, wpp, u[1], draft, prefix)
    dh.head.mtpc_draft_sample_prefix(hidden, wpp, u[0], draft, prefix)
    together.replay()
    assert same(1)
    accept()                                           # plain calls after a replayed draft, with another plain draft before it
    assert same(1)
    dh.head.mtpc_draft_sample_prefix(hidden, wpp, u[0], draft, prefix)
    alone.replay()
    accept()
    assert same(1)
    with torch.cuda.graph(joints):
        dh.head.mtpc_draft_sample(hidden, wpp, u[1], draft, joint)
    dh.head.mtpc_draft_sample_prefix(hidden, wpp, u[0], draft, prefix)
    joints.replay()
    prefix.copy_(want[1][0])
    accept()
    assert same(1)
    dh.head.mtpc_draft_sample(hidden, wpp, u[0], draft, joint)
    prefix.copy_(want[0][0])
    accept()
    assert same(0)
    accept()
    assert same(0)
    assert dh.head.mtpc_get_status() == 0
    del together, alone, joints
    dh.close()
