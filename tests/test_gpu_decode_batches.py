"""A decoding step gives a position what it gives it in any batch, bit for bit: small batches (one window per SM: the acceptance kernel that
asks for its logits ahead; a last, partial group of positions in the factored head's expansion) against the first positions of
a batch of 192 windows (the other build). Units r below, at and above the 16 and 32 logits asked for ahead; a vocabulary above one
thread per byte."""
import pytest
import torch

from paper_2511_11346_b200 import inputs as I
from paper_2511_11346_b200.runner import DeviceHead

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("family,n,r,v,rank", [(I.CP, 3, 2, 48, 0), (I.CP, 3, 8, 320, 16), (I.HMM, 5, 16, 64, 0), (I.HMM, 4, 32, 320, 32), (I.BTREE, 4, 32, 256, 0),
                                               (I.CP, 2, 128, 64, 0), (I.HMM_CTX, 3, 8, 1024, 0)])
def test_small_batches_agree_with_a_large_one(family, n, r, v, rank):
    P, wpp, d = 64, 3, 128
    wl = I.make_workload("batches", I.HeadShape(family, n, r, v, d), P, seed=9400 + r, wpp=wpp, weight_std=0.2)
    dh = DeviceHead(wl, lowrank=I.lowrank_parameters(n, r, v, d, rank, seed=9500, weight_std=0.2, adaptor_std=0.2) if rank else None)
    W = P * wpp
    h, u = dh.hidden_device(), torch.from_numpy(wl.uniforms).cuda()
    tp = torch.softmax(torch.from_numpy(0.5 * I._normal(43, 2, (W, n + 1, v), 1.0)).cuda(), dim=-1)
    ua = torch.from_numpy(I.uniforms(43, 3, (W, n + 1))).cuda()

    def step(p):
        w = p * wpp
        draft, prefix = dh.draft_sample_prefix(wpp, h[:p].contiguous(), u[:w].contiguous())
        return draft, prefix, *dh.speculative_accept(p, wpp, draft, prefix, tp[:w].contiguous(), ua[:w].contiguous())

    want = step(P)
    assert ((want[2] >= 0) & (want[2] < n)).any()            # some windows are rejected
    for p in (1, 9, 23, 40):
        for a, b in zip(step(p), want):
            assert torch.equal(a, b[: p * wpp]), p
    assert dh.head.mtpc_get_status() == 0
    dh.close()
