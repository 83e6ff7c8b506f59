"""Gradients through the adaptors from one reading of the logit gradients, which heads of many units use: held to the oracle's
chain rule with the bars of tests/test_gpu_lowrank.py (derived there from the magnitudes behind every entry). One unit's symbols fill
an odd and an even number of 64-symbol boxes, one box only, and the most there can be; positions one past a tile of 128, one alone,
and a whole tile; more units than SMs; ranks 16 and 32."""
import pytest
import test_gpu_lowrank
import torch

from paper_2511_11346_b200 import binding as B
from paper_2511_11346_b200 import inputs as I
from paper_2511_11346_b200.runner import to_device_bf16

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("family,n,r,v,vv,d,k,T", [
    (I.CP, 2, 64, 320, 0, 64, 16, 140),
    (I.HMM, 5, 16, 272, 261, 64, 32, 129),
    (I.BTREE, 8, 32, 16, 0, 64, 16, 1),
    (I.CP, 2, 64, 512, 0, 64, 32, 128),
    (I.CP, 3, 128, 176, 0, 64, 16, 30),
])
def test_one_reading_of_the_logit_gradients(family, n, r, v, vv, d, k, T):
    test_gpu_lowrank.test_factored_backward_is_the_chain_rule_through_the_composition(family, n, r, v, vv, d, k, T)


@pytest.mark.parametrize("n,r,v,vv,target", [
    (3, 4, 272, 0, 277), (3, 4, 272, 260, 300),     # a last block of sixteen columns: inside its 64, in its first and second half
    (2, 64, 16, 0, 40),                             # one block, most of it beyond the unit; adaptors in one reading
])
def test_a_refused_target_reaches_no_other_unit(n, r, v, vv, target):
    """A target past the vocabulary makes its window NaN and nothing else: where the window's later slots are marginalised, the
    gradients of the next one's adaptors are those of a call in which the refused target is a valid one, bit for bit."""
    d, k, T, bad = 64, 16, 140, 37
    wl = I.make_workload("stray", I.HeadShape(I.CP, n, r, v, d, v_valid=vv), T, seed=77 + v + r, weight_std=0.2)
    W, A, Bm = (to_device_bf16(x) for x in I.lowrank_parameters(n, r, v, d, k, seed=78, weight_std=0.2, adaptor_std=0.1))
    head = B.MtpcHead(B.MTPC_CP, n, r, v, d, B.MTPC_BF16, T, 1, None, to_device_bf16(wl.W_sum_q), v_valid=vv, lowrank=(W, A, Bm))
    weight = torch.full((T,), -1.0 / T, device="cuda")
    got = []
    for first in (target, 3):
        t = torch.from_numpy(wl.targets.copy()).cuda()
        t[bad, 0], t[bad, 1:] = first, -1
        g = [torch.full(s, 7.0, device="cuda") for s in ((T, d), (n, v, d), (n, r, v, k), (n, r, k, d), (r, d))]
        out = torch.empty(T, device="cuda")
        head.mtpc_lowrank_window_logprob_backward(to_device_bf16(wl.hidden_q), t, weight, out, *g)
        status = head.mtpc_get_status()
        assert status == (B.STATUS_BAD_TARGET if first == target else 0)
        assert (~torch.isfinite(out)).nonzero().flatten().tolist() == ([bad] if first == target else [])
        got.append(g)
    (dh, dWb, dA, dB, _), (dh0, dWb0, dA0, dB0, _) = got
    keep = torch.arange(T, device="cuda") != bad
    assert torch.equal(dh[keep], dh0[keep])
    assert torch.equal(dWb[1], dWb0[1]) and torch.equal(dA[1], dA0[1]) and torch.equal(dB[1], dB0[1])
    assert torch.isfinite(dA[1]).all() and torch.isnan(dA[0]).any()
    head.mtpc_destroy()
