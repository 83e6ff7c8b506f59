"""The projection's epilogue: two warps take a unit's columns in turn, in batches of 32 (16 where v is no multiple of 32), and one adds their shares
up. Units of one batch (a warp then has none), of a few and of several accumulator tiles, odd numbers of batches, the last columns padding,
every column the target once, a marginalised and a refused target; CTAs alone and in pairs give the same bits.

Tolerance: a logit is a sum of d products in fp32, off by at most d 2^-24 of the sum of their magnitudes; the sum of exponentials adds
2^-22 relative for each of them and for the logarithm, in units of log2, and the rounding of the maximum's product with log2 e: with logits of a
few units below 4e-6 together."""
import pytest
import torch

from paper_2511_11346_b200 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("v,v_valid", [(16, 9), (32, 0), (48, 41), (64, 0), (96, 81), (256, 0), (272, 268), (320, 0), (800, 793), (1040, 0)])
def test_log_softmax_of_every_column(v, v_valid):
    n, r, d = 2, 1, 64
    vv = v_valid or v
    T = max(300, vv)
    g = torch.Generator(device="cuda")
    g.manual_seed(v)
    W = (0.3 * torch.randn(n, r, v, d, device="cuda", generator=g)).bfloat16()
    hidden = torch.randn(T, d, device="cuda", generator=g).bfloat16()
    zero = torch.zeros(r, d, device="cuda", dtype=torch.bfloat16)
    head = B.MtpcHead(B.MTPC_CP, n, r, v, d, B.MTPC_BF16, T, 1, W, zero, None, v_valid=v_valid)
    targets = torch.full((T, n), -1, dtype=torch.int32, device="cuda")
    targets[:, 0] = torch.arange(T, device="cuda") % vv
    targets[:T // 2, 1] = (torch.arange(T // 2, device="cuda") * 7) % vv          # the other half is marginalised
    out = torch.empty(T, device="cuda")
    head.mtpc_debug_set_projection_variant(1)
    head.mtpc_window_logprob(hidden, targets, out)
    alone = out.clone()
    head.mtpc_debug_set_projection_variant(2)
    head.mtpc_window_logprob(hidden, targets, out)
    assert torch.equal(out, alone)
    assert head.mtpc_get_status() == 0
    want = torch.zeros(T, dtype=torch.float64, device="cuda")
    slack = torch.zeros_like(want)
    for i in range(n):
        U = W[i, 0, :vv].double()
        logits = hidden.double() @ U.T
        t = targets[:, i].long()
        want += torch.where(t < 0, 0.0, torch.log_softmax(logits, -1).gather(1, t.clamp_min(0)[:, None])[:, 0])
        slack += 2 * d * 2.0 ** -24 * (hidden.double().abs() @ U.abs().T).max(-1).values + 4e-6
    assert ((out.double() - want).abs() <= slack).all()
    targets[3, 0] = vv                                  # refused: NaN there, and nowhere else
    head.mtpc_window_logprob(hidden, targets, out)
    assert torch.isnan(out[3]) and torch.isfinite(out).sum() == T - 1
