"""The digits of the factored log-likelihood's exponentials, a quarter of which are polynomials: units whose mass is all on one symbol, so that the
unit's log-sum-exp is that symbol's logit plus the relative error of its one exponential. Every column of a unit carries the mass for sixteen logits
between -3.9 and 3.9 (bf16 values: adaptors of one column and one-hot hidden states make every logit exact); the others lie at -30.

Tolerance: the exponent's product with log2 e, below 8, is off by 2^-22 + 1e-7 and the exponential by 2^-22 relative (the unit; the polynomial 8e-8); the
logarithm of the sum, below 8 in magnitude, by 2^-22 relative, its merge by another 2^-22 and the target's difference by 2^-22: 2.0e-6 together."""
import pytest
import torch

from paper_2511_11346_b200 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("v,k", [(64, 16), (64, 32), (80, 16)])
def test_one_symbol_at_a_time(v, k):
    n, d = 64, 64
    count = n * k
    g = torch.Generator(device="cuda")
    g.manual_seed(v + k)
    y = torch.linspace(-3.9, 3.9, count, device="cuda")[torch.randperm(count, device="cuda", generator=g)].bfloat16()
    column = torch.arange(count, device="cuda") % v
    A = torch.full((n, 1, v, k), -30.0, device="cuda", dtype=torch.bfloat16)
    slot, c = torch.arange(count, device="cuda") // k, torch.arange(count, device="cuda") % k
    A[slot, 0, column, c] = y
    Bm = torch.eye(k, d, device="cuda", dtype=torch.bfloat16).expand(n, 1, k, d).contiguous()
    head = B.MtpcHead(B.MTPC_CP, n, 1, v, d, B.MTPC_BF16, count, 1, None, torch.zeros(1, d, device="cuda", dtype=torch.bfloat16),
                      lowrank=(torch.zeros(n, v, d, device="cuda", dtype=torch.bfloat16), A, Bm))
    hidden = torch.zeros(count, d, device="cuda", dtype=torch.bfloat16)
    hidden[torch.arange(count, device="cuda"), c] = 1.0
    targets = torch.full((count, n), -1, dtype=torch.int32, device="cuda")
    targets[torch.arange(count, device="cuda"), slot] = column.int()
    out = torch.empty(count, device="cuda")
    head.mtpc_window_logprob(hidden, targets, out)
    logits = A[slot, 0, :, c].double()
    want = torch.log_softmax(logits, -1).gather(1, column[:, None])[:, 0]
    assert head.mtpc_get_status() == 0
    assert (out.double() - want).abs().max() <= 2.0e-6
    head.mtpc_destroy()
