"""Factored log-likelihood where the sums of exponentials are hard: corrections of either sign far beyond the base logits (their maximum is then
no reference, and a quarter of the exponentials are polynomials on a clamped argument), hidden states that are no numbers. One unit's
log-softmax per component against fp64 on the composed matrix. Tolerance: z = B h reaches the tensor cores as two bf16 halves, 2^-17 relative, and
the sums are fp32: 2^-16 of the largest magnitude in a logit's products, and 2e-3 as everywhere."""
import pytest
import torch

from paper_2511_11346_b200 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("v,v_valid,k,r,scale", [(32, 0, 16, 1, 0.05), (80, 70, 16, 2, 3.0), (320, 0, 16, 4, 8.0), (272, 268, 32, 2, 5.0), (48, 0, 32, 1, 20.0)])
def test_corrections(v, v_valid, k, r, scale):
    n, d, T = 1, 64, 200
    g = torch.Generator(device="cuda")
    g.manual_seed(v + k)

    def normal(*shape, std):
        return torch.empty(shape, device="cuda", dtype=torch.bfloat16).normal_(0.0, std, generator=g)

    W, A, Bm = normal(n, v, d, std=0.2), normal(n, r, v, k, std=scale * k ** -0.5), normal(n, r, k, d, std=d ** -0.5)
    head = B.MtpcHead(B.MTPC_CP, n, r, v, d, B.MTPC_BF16, T, 1, None, torch.zeros(r, d, device="cuda", dtype=torch.bfloat16), None,
                      v_valid=v_valid, lowrank=(W, A, Bm))
    hidden = normal(T, d, std=1.0)
    hidden[3, 5] = float("nan")
    hidden[190, 0] = float("inf")
    vv = v_valid or v
    targets = torch.randint(0, vv, (T, n), device="cuda", generator=g, dtype=torch.int32)
    out = torch.empty(T, device="cuda")
    head.mtpc_window_logprob(hidden, targets, out)
    h = hidden.double()
    corr = (h @ Bm[0].double().transpose(-1, -2)) @ A[0].double().transpose(-1, -2)                     # [r, T, v]
    logits = (h @ W[0].double().T + corr)[..., :vv]
    want = torch.logsumexp(torch.log_softmax(logits, -1).gather(2, targets.long().expand(r, T, 1))[..., 0], 0) - torch.log(torch.tensor(float(r)))
    good = torch.ones(T, dtype=torch.bool, device="cuda")
    good[3] = good[190] = False
    assert torch.isnan(out[~good]).all() and torch.isfinite(out[good]).all()
    tol = 2e-3 + 2.0 ** -16 * (h.abs() @ Bm[0].double().abs().transpose(-1, -2) @ A[0].double().abs().transpose(-1, -2)).amax((0, 2))
    assert ((out.double() - want).abs() <= tol)[good].all()
