"""Heads of so many weight rows that a CTA of the few-position weight pass has seven and more tiles: passes of two (ten tiles, d >= 2048), the
shorter ring, last passes of one and of two tiles, sum units' tiles among them. Bit for bit what the same positions draw in a batch of
more than 32, which takes the general passes, and the prefix marginals are those that the evaluation's projection gives the
drafted bytes: fp32 sums of the same bf16 products in another order, of at most a few units each: 1e-4."""
import pytest
import torch

from paper_2511_11346_b200 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("family,ctx,n,r,v,d", [
    (B.MTPC_CP, False, 16, 32, 320, 2048),        # 10 tiles of 112 rows
    (B.MTPC_CP, False, 16, 32, 320, 192),         # the same, K too short for passes of two
    (B.MTPC_HMM, True, 16, 32, 272, 64),          # 11 of 96, one K block
    (B.MTPC_BTREE, False, 16, 32, 256, 128),      # 9 of 112
    (B.MTPC_CP, False, 16, 64, 320, 128),         # 31 of 72
    (B.MTPC_HMM, False, 16, 32, 256, 320),        # 7 of 128
])
def test_long_runs_of_tiles(family, ctx, n, r, v, d):
    P = 40
    g = torch.Generator(device="cuda")
    g.manual_seed(n * r + d)

    def normal(*shape, std):
        return torch.empty(shape, device="cuda", dtype=torch.bfloat16).normal_(0.0, std, generator=g)

    sums = 1 + (n - 1) * r if ctx else 1 + (n - 2) * r if family == B.MTPC_BTREE else 1
    trans = torch.randn(n - 1, r, r, device="cuda", generator=g) if family == B.MTPC_HMM else None
    head = B.MtpcHead(family, n, r, v, d, B.MTPC_BF16, P, 1, normal(n, r, v, d, std=d ** -0.5), normal(sums * r, d, std=d ** -0.5), trans,
                      flags=B.MTPC_FLAG_HMM_CONTEXTUAL if ctx else 0)
    hidden, uniforms = normal(P, d, std=1.0), torch.rand(P, 2 * n, device="cuda", generator=g)

    def draft(p):
        out, prefix = torch.empty(p, n, dtype=torch.int32, device="cuda"), torch.empty(p, n, device="cuda")
        head.mtpc_draft_sample_prefix(hidden[:p].contiguous(), 1, uniforms[:p].contiguous(), out, prefix)
        return out, prefix

    want = draft(P)
    for p in (1, 16, 17, 32):
        for a, b in zip(draft(p), want):
            assert torch.equal(a, b[:p]), p
    again = torch.empty(P, n, device="cuda")
    head.mtpc_window_prefix_logprob(hidden, want[0], again)
    assert head.mtpc_get_status() == 0
    assert ((want[0] >= 0) & (want[0] < v)).all() and (again - want[1]).abs().max() <= 1e-4
    head.mtpc_destroy()
