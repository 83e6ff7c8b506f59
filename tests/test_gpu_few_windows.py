"""Launch shapes that depend on how many windows a call has: the HMM's circuit gives a CTA eight windows, or four or two where they are few, and
the per-slot draws of many (position, slot) pairs take a build of which three CTAs share an SM. A window's arithmetic does not depend on
either, so its results are bit for bit those that it has in a call of another size."""
import pytest
import torch

from paper_2511_11346_b200 import binding as B

pytestmark = pytest.mark.gpu


def _head(family, n, r, v, d, positions, wpp, v_valid=0):
    g = torch.Generator(device="cuda")
    g.manual_seed(n * r + v)

    def normal(*shape, std):
        return torch.empty(shape, device="cuda", dtype=torch.bfloat16).normal_(0.0, std, generator=g)

    sums = 1 + (n - 2) * r if family == B.MTPC_BTREE else 1
    trans = torch.randn(n - 1, r, r, device="cuda", generator=g) if family == B.MTPC_HMM else None
    head = B.MtpcHead(family, n, r, v, d, B.MTPC_BF16, positions, wpp, normal(n, r, v, d, std=2 * d ** -0.5), normal(sums * r, d, std=d ** -0.5),
                      trans, v_valid=v_valid)
    return head, normal(positions, d, std=1.0), g


@pytest.mark.parametrize("n,r", [(5, 32), (16, 16), (2, 16), (64, 32)])       # (64 x 32: tables in chunks)
def test_windows_per_cta(n, r):
    T = 1300
    head, hidden, g = _head(B.MTPC_HMM, n, r, 16, 64, T, 1)
    targets = torch.randint(0, 16, (T, n), device="cuda", generator=g, dtype=torch.int32)
    targets[7, -1] = -1

    def run(t):
        joint, prefix = torch.empty(t, device="cuda"), torch.empty(t, n, device="cuda")
        head.mtpc_window_logprob(hidden[:t].contiguous(), targets[:t].contiguous(), joint)
        head.mtpc_window_prefix_logprob(hidden[:t].contiguous(), targets[:t].contiguous(), prefix)
        return joint, prefix

    want = run(T)                                    # eight windows a CTA
    assert torch.isfinite(want[1]).all()
    for t in (1, 2, 3, 295, 296, 297, 591, 592, 593):     # two, four and eight on 148 SMs
        joint, prefix = run(t)
        assert torch.equal(joint, want[0][:t]) and torch.equal(prefix, want[1][:t])
    assert head.mtpc_get_status() == 0


@pytest.mark.parametrize("family,n,r,v,v_valid,wpp", [
    (B.MTPC_CP, 16, 16, 320, 0, 16), (B.MTPC_CP, 8, 64, 112, 0, 1), (B.MTPC_BTREE, 8, 32, 256, 0, 3), (B.MTPC_HMM, 16, 32, 272, 268, 2),
    (B.MTPC_CP, 16, 8, 400, 0, 4)])
def test_draws_of_many_slots(family, n, r, v, v_valid, wpp):
    P = 100                                          # n P > 2 x 148
    few = 148 // n
    head, hidden, g = _head(family, n, r, v, 64, P, wpp, v_valid)
    uniforms = torch.rand(P * wpp, 2 * n, device="cuda", generator=g)
    uniforms[5, n] = 1.0                             # one refused draw

    def draft(p):
        out, prefix = torch.empty(p * wpp, n, dtype=torch.int32, device="cuda"), torch.empty(p * wpp, n, device="cuda")
        head.mtpc_draft_sample_prefix(hidden[:p].contiguous(), wpp, uniforms[:p * wpp].contiguous(), out, prefix)
        return out, prefix

    many, some = draft(P), draft(few)
    assert torch.equal(some[0], many[0][:few * wpp]) and torch.equal(some[1].nan_to_num(1.0), many[1][:few * wpp].nan_to_num(1.0))
    assert (many[0] < 0).sum() == 1 and many[0][5, 0] == -1 and (many[0] < (v_valid or v)).all()
