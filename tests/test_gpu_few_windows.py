"""Launch shapes that depend on how many windows a call has: the HMM's circuit gives a CTA eight windows, or four or two where they are few.
A window's arithmetic does not depend on it, so its results are bit for bit those that it has in a call of another size."""
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
