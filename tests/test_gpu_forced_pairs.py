"""The build of the projection kernel that a caller asks for is the one that runs, also for the sum units of a factored head, which are a launch of
few columns that lone CTAs take by default; and both give the same bits."""
import pytest
import torch

from paper_2511_11346_b200 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("family,r", [(B.MTPC_CP, 8), (B.MTPC_CP, 32), (B.MTPC_BTREE, 16)])    # 16, 32 and several tiles of 256 columns
def test_sum_units_of_a_factored_head(family, r):
    n, v, d, k, T = 4, 64, 256, 16, 300
    g = torch.Generator(device="cuda")
    g.manual_seed(5)

    def normal(*shape, std):
        return torch.empty(shape, device="cuda", dtype=torch.bfloat16).normal_(0.0, std, generator=g)

    sums = 1 + (n - 2) * r if family == B.MTPC_BTREE else 1
    head = B.MtpcHead(family, n, r, v, d, B.MTPC_BF16, T, 1, None, normal(sums * r, d, std=0.1),
                      lowrank=(normal(n, v, d, std=0.1), normal(n, r, v, k, std=0.2), normal(n, r, k, d, std=0.05)))
    hidden = normal(T, d, std=1.0)
    targets = torch.randint(0, v, (T, n), device="cuda", generator=g, dtype=torch.int32)
    got = []
    for variant in (1, 2):
        head.mtpc_debug_set_projection_variant(variant)
        out = torch.empty(T, device="cuda")
        head.mtpc_window_logprob(hidden, targets, out)
        with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CUDA], acc_events=True) as trace:
            head.mtpc_window_logprob(hidden, targets, out)
            torch.cuda.synchronize()
        names = [e.name for e in trace.events() if "mtpc_gemm_kernel" in e.name]
        if not names and not any("circuit" in e.name for e in trace.events()):
            pytest.skip("no kernel records from the profiler")
        assert len(names) == 1 and f"<0, {variant}," in names[0], names
        got.append(out)
    assert torch.equal(*got)
    assert head.mtpc_get_status() == 0
    head.mtpc_destroy()
