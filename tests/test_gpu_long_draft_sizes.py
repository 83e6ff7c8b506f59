"""Drafts of more than 128 positions: the latent draws ask for shared memory by the number of windows, so that the SMs share their CTAs of four windows
evenly. Batches at the edges of one, two and sixteen CTAs an SM, and beyond; a window's draws do not depend on the batch, so the first
windows of every batch are bit for bit those of the smallest."""
import json

import pytest
import torch

from paper_2511_11346_b200 import binding as B

pytestmark = pytest.mark.gpu


def _sms():
    return torch.cuda.get_device_properties(0).multi_processor_count


def _head(family, T):
    n, r, v, d = 4, 8, 32, 64
    g = torch.Generator(device="cuda")
    g.manual_seed(11)

    def normal(*shape, std):
        return torch.empty(shape, device="cuda", dtype=torch.bfloat16).normal_(0.0, std, generator=g)

    sums = 1 + (n - 2) * r if family == B.MTPC_BTREE else 1
    trans = torch.randn(n - 1, r, r, device="cuda", generator=g) if family == B.MTPC_HMM else None
    head = B.MtpcHead(family, n, r, v, d, B.MTPC_BF16, T, 1, normal(n, r, v, d, std=0.3), normal(sums * r, d, std=0.2), trans)
    return head, normal(T, d, std=1.0), torch.rand(T, 2 * n, device="cuda", generator=g)


@pytest.mark.parametrize("family", [B.MTPC_CP, B.MTPC_HMM, B.MTPC_BTREE])
def test_first_windows(family):
    n, v, sms = 4, 32, _sms()
    sizes = [129, 4 * sms, 4 * sms + 1, 8 * sms, 8 * sms + 3, 64 * sms, 64 * sms + 1]
    head, hidden, uniforms = _head(family, sizes[-1])

    def draft(t):
        out, prefix = torch.empty(t, n, dtype=torch.int32, device="cuda"), torch.empty(t, n, device="cuda")
        head.mtpc_draft_sample_prefix(hidden[:t].contiguous(), 1, uniforms[:t].contiguous(), out, prefix)
        return out, prefix

    want = draft(sizes[-1])
    assert ((want[0] >= 0) & (want[0] < v)).all() and torch.isfinite(want[1]).all()
    for t in sizes[:-1]:
        out, prefix = draft(t)
        assert torch.equal(out, want[0][:t]) and torch.equal(prefix, want[1][:t])
    assert head.mtpc_get_status() == 0
    head.mtpc_destroy()


@pytest.mark.parametrize("per_sm", [1, 2, 5, 16])
def test_no_sm_takes_more_than_its_share(per_sm, tmp_path):
    """What the launch asks for leaves no room for one CTA more than the share, in the 228 KB of an SM of which every CTA takes another 1 KB (or, at
    sixteen CTAs of 128 threads, none beside an SM's 2048 threads)."""
    T = per_sm * 4 * _sms()
    head, hidden, uniforms = _head(B.MTPC_BTREE, T)
    out, prefix = torch.empty(T, 4, dtype=torch.int32, device="cuda"), torch.empty(T, 4, device="cuda")
    head.mtpc_draft_sample_prefix(hidden, 1, uniforms, out, prefix)
    with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CUDA], acc_events=True) as trace:
        head.mtpc_draft_sample_prefix(hidden, 1, uniforms, out, prefix)
        torch.cuda.synchronize()
    path = tmp_path / "trace.json"
    trace.export_chrome_trace(str(path))
    kernels = [e for e in json.loads(path.read_text())["traceEvents"] if e.get("cat") == "kernel"]
    if not kernels:
        pytest.skip("no kernel records from the profiler")
    (draws,) = [e["args"] for e in kernels if "latent_sample_kernel" in e["name"]]
    assert draws["grid"][0] == per_sm * _sms()
    assert per_sm * (draws["shared memory"] + 1024) <= 228 * 1024
    assert (per_sm + 1) * (draws["shared memory"] + 1024) > 228 * 1024 or (per_sm + 1) * 128 > 2048
    head.mtpc_destroy()
