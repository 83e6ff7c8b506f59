"""Calls that follow one another without a pause. The kernels of a call, and the first kernel of the next one, are scheduled before
the kernel ahead has finished and wait for it on the device; the kernels that hand out windows through a counter rely on the
projection (or the per-slot kernel) before them to zero it. So back-to-back calls on alternating inputs must give, bit for bit, what
each call gives alone on an idle device. (fp32 heads: the gradient of a static transition table is summed by atomics and is left
out.) d = 1600 runs the projection in CTA pairs, d < 1536 in single CTAs; an fp32 hidden state at an odd multiple of four bytes
takes the scalar conversion, an aligned one the 16-byte conversion."""
import pytest
import torch

from paper_2511_11346_b200 import inputs as I
from paper_2511_11346_b200.runner import DeviceHead

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("family,n,r,v,d,T,dtype", [
    (I.BTREE, 8, 16, 64, 128, 150, "f32"),
    (I.BTREE, 4, 8, 48, 1600, 300, "bf16"),
    (I.HMM, 5, 8, 64, 1024, 257, "f32"),
    (I.CP, 3, 8, 320, 64, 200, "f32"),
])
def test_back_to_back_calls_equal_isolated_ones(family, n, r, v, d, T, dtype):
    shape = I.HeadShape(family, n, r, v, d, io_dtype=I.F32 if dtype == "f32" else I.BF16)
    wl = I.make_workload("chain", shape, T, seed=41, wpp=2, weight_std=0.25)
    dh = DeviceHead(wl)
    torch.manual_seed(7)
    hidden = [dh.hidden_device()]
    hidden.append(torch.randn_like(hidden[0]))
    targets = [torch.from_numpy(wl.targets).cuda(), torch.randint(v, (T, n), dtype=torch.int32, device="cuda")]
    if dtype == "f32":                                   # the same values, four bytes off a 16-byte boundary
        room = torch.empty(hidden[1].numel() + 1, dtype=torch.float32, device="cuda")
        hidden[1] = room[1:].view_as(hidden[1]).copy_(hidden[1])
    head = dh.head
    uniforms = torch.rand(2 * T, 2 * n, device="cuda")
    weight = torch.full((T,), -1.0 / T, device="cuda")

    def calls(i, small):
        P = 3 if small else T
        out = {k: torch.empty(T, device="cuda") for k in ("lp", "blp")}
        out["pre"] = torch.empty(T, n, device="cuda")
        out["bytes"] = torch.empty(2 * P, n, dtype=torch.int32, device="cuda")
        out["dlp"] = torch.empty(2 * P, device="cuda")
        g = {k: torch.empty(s, device="cuda") for k, s in
             (("dh", (T, d)), ("dWe", (n, r, v, d)), ("dWs", tuple(dh.W_sum.shape)))}
        dT = torch.empty(max(n - 1, 1), r, r, device="cuda") if family == I.HMM else None
        steps = [lambda: head.mtpc_window_logprob(hidden[i], targets[i], out["lp"]),
                 lambda: head.mtpc_draft_sample(hidden[i][:P], 2, uniforms[:2 * P], out["bytes"], out["dlp"]),
                 lambda: head.mtpc_window_logprob_backward(hidden[i], targets[i], weight, out["blp"], g["dh"], g["dWe"], g["dWs"], dT),
                 lambda: head.mtpc_window_prefix_logprob(hidden[i], targets[i], out["pre"])]
        return steps, {**out, **g}

    def run(alone):
        results = []
        for i, small in ((0, True), (1, False), (0, False), (1, True)):
            steps, out = calls(i, small)
            for step in steps:
                if alone:
                    torch.cuda.synchronize()
                step()
            results.append(out)
        torch.cuda.synchronize()
        return results

    for a, b in zip(run(alone=True), run(alone=False)):
        for k in a:
            assert torch.equal(a[k], b[k]), k
            assert not a[k].is_floating_point() or torch.isfinite(a[k]).all(), k
    assert head.mtpc_get_status() == 0
    dh.close()


@pytest.mark.parametrize("n,r,v,d,T,P,wpp,dtype", [
    (8, 16, 64, 128, 150, 6, 8, "bf16"), (3, 32, 48, 64, 40, 1, 1, "bf16"), (5, 4, 32, 1600, 300, 9, 16, "f32"),
])
def test_parameters_updated_between_calls(n, r, v, d, T, P, wpp, dtype):
    """Static transition tables are copied to shared memory before a kernel waits for the one ahead of it (the per-slot kernel of a
    short draft, the circuit). That is sound because the kernel that writes them is launched plainly and the first kernel of
    every call waits before it lets the next one start. Updates with alternating tables right before the calls must therefore give what
    they give with the device idle in between, in one launch for a bf16 head."""
    wl = I.make_workload("update", I.HeadShape(I.HMM, n, r, v, d, io_dtype=I.F32 if dtype == "f32" else I.BF16), T, seed=53, wpp=wpp,
                         weight_std=0.25)
    dh = DeviceHead(wl)
    hidden, targets = dh.hidden_device(), torch.from_numpy(wl.targets).cuda()
    tables = [dh.T_static, 3.0 * torch.flip(dh.T_static, dims=(2,)).contiguous()]
    u = torch.from_numpy(wl.uniforms).cuda()[:P * wpp].contiguous()
    few = hidden[:P].contiguous()

    def run(alone):
        got = []
        for i in range(6):
            before = dh.head.mtpc_launch_count()
            dh.head.mtpc_update_parameters(dh.W_emit, dh.W_sum, tables[i % 2])
            assert dh.head.mtpc_launch_count() - before == (1 if dtype == "bf16" else 3)
            for call in (lambda: (dh.window_prefix_logprob(hidden=hidden, targets=targets),),
                         lambda: dh.draft_sample_prefix(wpp, hidden=few, uniforms=u)) if i % 3 else (
                         lambda: dh.draft_sample_prefix(wpp, hidden=few, uniforms=u),
                         lambda: (dh.window_logprob(hidden=hidden, targets=targets),)):
                if alone:
                    torch.cuda.synchronize()
                got += call()
        torch.cuda.synchronize()
        return got

    want, got = run(alone=True), run(alone=False)
    assert dh.head.mtpc_get_status() == 0
    for a, b in zip(want, got):
        assert torch.equal(a, b)
    per = len(want) // 6
    assert not torch.equal(want[per], want[2 * per])       # the tables matter
    dh.close()


@pytest.mark.parametrize("family,n,r,v,d,N,L,dtype,rank", [
    (I.HMM, 6, 32, 64, 128, 4, 500, "bf16", 0), (I.HMM, 4, 8, 48, 1600, 3, 100, "f32", 0), (I.BTREE, 8, 16, 64, 128, 2, 400, "bf16", 0),
    (I.CP, 3, 8, 320, 64, 5, 60, "f32", 0), (I.HMM, 6, 32, 64, 128, 4, 500, "bf16", 16), (I.CP, 2, 64, 80, 64, 2, 90, "bf16", 32),
])
def test_training_calls_follow_one_another(family, n, r, v, d, N, L, dtype, rank):
    """Training calls of the loss over overlapping windows. Three of their kernels work before they wait: the static HMM's sweep copies its
    tables, the coefficients are formed from the targets, the loss from the prefixes. What they read and write so early must be the work of
    kernels that have ended, and nobody's any more. On inputs that alternate, and static tables updated right before, each call must give what it
    gives on an idle device, bit for bit (the gradient of a static table, added up by atomics: 1e-5 of its largest entry)."""
    T = N * L
    wl = I.make_workload("train_chain", I.HeadShape(family, n, r, v, d, io_dtype=I.F32 if dtype == "f32" else I.BF16), T, seed=67 + rank, weight_std=0.25)
    lowrank = I.lowrank_parameters(n, r, v, d, rank, seed=68, weight_std=0.2, adaptor_std=0.1) if rank else None
    dh = DeviceHead(wl, lowrank=lowrank) if rank else DeviceHead(wl)
    torch.manual_seed(11)
    hidden = [dh.hidden_device()]
    hidden.append(torch.randn_like(hidden[0]))
    targets = [torch.from_numpy(wl.targets).cuda(), torch.randint(v, (T, n), dtype=torch.int32, device="cuda")]
    targets[1][::3, n - 1] = -1
    static = family == I.HMM
    tables = [dh.T_static, 3.0 * torch.flip(dh.T_static, dims=(2,)).contiguous()] if static else None
    shapes = dict(W_base=(n, v, d), A=(n, r, v, rank), B=(n, r, rank, d)) if rank else dict(W_emit=(n, r, v, d))

    def run(alone):
        got = []
        for i in range(6):
            out = {k: torch.full(s, 7.0, device="cuda") for k, s in
                   dict(slot=(n,), loss=(1,), dh=(T, d), **shapes, W_sum=tuple(dh.W_sum.shape)).items()}
            if static:
                out["T_static"] = torch.full((n - 1, r, r), 7.0, device="cuda")
                if not rank:
                    dh.head.mtpc_update_parameters(dh.W_emit, dh.W_sum, tables[(i // 2) % 2])
            if alone:
                torch.cuda.synchronize()
            call = dh.head.mtpc_lowrank_window_loss_backward if rank else dh.head.mtpc_window_loss_backward
            call(hidden[i % 2], targets[(i // 3) % 2], N, L, 0.9, *[out[k] for k in ("slot", "loss", "dh", *shapes, "W_sum")], out.get("T_static"))
            got.append(out)
        torch.cuda.synchronize()
        return got

    want, got = run(alone=True), run(alone=False)
    assert dh.head.mtpc_get_status() == 0
    for a, b in zip(want, got):
        for k in a:
            assert torch.isfinite(a[k]).all(), k
            if k == "T_static":
                assert (a[k] - b[k]).abs().max() <= 1e-5 * a[k].abs().max()
            else:
                assert torch.equal(a[k], b[k]), k
    assert not torch.equal(want[0]["slot"], want[1]["slot"]) and not torch.equal(want[2]["slot"], want[3]["slot"])
    dh.close()
