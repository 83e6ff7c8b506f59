"""Pieces of a host-buffer call: growing ones where the kernels take longer than the link, shrinking ones where the link does, one
piece, and a remainder that joins the last piece. The arithmetic per position is the device-buffer call's, so the results are
equal bit for bit."""
import pytest
import torch

from paper_2511_11346_b200 import inputs as I
from paper_2511_11346_b200.runner import DeviceHead

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("family,n,r,v,d,T,io", [
    (I.CP, 2, 2, 16, 64, 3000, I.F32),       # the link bounds it: the last piece is the smallest
    (I.CP, 8, 32, 512, 64, 2500, I.BF16),    # the kernels do
    (I.BTREE, 4, 4, 64, 64, 767, I.BF16),    # 512 and a remainder below half of it
    (I.HMM, 3, 8, 32, 128, 769, I.BF16),
    (I.CP, 2, 4, 32, 64, 1, I.BF16),
])
def test_host_call_in_pieces_equals_the_device_call(family, n, r, v, d, T, io):
    wl = I.make_workload("pieces", I.HeadShape(family, n, r, v, d, io_dtype=io), T, seed=600 + T, weight_std=0.2)
    dh = DeviceHead(wl)
    dev = dh.window_logprob().cpu()
    for _ in range(2):
        out = torch.full((T,), 7.0).pin_memory()
        dh.head.mtpc_window_logprob_host(dh.hidden_host(), torch.from_numpy(wl.targets).pin_memory(), out)
        assert torch.equal(out, dev)
    assert dh.head.mtpc_get_status() == 0
    dh.close()
