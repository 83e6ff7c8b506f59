"""How the projection's work items are dealt out: the workers without an emission item in the last round take the sum tiles, up to
an emission item's worth, and the rest is spread over all. Every sum unit and every input unit enters the log-marginals, so an item
left out or taken by two accumulator owners shows up against the oracle (bar 2e-3, as everywhere; the weights' spread makes the
marginals of one window differ by whole nats)."""
import numpy as np
import pytest

from oracle import mtpc_oracle as orc
from paper_2511_11346_b200 import inputs as I
from paper_2511_11346_b200.runner import DeviceHead

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("family,n,r,v,d,T,variant", [
    (I.BTREE, 8, 32, 16, 64, 300, 1),       # 28 sum tiles a row of tiles, few emission items: sums beyond the idle workers' room
    (I.BTREE, 8, 32, 256, 64, 150, 1),      # a last round with room for every sum tile
    (I.HMM_CTX, 5, 32, 272, 64, 513, 2),    # pairs; units that straddle tiles
    (I.HMM, 4, 32, 256, 64, 1200, 1),       # several rounds of emission items, a few sum tiles
    (I.CP, 2, 4, 16, 64, 40, 0),            # fewer items than SMs
])
def test_every_item_is_taken_once(family, n, r, v, d, T, variant):
    wl = I.make_workload("items", I.HeadShape(family, n, r, v, d), T, seed=8800 + n + r + v, weight_std=0.25)
    dh = DeviceHead(wl)
    dh.head.mtpc_debug_set_projection_variant(variant)
    for _ in range(2):
        got = dh.window_logprob().cpu().numpy()
        assert dh.head.mtpc_get_status() == 0
        want = orc.window_logprob(family, wl.hidden_q, wl.W_emit_q, wl.W_sum_q, wl.T_static, wl.targets)
        assert np.abs(got - want).max() <= 2e-3
    dh.close()
