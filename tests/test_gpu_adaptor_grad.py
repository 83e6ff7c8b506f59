"""Gradients through the adaptors from one reading of the logit gradients, which heads of many units use: held to the oracle's
chain rule with the bars of tests/test_gpu_lowrank.py (derived there from the magnitudes behind every entry). One unit's symbols fill
an odd and an even number of 64-symbol boxes, one box only, and the most there can be; positions one past a tile of 128, one alone,
and a whole tile; more units than SMs; ranks 16 and 32."""
import pytest
import test_gpu_lowrank

from paper_2511_11346_b200 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("family,n,r,v,vv,d,k,T", [
    (I.CP, 2, 64, 320, 0, 64, 16, 140),
    (I.HMM, 5, 16, 272, 261, 64, 32, 129),
    (I.BTREE, 8, 32, 16, 0, 64, 16, 1),
    (I.CP, 2, 64, 512, 0, 64, 32, 128),
    (I.CP, 3, 128, 176, 0, 64, 16, 30),
])
def test_one_reading_of_the_logit_gradients(family, n, r, v, vv, d, k, T):
    test_gpu_lowrank.test_factored_backward_is_the_chain_rule_through_the_composition(family, n, r, v, vv, d, k, T)
