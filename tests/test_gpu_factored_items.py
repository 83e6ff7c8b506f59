"""Training calls of a factored head where the gradient kernel's items and rounds are cut: one component (its copy has no weight) at
either rank, two, and several rounds of eight; a last block of 16 columns; position groups of 32 with one row and without any. Bars of
test_gpu_lowrank (two bf16-rounded factors per product)."""
import pytest

import test_gpu_lowrank as lowrank
from paper_2511_11346_b200 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("family,n,r,v,vv,d,k,T", [
    (I.CP, 2, 1, 80, 0, 64, 32, 33), (I.CP, 2, 2, 144, 0, 64, 16, 65), (I.HMM, 3, 16, 80, 76, 64, 16, 129), (I.HMM, 2, 32, 64, 0, 64, 32, 31),
    (I.CP, 2, 64, 16, 0, 64, 16, 40),
])
def test_gradients_at_the_edges_of_items_and_rounds(family, n, r, v, vv, d, k, T):
    lowrank.test_factored_backward_is_the_chain_rule_through_the_composition(family, n, r, v, vv, d, k, T)
