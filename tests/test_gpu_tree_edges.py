"""The tree walk where the codes are dealt to another number of CTAs and the last part is not full."""
import pytest

import test_gpu_decide as D
from vvs_synth.configs import MODE_RELAXED, MODE_STRICT

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode,nbr_k,delta,adjusted", [(MODE_STRICT, 1, float("inf"), False), (MODE_RELAXED, 24, 0.2, True)])
@pytest.mark.parametrize("v", [4095, 8193, 16385])
def test_tree_walk_parts(v, mode, nbr_k, delta, adjusted):
    D.test_tree_walk_is_exact_on_random_trees(v, 16, 20, 1, 1.0, 2.5, 0, mode, nbr_k, delta, adjusted)
