"""The LM head at the edges of its kernels for few and for many feature rows: one k-block, rings that are used once and again,
48 guided rows (96 feature rows, the most of the one) and 49, tiles that are not full, more tiles than SMs."""
import numpy as np
import pytest

import helpers as H
from oracle import vvs_oracle as O
from test_gpu_epilogue_fcache import _epilogue_case, _run_epilogue
from vvs_synth.configs import MODE_STRICT

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,v,n_images,n_cfg,k", [(64, 130, 1, 1, 1), (704, 385, 3, 2, 15), (1096, 1000, 5, 2, 8), (832, 257, 3, 1, 31),
                                                  (840, 19080, 2, 2, 4), (328, 700, 7, 2, 6)])
def test_lmhead_edges(d, v, n_images, n_cfg, k):
    case = _epilogue_case(d, v, n_images, n_cfg, k, k + 1, 0, MODE_STRICT, 1, float("inf"), seed=d + v)
    gpu = _run_epilogue(case)
    ora = O.epilogue(case["ms"], case["w"], case["hidden_in"], case["drafts"], case["n_draft"], 1, case["draft_probs"],
                     case["uniforms"], n_cfg, case["cfg_scale"], case["temperature"], MODE_STRICT, None, None, 1, float("inf"))
    assert gpu["status"] == 0
    np.testing.assert_allclose(gpu["target_probs"], ora["target_probs"], rtol=6e-2, atol=2e-4)
    H.check_replay(case, gpu)


@pytest.mark.parametrize("d,v,n_images,n_cfg,k", [(64, 300, 69, 2, 12), (200, 129, 10, 2, 12), (72, 4100, 20, 1, 12)])
def test_lmhead_pair_chunks(d, v, n_images, n_cfg, k):
    """Passes whose last is one decision row (897 in eight of 128: most epilogue groups have none), 50 (130 in two of 80), 100 of 160."""
    test_lmhead_edges(d, v, n_images, n_cfg, k)
