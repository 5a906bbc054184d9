"""The folded step where a projection's weights are beyond what stays in L2: matrices of 20 to 64 MB (passes of up to 64 tokens)
and of more (one pass of up to 128, above that passes side by side), with a last tile and a last k-block that are not full."""
from dataclasses import replace

import pytest

import helpers as H
from test_gpu_verify import _check_end_to_end
from vvs_synth.configs import B7

pytestmark = pytest.mark.gpu

# QKV 25 MB; gate/up 136 MB and down 68 MB, 130 tiles and 8 rows, 260 k-blocks and 8 columns
LARGE = replace(B7, name="large", n_layers=1, d_model=2048, n_heads=16, d_ff=16648, vocab=1096, vocab_offset=64, lm_rows=2048,
                tok_rows=0, s_max=160)


@pytest.fixture(scope="module")
def weights():
    return H.gen.make_weights(LARGE, 2600)


@pytest.mark.parametrize("n_images,n_forced,k", [
    (4, 1, 8),         # 72 tokens
    (11, 1, 5),        # 132 tokens: three passes, the last not full
    (13, 2, 12)])      # 364 tokens: six passes
def test_large_projections(weights, n_images, n_forced, k):
    fills = [(37 * i) % (LARGE.s_max - n_forced - k) for i in range(n_images)]
    case = H.build_case_independent(LARGE, 2600 + k, n_images, 2, n_forced, k, fills, logit_std=0.6, w=weights)
    run = H.GpuRunner(LARGE, weights, 2 * n_images, n_forced + k)
    _check_end_to_end(case, run.verify(case), H.run_oracle(case))
    run.close()
