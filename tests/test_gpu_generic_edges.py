"""The float32 step where a row product's pieces are not full: d_ff and vocabularies that are no multiple of a warp's piece,
one to seventeen activation rows, one and many columns left over."""
from dataclasses import replace

import pytest

import helpers as H
from test_gpu_verify import _check_end_to_end
from vvs_synth.configs import TINY

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,heads,ff,vocab,n_images,n_cfg,k,fills", [
    (64, 1, 72, 33, 1, 1, 1, [0]), (192, 3, 200, 130, 1, 1, 6, [1]), (256, 4, 1032, 515, 1, 1, 7, [100]),
    (320, 5, 8, 66, 2, 2, 3, [17, 90])])
def test_float32_step_edges(d, heads, ff, vocab, n_images, n_cfg, k, fills):
    ms = replace(TINY, name=f"tiny{d}", d_model=d, n_heads=heads, d_ff=ff, vocab=vocab, lm_rows=0, tok_rows=0)
    case = H.build_case_independent(ms, 900 + d, n_images, n_cfg, 1, k, fills, logit_std=0.6)
    run = H.GpuRunner(ms, case["w"], n_images * n_cfg, 1 + k)
    _check_end_to_end(case, run.verify(case), H.run_oracle(case))
    run.close()
