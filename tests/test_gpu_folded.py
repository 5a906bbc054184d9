"""The folded-epilogue step of wide models (d_model >= 1024) on two layers: every split of the K range, one and several
token passes, quads and row parts that are not full, both head sizes, chains and trees, against the oracle."""
from dataclasses import replace

import numpy as np
import pytest

import helpers as H
from test_gpu_tree import _check_tree
from test_gpu_verify import _check_end_to_end
from vvs_synth.configs import B7, XL

pytestmark = pytest.mark.gpu

# 1096 codes; 2744 = 21 weight tiles and 56 rows; 24 and 16 k-blocks
WIDE64 = replace(XL, name="wide64", n_layers=2, d_model=1536, n_heads=24, d_ff=2744, vocab=1096, lm_rows=0, tok_rows=0, s_max=208)
WIDE128 = replace(B7, name="wide128", n_layers=2, d_model=1024, n_heads=8, d_ff=1368, vocab=1096, vocab_offset=64, lm_rows=2048,
                  tok_rows=0, s_max=700)


@pytest.mark.parametrize("ms,n_images,n_cfg,n_forced,k,fills", [
    (WIDE64, 1, 1, 1, 1, [1]),                            # 2 tokens
    (WIDE64, 1, 2, 1, 8, [199]),                          # 18 tokens, a cache the block fills exactly
    (WIDE64, 1, 2, 6, 8, [16]),                           # 28 tokens
    (WIDE64, 3, 2, 2, 15, [0, 47, 150]),                  # 102 tokens, 17 rows per sequence, an empty cache
    (WIDE64, 16, 2, 1, 9, list(range(3, 195, 12))),       # 320 tokens: several passes
    (WIDE128, 1, 2, 1, 4, [513]),                         # keys of a head over a cluster
    (WIDE128, 5, 1, 3, 20, [5, 160, 333, 64, 677]),       # 115 tokens, 23 rows per sequence
    (WIDE64, 7, 2, 2, 15, [3, 20, 37, 90, 111, 144, 170]),   # more (sequence, head) items than CTAs, 17 rows per sequence
    (WIDE128, 19, 2, 1, 2, list(range(1, 96, 5)))])       # the same, heads of 128
def test_folded_step(ms, n_images, n_cfg, n_forced, k, fills):
    case = H.build_case_independent(ms, 1700 + k, n_images, n_cfg, n_forced, k, fills, logit_std=0.6)
    run = H.GpuRunner(ms, case["w"], n_images * n_cfg, n_forced + k)
    gpu = run.verify(case)
    _check_end_to_end(case, gpu, H.run_oracle(case))
    again = run.verify(case)
    for key in ("accept_len", "next_token", "target_probs", "hidden", "kv_k", "kv_v"):
        np.testing.assert_array_equal(gpu[key], again[key], err_msg=key)
    run.close()


@pytest.mark.parametrize("ms,n_images,parent,fills", [
    (WIDE64, 1, [-1, 0, 0, 1, 1, 2, 3, 3, 6], [77]),
    (WIDE128, 2, [-1, 0, 0, 0, 1, 2, 2, 4, 4, 5, 6, 7, 8, 8, 9, 10, 11, 12, 12], [130, 15])])
def test_folded_tree(ms, n_images, parent, fills):
    case = H.build_tree_case(ms, 1800 + n_images, n_images, 2, 1, parent, fills, q_noise=0.7)
    run = H.GpuRunner(ms, case["w"], 2 * n_images, len(parent))
    _check_tree(case, H.run_tree_gpu(run, case), H.run_tree_oracle(case))
    run.close()
