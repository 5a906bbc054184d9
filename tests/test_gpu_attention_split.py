"""Heads of 64 whose keys a cluster of CTAs shares (few items, a cache of 1536 slots or more): two and four CTAs, up to 16 and
more rows per sequence, an empty cache, one slice, a last slice that is not full, a cache the block fills exactly."""
from dataclasses import replace

import numpy as np
import pytest

import helpers as H
from test_gpu_verify import _check_end_to_end
from vvs_synth.configs import XL

pytestmark = pytest.mark.gpu

LONG = replace(XL, name="long64", n_layers=2, d_model=1024, n_heads=16, d_ff=1368, vocab=1096, lm_rows=0, tok_rows=0, s_max=1541,
               rope_grid_w=40)


@pytest.mark.parametrize("s_max,n_images,n_cfg,n_forced,k,fills", [
    (1541, 2, 2, 1, 8, [0, 1532]),          # 64 items, two CTAs each
    (1541, 1, 2, 2, 20, [1000]),            # more than 16 rows: two groups of warps
    (3079, 1, 1, 1, 8, [3070]),             # 16 items, four CTAs each
    (3079, 1, 2, 1, 8, [17]),               # 32 items; ranks without a slice of their own
    (3079, 2, 1, 3, 22, [2500, 257])])
def test_heads_of_64_over_a_cluster(s_max, n_images, n_cfg, n_forced, k, fills):
    ms = replace(LONG, s_max=s_max)
    case = H.build_case_independent(ms, 2700 + k + s_max, n_images, n_cfg, n_forced, k, fills, logit_std=0.6)
    run = H.GpuRunner(ms, case["w"], n_images * n_cfg, n_forced + k)
    gpu = run.verify(case)
    _check_end_to_end(case, gpu, H.run_oracle(case))
    again = run.verify(case)
    for key in ("accept_len", "next_token", "target_probs", "hidden", "kv_k", "kv_v"):
        np.testing.assert_array_equal(gpu[key], again[key], err_msg=key)
    run.close()
