"""Attention of many (sequence, head) items, where a CTA takes several and requests the keys of the next before it merges the last,
and of few: fills at the edges of slices of 16 and 32 keys, empty caches, more slices than one item's warps hold at once, both
head sizes, up to 16 block rows and more."""
from dataclasses import replace

import numpy as np
import pytest

import helpers as H
from test_gpu_verify import _check_end_to_end
from vvs_synth.configs import B7, XL

pytestmark = pytest.mark.gpu

MS64 = replace(XL, name="items64", n_layers=2, d_model=1024, n_heads=16, d_ff=320, vocab=1096, lm_rows=0, tok_rows=0, s_max=592)
MS128 = replace(B7, name="items128", n_layers=2, d_model=1024, n_heads=8, d_ff=320, vocab=1096, vocab_offset=64, lm_rows=2048,
                tok_rows=0, s_max=300)


@pytest.mark.parametrize("ms,n_cfg,n_forced,k,fills", [
    (MS64, 2, 1, 8, [0, 15, 16, 17, 31, 32, 33, 150, 47, 48, 583, 64, 8, 1, 290, 128]),             # 512 items, 444 CTAs
    (MS64, 2, 1, 3, [0, 12, 13, 28, 29, 300]),                                                      # 192: one each
    (MS64, 1, 3, 17, [0, 12, 31, 32, 33, 44, 64, 100, 13, 1, 199, 572, 80, 96, 95, 97, 11, 300, 45, 46, 250]),  # 336, 296 CTAs
    (MS64, 2, 1, 8, [583]),                                                                         # 32: 19 slices, 16 warps
    (MS64, 1, 2, 30, [0, 17, 289, 288, 223]),                                                       # 80, two groups of warps
    (MS128, 2, 1, 8, [0, 7, 8, 15, 16, 17, 31, 32, 33, 150, 291, 47, 48, 63, 64, 20, 1, 2, 100, 90]),   # 320 items, 296 CTAs
    (MS128, 2, 1, 20, [0, 1, 11, 12, 27, 28, 200, 279, 130, 16])])                                  # 160: one each
def test_attention_items(ms, n_cfg, n_forced, k, fills):
    case = H.build_case_independent(ms, 3100 + k, len(fills), n_cfg, n_forced, k, fills, logit_std=0.6)
    run = H.GpuRunner(ms, case["w"], len(fills) * n_cfg, n_forced + k)
    gpu = run.verify(case)
    _check_end_to_end(case, gpu, H.run_oracle(case))
    again = run.verify(case)
    for key in ("accept_len", "next_token", "target_probs", "hidden", "kv_k", "kv_v"):
        np.testing.assert_array_equal(gpu[key], again[key], err_msg=key)
    run.close()
