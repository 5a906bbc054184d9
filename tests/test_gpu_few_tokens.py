"""The folded step of few tokens (proj_few.cu) on two layers: token counts at the edges of MMA widths, quads and the range itself
(97 tokens take proj_tc.cu), rings and stages that hold everything, K ranges that the slices and stages do not divide."""
from dataclasses import replace

import numpy as np
import pytest

import helpers as H
from test_gpu_tree import _check_tree
from test_gpu_verify import _check_end_to_end
from vvs_synth.configs import B7, XL

pytestmark = pytest.mark.gpu

# 43 k-blocks of the down projection in four slices of 10 and 11; 86 tiles of gate and up
FEW64 = replace(XL, name="few64", n_layers=2, d_model=1024, n_heads=16, d_ff=2752, vocab=1096, lm_rows=0, tok_rows=0, s_max=208)
# heads of two tiles; 18 tiles: sums of squares in rows of 18 and 72 parts; a down projection of 5 k-blocks, unsplit
FEW128 = replace(B7, name="few128", n_layers=2, d_model=1152, n_heads=9, d_ff=320, vocab=1096, vocab_offset=64, lm_rows=2048,
                 tok_rows=0, s_max=700)
# CTAs that would not all fit at once: QKV (150) and gate/up (160) go to proj_tc.cu, the others stay; gate/up of six CTAs, which request
# a part of the next QKV matrix only
WAVES_QKV = replace(FEW64, name="waves_qkv", d_model=1600, n_heads=25, d_ff=2048)
WAVES_GU = replace(FEW64, name="waves_gu", d_ff=5120)
NARROW = replace(FEW64, name="narrow", d_ff=192)
# weights that do not stay in L2: rings of two k-blocks, one CTA per SM; 47 k-blocks in four slices
STREAM1 = replace(XL, name="stream1", n_layers=1, d_model=1536, n_heads=24, d_ff=3008, vocab=1096, lm_rows=0, tok_rows=0, s_max=208)
# the same with two CTAs per SM (QKV, 192) and three (gate and up, 298)
STREAM3 = replace(B7, name="stream3", n_layers=1, d_model=2048, n_heads=16, d_ff=9536, vocab=1096, vocab_offset=64, lm_rows=2048,
                  tok_rows=0, s_max=700)


@pytest.mark.parametrize("ms,n_images,n_cfg,n_forced,k,fills", [
    (FEW64, 1, 1, 1, 0, [0]),                              # 1 token, no draft
    (FEW64, 1, 2, 1, 3, [199]),                            # 8
    (FEW64, 1, 1, 2, 7, [16]),                             # 9
    (FEW64, 3, 1, 1, 10, [0, 47, 150]),                    # 33
    (FEW64, 1, 2, 1, 24, [150]),                           # 50 and 58: thirteen and fifteen quads of sixteen items, the last half warp
    (FEW64, 1, 2, 1, 28, [77]),                            # of them in warps 1 and 0
    (STREAM3, 1, 2, 1, 24, [513]),
    (STREAM1, 1, 2, 1, 28, [77]),
    (FEW64, 2, 2, 6, 10, [3, 190]),                        # 64
    (FEW64, 5, 1, 3, 10, [3, 20, 37, 90, 190]),            # 65
    (FEW64, 3, 2, 1, 15, [0, 47, 150]),                    # 96
    (FEW64, 97, 1, 1, 0, list(range(97))),                 # 97
    (FEW128, 1, 2, 1, 8, [513]),                           # 18
    (FEW128, 3, 2, 1, 4, [5, 160, 677]),                   # 30
    (FEW128, 4, 1, 3, 20, [5, 160, 333, 64]),              # 92
    (WAVES_QKV, 1, 2, 1, 8, [199]),
    (WAVES_GU, 1, 2, 1, 8, [199]),
    (WAVES_GU, 3, 2, 1, 15, [0, 47, 150]),                 # 96
    (NARROW, 1, 2, 1, 8, [77]),
    (STREAM1, 1, 1, 1, 0, [0]),
    (STREAM1, 1, 2, 1, 8, [199]),
    (STREAM1, 3, 2, 1, 15, [0, 47, 150]),                  # 96
    (STREAM3, 1, 2, 1, 8, [513]),
    (STREAM3, 2, 2, 6, 10, [3, 677]),                      # 64
    (STREAM3, 3, 1, 3, 24, [5, 160, 333])])                # 81: gate and up (78 MB) in proj_tc.cu, the others here
def test_few_tokens(ms, n_images, n_cfg, n_forced, k, fills):
    case = H.build_case_independent(ms, 1900 + k, n_images, n_cfg, n_forced, k, fills, logit_std=0.6)
    run = H.GpuRunner(ms, case["w"], n_images * n_cfg, n_forced + k)
    gpu = run.verify(case)
    _check_end_to_end(case, gpu, H.run_oracle(case))
    again = run.verify(case)
    for key in ("accept_len", "next_token", "target_probs", "hidden", "kv_k", "kv_v"):
        np.testing.assert_array_equal(gpu[key], again[key], err_msg=key)
    run.close()


def test_few_tokens_tree():
    parent = [-1, 0, 0, 1, 1, 2, 3, 3, 6, 6, 4, 5, 9, 2, 7, 8, 8, 10, 11, 15, 1, 20]
    case = H.build_tree_case(FEW64, 1950, 2, 2, 1, parent, [77, 0], q_noise=0.7)
    run = H.GpuRunner(FEW64, case["w"], 4, len(parent))
    _check_tree(case, H.run_tree_gpu(run, case), H.run_tree_oracle(case))
    run.close()


@pytest.mark.parametrize("ms", [FEW64, STREAM1])
def test_gate_and_up_wherever_they_lie(ms):
    """They are loaded as one tensor of two matrices: up before gate gives the same bits, one matrix as both takes the other kernel."""
    import torch
    case = H.build_case_independent(ms, 1970, 1, 2, 1, 8, [150], logit_std=0.6)
    run = H.GpuRunner(ms, case["w"], 2, 9)
    want = run.verify(case)
    for layer in run.wd["layers"]:
        both = torch.stack([layer["w_up"], layer["w_gate"]])
        layer["w_up"], layer["w_gate"] = both[0], both[1]
    run.vb.vvs_bind_weights(run.ctx, run.wd)
    got = run.verify(case)
    for key in ("accept_len", "next_token", "target_probs", "hidden", "kv_k", "kv_v"):
        np.testing.assert_array_equal(want[key], got[key], err_msg=key)
    for layer in run.wd["layers"]:
        layer["w_up"] = layer["w_gate"].clone()
    run.vb.vvs_bind_weights(run.ctx, run.wd)
    want = run.verify(case)
    for layer in run.wd["layers"]:
        layer["w_up"] = layer["w_gate"]
    run.vb.vvs_bind_weights(run.ctx, run.wd)
    assert H.rel_err_rows(run.verify(case)["hidden"], want["hidden"]) < 1e-2      # (bf16 features, as against the oracle)
    run.close()
