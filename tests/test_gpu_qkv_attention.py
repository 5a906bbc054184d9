"""QKV and attention as one kernel (qkv_attention_few.cu, one to three sequences).  The rows of a sequence do not depend on what else is in a
call, and four or more sequences take the two kernels: images alone give the bits that they give in a batch, with a launch less per
layer.  Trees against the oracle, a sequence that does not fit its cache, what the launch counts as.  And the plan over sizes."""
import ctypes
import os
import subprocess
from dataclasses import replace

import pytest

import helpers as H
from test_gpu_same_bits import _ints, _weights
from vvs_synth.configs import XL

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2511_13587_b200", "csrc")
SHAPE = replace(XL, name="qkv_attention", n_layers=2, d_model=1024, n_heads=16, d_ff=1024, vocab=512, lm_rows=0, tok_rows=0, s_max=700)
HEADS17 = replace(SHAPE, name="heads17", d_model=1088, n_heads=17)       # K slices of eight and nine blocks in stages of five
HEADS22 = replace(SHAPE, name="heads22", d_model=1408, n_heads=22)       # eleven in three stages of four; as many clusters as fit


def _step(ctx_rows, w, block, parents, fills, n_cfg, kv, ms=SHAPE, status=0):
    """Launches, features and cache rows of one step on the given images (caches: cond rows, then uncond rows)."""
    import torch

    from paper_2511_13587_b200 import binding as vb
    b, t_len = block.shape
    rows = b * n_cfg
    ctx = vb.vvs_create(vb.make_desc(ms, ctx_rows, t_len, 1))
    vb.vvs_bind_weights(ctx, w)
    kv = [x.clone() for x in kv]
    zeros = lambda *shape: torch.zeros(shape, dtype=torch.int32, device="cuda")  # noqa: E731
    hidden = torch.zeros((rows, t_len, ms.d_model), dtype=torch.bfloat16, device="cuda")
    k = t_len - 1
    more = {} if parents is None else dict(tree_parent=torch.tensor([parents] * b, dtype=torch.int32, device="cuda"),
                                           target_probs=torch.zeros((b, t_len, ms.vocab), device="cuda"))
    vb.vvs_verify(ctx, n_images=b, n_cfg=n_cfg, n_forced=1, n_draft_max=k, block=block.contiguous(), kv_k=kv[0], kv_v=kv[1], kv_rows=rows,
                  cache_len=torch.tensor(fills * n_cfg, dtype=torch.int32, device="cuda"),
                  draft_probs=torch.full((b, max(k, 1), ms.vocab), 1.0 / ms.vocab, device="cuda"),
                  uniforms=torch.full((b, k + 1), 0.5, device="cuda"), cfg_scale=2.0 if n_cfg == 2 else 1.0, temperature=1.0, mode=0,
                  nbr_k=1, hidden=hidden, accept_len=zeros(b), next_token=zeros(b), new_len=zeros(rows), n_commit=zeros(rows),
                  accept_mask=torch.zeros((b, max(k, 1)), dtype=torch.uint8, device="cuda"), **more)
    assert vb.vvs_device_status(ctx, raise_on_error=False) == status
    launches = vb.vvs_last_launch_count(ctx)
    vb.vvs_destroy(ctx)
    out = [hidden] if parents else [hidden, *kv]             # (a tree call moves the accepted rows afterwards)
    return launches, [x.view(torch.int16).cpu() for x in out]


@pytest.mark.gpu
@pytest.mark.parametrize("n_cfg,group,t_len,tree,fills", [
    (2, 1, 9, False, [300, 0]), (2, 1, 9, False, [31, 32]), (2, 1, 9, False, [24, 23]), (2, 1, 1, False, [511, 512]),
    (2, 1, 9, False, [503, 504]), (2, 1, 9, False, [543, 691]),             # more than sixteen slices: a part takes two
    (2, 1, 16, False, [495, 497]), (2, 1, 13, True, [7, 640]),
    (2, 1, 17, False, [250, 239]), (2, 1, 24, False, [231, 668]),           # two row groups, eight parts each
    (1, 1, 9, False, [5, 570, 64, 200]), (1, 1, 24, False, [511, 256, 0, 668]), (1, 1, 16, True, [511, 256, 0, 668]),
    (1, 2, 9, False, [5, 570, 64, 200]), (1, 3, 10, False, [1, 33, 544, 690, 0, 100])])
def test_images_alone_or_in_a_batch(n_cfg, group, t_len, tree, fills):
    _check_alone(SHAPE, n_cfg, group, t_len, tree, fills)


@pytest.mark.gpu
@pytest.mark.parametrize("ms,n_cfg,group,t_len,fills", [
    (HEADS17, 2, 1, 9, [300, 31]), (HEADS17, 1, 3, 3, [1, 33, 544, 690, 0, 100]), (HEADS17, 1, 3, 24, [0, 33, 500, 670]),
    (HEADS22, 2, 1, 9, [300, 31]), (HEADS22, 1, 1, 24, [511, 256, 0, 668]), (HEADS22, 1, 3, 21, [0, 33, 500, 670]),
    (SHAPE, 1, 3, 17, [0, 33, 500, 670]), (SHAPE, 1, 3, 24, [668, 240, 7, 0])])     # three sequences of two row groups
def test_other_widths_and_three_long_sequences(ms, n_cfg, group, t_len, fills):
    _check_alone(ms, n_cfg, group, t_len, False, fills)


@pytest.mark.gpu
@pytest.mark.parametrize("ms,t_len,fills", [(SHAPE, 32, [0, 33, 668]), (SHAPE, 32, [487, 488, 7]), (HEADS17, 29, [500, 671, 16])])
def test_three_sequences_or_each_alone(ms, t_len, fills):
    """The longest of three sequences: more tokens than four could have in proj_few.cu.  Two CTAs share an item or six."""
    import torch
    w = _weights(ms, 8150)
    block = torch.randint(0, ms.vocab, (3, t_len), generator=torch.Generator().manual_seed(8151), dtype=torch.int32).cuda()
    kv = [_ints((ms.n_layers, 3, ms.n_heads, ms.s_max, ms.head_dim), 96, 32, 8152 + i) for i in range(2)]
    launches, want = _step(3, w, block, None, fills, 1, kv, ms)
    for i in range(3):
        same, got = _step(1, w, block[i:i + 1], None, fills[i:i + 1], 1, [x[:, i:i + 1].contiguous() for x in kv], ms)
        assert same == launches
        for a, e in zip(got[1:], want[1:]):
            assert torch.equal(a, e[:, i:i + 1])


def _check_alone(ms, n_cfg, group, t_len, tree, fills):
    import torch
    b = len(fills)
    w = _weights(ms, 8100)
    g = torch.Generator().manual_seed(8200 + t_len)
    block = torch.randint(0, ms.vocab, (b, t_len), generator=g, dtype=torch.int32).cuda()
    parents = [-1] + [int(torch.randint(0, t, (1,), generator=g)) for t in range(1, t_len)] if tree else None
    kv = [_ints((ms.n_layers, b * n_cfg, ms.n_heads, ms.s_max, ms.head_dim), 96, 32, 8300 + i) for i in range(2)]
    launches, want = _step(b * n_cfg, w, block, parents, fills, n_cfg, kv, ms)
    for at in range(0, b, group):
        images = list(range(at, min(at + group, b)))
        rows = [c * b + i for c in range(n_cfg) for i in images]
        fewer, got = _step(len(rows), w, block[images], parents, [fills[i] for i in images], n_cfg, [x[:, rows].contiguous() for x in kv], ms)
        assert fewer == launches - ms.n_layers
        if b * n_cfg * t_len <= 64:                # (the final norm of more rows takes its sums in another order)
            assert torch.equal(got[0], want[0][rows])
        for a, e in zip(got[1:], want[1:]):
            assert torch.equal(a, e[:, rows])


@pytest.mark.gpu
@pytest.mark.parametrize("t_len,n_cfg,fill", [(17, 2, 180), (27, 2, 77), (32, 2, 0), (32, 1, 300)])
def test_trees_of_two_row_groups(t_len, n_cfg, fill):
    from test_gpu_tree import _check_tree
    parent = [-1] + [max(0, (5 * t) // 8 - t % 3) for t in range(1, t_len)]
    ms = replace(SHAPE, name="tree")
    case = H.build_tree_case(ms, 8600 + t_len, 1, n_cfg, 1, parent, [fill], q_noise=0.7)
    run = H.GpuRunner(ms, case["w"], n_cfg, t_len)
    _check_tree(case, H.run_tree_gpu(run, case), H.run_tree_oracle(case))
    run.close()


@pytest.mark.gpu
@pytest.mark.parametrize("fills", [[699, 300], [300, 695], [-1, 20]])
def test_a_sequence_that_does_not_fit_beside_one_that_does(fills):
    """No keys, no parts and zeros for it, nothing in its cache; the other one as ever."""
    import torch

    from paper_2511_13587_b200 import binding as vb
    w = _weights(SHAPE, 8700)
    block = torch.randint(0, SHAPE.vocab, (4, 9), generator=torch.Generator().manual_seed(8701), dtype=torch.int32).cuda()
    kv = [_ints((SHAPE.n_layers, 4, SHAPE.n_heads, SHAPE.s_max, SHAPE.head_dim), 96, 32, 8702 + i) for i in range(2)]
    launches, want = _step(4, w, block, None, fills + [1, 2], 1, kv, status=vb.VVS_DEV_CACHE_OVERFLOW)
    fewer, got = _step(2, w, block[:2], None, fills, 1, [x[:, :2].contiguous() for x in kv], status=vb.VVS_DEV_CACHE_OVERFLOW)
    assert fewer == launches - SHAPE.n_layers
    bad = 0 if not 0 <= fills[0] <= SHAPE.s_max - 9 else 1
    assert torch.equal(got[0], want[0][:2])
    for a, e, before in zip(got[1:], want[1:], kv):
        assert torch.equal(a, e[:, :2])
        assert torch.equal(a[:, bad], before[:, bad].view(torch.int16).cpu()) and not torch.equal(a[:, 1 - bad], before[:, 1 - bad].view(torch.int16).cpu())


@pytest.mark.gpu
@pytest.mark.parametrize("n_images,one_kernel", [(1, True), (2, False)])
def test_classes_of_a_profiled_step(n_images, one_kernel):
    """One launch for QKV and attention of a layer counts with the projections (include/vvs.h); profiling changes no result."""
    case = H.build_case_independent(SHAPE, 8650, n_images, 2, 1, 8, [77, 300][:n_images], logit_std=0.6)
    run = H.GpuRunner(SHAPE, case["w"], 2 * n_images, 9)
    want = run.verify(case)
    run.vb.vvs_profile_enable(run.ctx, True)
    got = run.verify(case)
    ms, launches = run.vb.vvs_profile_read(run.ctx)
    run.vb.vvs_profile_enable(run.ctx, False)
    assert (got["hidden"] == want["hidden"]).all() and sum(launches) == want["launches"] == got["launches"]
    assert launches[:2] == [4 * SHAPE.n_layers + 1, 0 if one_kernel else SHAPE.n_layers] and launches[3] == 0
    assert ms[0] > 0 and (ms[1] > 0) == (not one_kernel)
    run.close()


def test_plan(tmp_path):
    """Everything that lies over the stages lies inside the shared memory of a CTA, for every size that the kernel takes."""
    src, lib = str(tmp_path / "shim.cc"), str(tmp_path / "shim.so")
    with open(src, "w") as f:
        f.write("""
#include "launch_plans.h"
extern "C" void plan(int rows, int t, int d, int s_max, int* o) {
  const vvs::ProjFewPlan q = vvs::plan_proj_few(rows * t, 3 * d, d, false, false, true, 148);
  const vvs::QkvAttentionPlan p = vvs::plan_qkv_attention(q, d / 64, 64, d, rows, t, s_max, 148);
  const int v[] = {p.per_item, p.part_off, p.recv_off, p.new_off, p.smem_bytes, q.stages * q.group * (8192 + q.nt * 128), q.nt};
  for (int i = 0; i < 7; ++i) o[i] = v[i];
}
""")
    subprocess.run([os.environ.get("CXX", "g++"), "-std=c++17", "-Wall", "-Werror", "-shared", "-fPIC", "-I", CSRC, src, "-o", lib], check=True)
    plan, taken = ctypes.CDLL(lib).plan, 0
    for d in range(1024, 2049, 64):
        for rows in range(1, 6):
            for t in range(1, 33):
                o = (ctypes.c_int * 7)()
                plan(rows, t, d, 592, o)
                per_item, part_off, recv_off, new_off, smem, stages, nt = o
                if per_item == 0:
                    continue
                taken += 1
                assert rows <= 3 and per_item * rows == 6 and d // 64 * 6 <= 132 and d // 16 <= 128   # (sums of squares of a token)
                assert -(-16 // per_item) <= 8 and part_off == -(-16 // per_item) * 8192      # a part a warp, a slot each
                assert part_off + 16 * min(t, 16) * 102 * 4 <= recv_off and stages <= recv_off
                assert recv_off + (nt + 3) // 4 * 1024 <= new_off and new_off + 384 * t + 1024 <= smem <= 226 * 1024
                plan(rows, t, d, 4608, o)                                                     # long caches are split over clusters
                assert o[0] == 0 or rows * d // 64 * 2 > 148
    assert taken > 100
