"""How a call is dealt to CTAs (csrc/launch_plans.h), checked over sizes on the host: the header holds no CUDA and is compiled
with the host compiler."""
import ctypes
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2511_13587_b200", "csrc")
N_SMS = 148
FIELDS = ("nt", "passes", "tiles", "kb_total", "splits", "stages", "alias", "recv_off", "smem_bytes", "tmem_cols", "threads",
          "tiles_on_z")
FEW_FIELDS = ("nt", "tiles", "kb_total", "splits", "group", "stages", "ring", "recv_off", "smem_bytes", "tmem_cols",
              "parts", "acc_ld")
PAIR_FIELDS = ("pairs", "passes", "nt", "kb_total", "sub", "stages", "smem_bytes", "tmem_cols")
SHIM = """
#include "launch_plans.h"
extern "C" void proj(int m, int n, int k, int dual, int n_sms, int* o) {
  const vvs::ProjPlan p = vvs::plan_proj(m, n, k, dual != 0, n_sms);
  const int v[] = {%s, vvs::proj_ss_parts(p)};
  for (unsigned i = 0; i < sizeof(v) / sizeof(v[0]); ++i) o[i] = v[i];
}
extern "C" void few(int m, int n, int k, int dual, int add, int in_l2, int n_sms, int* o) {
  const vvs::ProjFewPlan p = vvs::plan_proj_few(m, n, k, dual != 0, add != 0, in_l2 != 0, n_sms);
  const int v[] = {%s, vvs::proj_ss_parts(p)};
  for (unsigned i = 0; i < sizeof(v) / sizeof(v[0]); ++i) o[i] = v[i];
}
extern "C" void pair(int m, int ff, int k, int n_sms, int* o) {
  const vvs::GateupPairPlan p = vvs::plan_gateup_pair(m, ff, k, n_sms);
  const int v[] = {%s, vvs::proj::kPairTok};
  for (unsigned i = 0; i < sizeof(v) / sizeof(v[0]); ++i) o[i] = v[i];
}
extern "C" void ahead(unsigned bytes, unsigned n_cta, unsigned* o) {
  const vvs::AheadShare s = vvs::ahead_share(bytes, n_cta);
  o[0] = s.every;
  o[1] = s.bytes;
}
extern "C" int tree_parts(int vocab, int n_images, int n_sms) { return vvs::tree_walk_parts(vocab, n_images, n_sms); }
extern "C" int att_split(int hd, int items, int s_max, int n_sms) { return vvs::attention_split(hd, items, s_max, n_sms); }
""" % (", ".join("p." + f for f in FIELDS), ", ".join("p." + f for f in FEW_FIELDS), ", ".join("p." + f for f in PAIR_FIELDS))

# (d_model, d_ff): the benchmark shapes, one between them, one below and one above
WIDTHS = [(1024, 2752), (1280, 3456), (1536, 2744), (2048, 5504), (4096, 11008), (8192, 22016)]


@pytest.fixture(scope="module")
def plans(tmp_path_factory):
    d = tmp_path_factory.mktemp("plans")
    src, lib = str(d / "shim.cc"), str(d / "shim.so")
    with open(src, "w") as f:
        f.write(SHIM)
    subprocess.run([os.environ.get("CXX", "g++"), "-std=c++17", "-O1", "-Wall", "-Werror", "-shared", "-fPIC", "-I", CSRC, src,
                    "-o", lib], check=True)
    return ctypes.CDLL(lib)


def _proj(plans, m, n, k, dual):
    out = (ctypes.c_int * (len(FIELDS) + 1))()
    plans.proj(m, n, k, int(dual), N_SMS, out)
    return dict(zip(FIELDS + ("ss_parts",), out))


def _projections(d, ff):
    return [(3 * d, d, False), (d, d, False), (ff, d, True), (d, ff, False)]


@pytest.mark.parametrize("d,ff", WIDTHS)
def test_projection_plans_fit_the_hardware(plans, d, ff):
    for m in list(range(1, 130)) + list(range(130, 1537, 7)):
        for n, k, dual in _projections(d, ff):
            p = _proj(plans, m, n, k, dual)
            at = (m, n, k, dual, p)
            nacc, kb = 2 if dual else 1, -(-p["kb_total"] // p["splits"])
            assert p["nt"] % 16 == 0 and 16 <= p["nt"] <= 128 and (p["passes"] - 1) * p["nt"] < m <= p["passes"] * p["nt"], at
            assert p["tiles"] == -(-n // 128) and p["kb_total"] == -(-k // 64), at
            assert p["splits"] in (1, 2, 4, 8) and p["splits"] <= p["kb_total"], at
            # a ring that is used again belongs stage by stage to the same one of two issuers
            assert 1 <= p["stages"] <= min(12, kb) and (p["stages"] == kb or p["stages"] >= 2), at
            assert dual or p["stages"] == kb or p["stages"] % 2 == 0, at
            stage = 128 * 64 * 2 * nacc + p["nt"] * 128
            recv = nacc * p["nt"] // 4 * 128 * 16 if p["splits"] > 1 else 0
            need = max(p["stages"] * stage, recv) if p["alias"] else p["stages"] * stage + recv
            assert p["recv_off"] == (0 if p["alias"] else p["stages"] * stage), at
            if p["splits"] == 1:
                need = max(need, p["nt"] * 272)                     # the finished tile, token-major
            assert need + 1024 <= p["smem_bytes"] <= 222 * 1024, at
            # two accumulators; a CTA takes at least as large a share of shared memory as of tensor memory
            assert 2 * p["nt"] <= p["tmem_cols"] <= 512 and p["tmem_cols"] in (32, 64, 128, 256, 512), at
            assert (p["smem_bytes"] + 1024) * 512 >= p["tmem_cols"] * 228 * 1024 - 512, at
            assert p["threads"] in (256, 512) and p["threads"] % (128 // p["splits"]) == 0, at
            assert p["ss_parts"] % 4 == 0 and p["ss_parts"] <= p["tiles"] * 8, at

# Up to how many tokens each projection is taken (QKV, output, gate/up, down projection): those whose CTAs fit at once.  Weights from
# HBM: none where more than three CTAs per SM would be needed (d_model 8192), matrices beyond 64 MB at most 80, otherwise what the
# ranks of plan_proj allow.
TAKEN = {(1024, 5120): [96, 96, 0, 96], (1600, 2048): [0, 96, 96, 96], (2048, 832): [0, 96, 96, 96], (2048, 128): [0, 96, 96, 96],
         (1536, 3008): [96, 83, 96, 80], (1536, 4096): [96, 83, 96, 83], (2048, 5504): [64, 0, 96, 96], (3072, 8192): [32, 0, 80, 64],
         (4096, 11008): [52, 32, 80, 0], (5120, 13824): [80, 0, 80, 0], (8192, 28672): [0, 0, 0, 0], (1024, 65536): [64, 42, 0, 80],
         (16384, 64): [0, 0, 64, 0]}


@pytest.mark.parametrize("d,ff,in_l2", [(1024, 320, 1), (1024, 2752, 1), (1024, 5120, 1), (1600, 2048, 1), (2048, 832, 1),
                                        (1152, 3072, 1), (1280, 3456, 1), (1280, 64, 1), (2048, 128, 1), (1536, 3008, 0), (1536, 4096, 0), (2048, 5504, 0), (3072, 8192, 0), (4096, 11008, 0),
                                        (5120, 13824, 0), (8192, 28672, 0), (1024, 65536, 0), (16384, 64, 0)])
def test_few_token_plans_fit_the_hardware(plans, d, ff, in_l2):
    taken = [0, 0, 0, 0]                                            # calls of up to so many tokens: QKV, output, gate/up, down projection
    for m in range(1, 97):
        for i, (n, k, dual, add) in enumerate(((3 * d, d, 0, 0), (d, d, 0, 1), (ff, d, 1, 0), (d, ff, 0, 1))):
            out = (ctypes.c_int * (len(FEW_FIELDS) + 1))()
            plans.few(m, n, k, dual, add, in_l2, N_SMS, out)
            p = dict(zip(FEW_FIELDS + ("ss_parts",), out))
            at = (m, n, k, dual, add, p)
            if p["stages"] == 0:
                continue                                            # left to proj_tc.cu
            assert taken[i] == m - 1, at
            taken[i] = m
            assert p["nt"] % 8 == 0 and p["nt"] - 8 < m <= p["nt"], at
            assert p["tiles"] == -(-n // (32 if dual else 64)) and p["kb_total"] == k // 64, at
            # where the sums are kept apart: whole slices of the other kernel's plan, and for an ADD its ranks of 16 rows
            wide = _proj(plans, m, n, k, dual)["splits"]
            assert (p["parts"] == 0 if in_l2 else p["parts"] * p["splits"] == wide) and (in_l2 or not add or wide == 8), at
            n_acc = max(1, p["parts"] * (1 if dual else 2))
            # the kernels that exist, (slices, k-blocks a stage, ring, sums apart): gate/up unsplit, QKV split unless its sums are kept
            # apart, an output or down projection split or of less than eight k-blocks
            kernel = p["splits"], p["group"], bool(p["ring"]), p["parts"] > 0
            own = [(4, True, False), (4, False, False), (5, False, False), (7, False, False)]
            assert kernel[1:] in own + [(2, True, True)], at
            assert p["splits"] in ((1,) if dual else (1, 4) if add else (1, 2)) and p["splits"] <= p["kb_total"], at
            assert dual or p["splits"] > 1 or (kernel[1:] in own[1:] if add else p["parts"] > 0), at
            per_cta = -(-p["kb_total"] // p["splits"])
            groups = -(-per_cta // p["group"])
            assert p["group"] in (2, 4, 5, 7) and 1 <= p["stages"] <= min(12, groups) and p["ring"] == (not in_l2 or p["stages"] < groups), at
            assert not p["ring"] or p["group"] == (4 if in_l2 else 2), at
            assert p["stages"] >= min(2, groups), at
            # stages, and the tile's rows beside them (split) or over them
            stage, recv = p["group"] * (64 + p["nt"]) * 128, -(-m // 4) * 1024 * (max(1, p["parts"]) if p["splits"] > 1 else 1)
            assert p["recv_off"] == (p["stages"] * stage if p["splits"] > 1 else 0), at
            need = p["stages"] * stage + recv if p["splits"] > 1 else max(p["stages"] * stage, recv)
            assert need + 1024 <= p["smem_bytes"] <= 226 * 1024, at
            assert p["acc_ld"] % 32 == 0 and p["nt"] <= p["acc_ld"] and p["tmem_cols"] in (32, 64, 128, 256, 512), at
            assert (p["nt"] if n_acc == 1 else p["acc_ld"] * n_acc) <= p["tmem_cols"], at
            assert (p["smem_bytes"] + 2048) * 512 >= p["tmem_cols"] * 228 * 1024 - 512, at
            # the sums of squares: whole float4, room for d / 16 of them per token
            assert p["ss_parts"] % 4 == 0 and p["tiles"] * p["splits"] <= p["ss_parts"] < p["tiles"] * p["splits"] + 4, at
            assert not add or p["ss_parts"] <= (d + 127) // 128 * 8, at
            # all CTAs at once, with 1 KB each for the system and what is static
            per_sm = 228 * 1024 // (p["smem_bytes"] + 2048) if p["smem_bytes"] <= 112 * 1024 else 1
            assert p["tiles"] * p["splits"] <= min(per_sm, 3) * N_SMS * (33 / 37 if p["splits"] == 4 else 1), at
    assert taken == TAKEN.get((d, ff), [96] * 4)


def _pair(plans, m, ff, k):
    out = (ctypes.c_int * (len(PAIR_FIELDS) + 1))()
    plans.pair(m, ff, k, N_SMS, out)
    return dict(zip(PAIR_FIELDS + ("most",), out))


@pytest.mark.parametrize("d", [1024, 1088, 1280, 1408, 1536, 2048])
def test_pair_plans_fit_the_hardware(plans, d):
    """Gate/up on CTA pairs: one wave of passes, none of them empty, everything inside a CTA's shared and tensor memory."""
    taken = 0
    for ff in (64, 512, 1024, 1536, 2048, 2560, 2752, 3072, 3456, 4096, 4800, 5120, 6144):
        for m in list(range(1, 400)) + list(range(400, 1300, 13)):
            p = _pair(plans, m, ff, d)
            if p["pairs"] == 0:
                continue
            taken += 1
            at = (m, ff, d, p)
            one = _proj(plans, m, ff, d, True)                       # the kernel whose place it takes: unsplit, weights that stay in L2
            assert one["splits"] == 1 and not one["tiles_on_z"] and ff * d * 4 <= 20 << 20, at
            assert p["pairs"] == -(-ff // 128) and p["pairs"] * p["passes"] <= N_SMS // 2, at
            assert p["nt"] % 32 == 0 and 32 <= p["nt"] <= p["most"] and (p["passes"] - 1) * p["nt"] < m <= p["passes"] * p["nt"], at
            assert p["sub"] in (1, 2) and p["kb_total"] * p["sub"] >= d // 64 > (p["kb_total"] - 1) * p["sub"], at
            assert min(2, p["kb_total"]) <= p["stages"] <= min(12, p["kb_total"]), at
            stage = p["sub"] * (128 + p["nt"] // 2) * 128            # a CTA's rows of gate and up, half of the tokens
            assert max(p["stages"] * stage, p["nt"] * 144) + 1024 <= p["smem_bytes"] <= 222 * 1024, at
            assert p["nt"] <= p["tmem_cols"] and p["tmem_cols"] in (32, 64, 128, 256), at
            assert (p["smem_bytes"] + 1024) * 512 >= p["tmem_cols"] * 228 * 1024 - 512, at
            # passes no longer than the K range pays for
            assert p["nt"] <= (160 if ff * d * 4 * (d // 64) >= 270 << 20 else 128 if d >= 1152 else 64), at
    assert taken > 100, taken


def test_pairs_are_taken_where_their_bits_are_compared(plans):
    from test_gpu_gateup_pair import CASES, FEW_CASES, NOT_TAKEN
    widths = set()
    for ms, n_images, n_cfg, k, _ in CASES:
        m = n_images * n_cfg * (1 + k)
        p = _pair(plans, m, ms.d_ff, ms.d_model)
        assert (p["pairs"] == 0) == ((ms.name, m) in NOT_TAKEN), (ms.name, m, p)
        widths.add((p["sub"], p["nt"]))
    assert {(2, 64), (2, 96), (1, 128), (1, 160)} <= widths, widths
    for ms, n_images, n_cfg, k in FEW_CASES:
        m, out = n_images * n_cfg * (1 + k), (ctypes.c_int * (len(FEW_FIELDS) + 1))()
        plans.few(m, ms.d_ff, ms.d_model, 1, 0, 1, N_SMS, out)
        assert dict(zip(FEW_FIELDS, out))["stages"] == 0 and _pair(plans, m, ms.d_ff, ms.d_model)["pairs"] > 0, (ms.name, m)


def test_requests_into_l2_are_shared_out(plans):
    """Whole requests, all of the weights where there are CTAs enough, and no CTA kept at it for long."""
    for n_cta in (1, 2, 26, 27, 80, 108, 128, 132, 192):
        for n_bytes in (0, 16, 4096, 4112, 128 * 1024, 3276800, 9830400, 17694720, 31850496):
            out = (ctypes.c_uint * 2)()
            plans.ahead(n_bytes, n_cta, out)
            every, part = out
            assert every % 4096 == 0 and n_bytes <= every * n_cta < n_bytes + n_cta * 4096, (n_cta, n_bytes)
            assert part == min(every, 256 << 10), (n_cta, n_bytes)


def test_passes_over_weights_that_exceed_l2(plans):
    """Up to 128 tokens stream such weights once; more take the fewest passes of up to 64, those of a tile side by side."""
    for m in list(range(1, 260)) + [288, 504, 576, 1152]:
        for n, k, dual in _projections(4096, 11008):
            p = _proj(plans, m, n, k, dual)
            if n * k * 2 * (2 if dual else 1) <= 64 << 20:
                assert not p["tiles_on_z"], (m, n, k, p)
            elif m <= 128:
                assert p["passes"] == 1 and not p["tiles_on_z"], (m, n, k, p)
            else:
                assert p["passes"] == -(-m // 64) and p["nt"] <= 64 and p["tiles_on_z"], (m, n, k, p)


@pytest.mark.parametrize("hd", [64, 128])
def test_attention_split(plans, hd):
    for items in range(1, 400):
        for s_max in (1, 511, 512, 592, 1023, 1024, 1535, 1536, 3071, 3072, 4608, 1 << 20):
            s = plans.att_split(hd, items, s_max, N_SMS)
            assert s in (1, 2, 4) and (s == 1 or items * s <= N_SMS), (items, s_max, s)
    # one image of 20 heads, with and without guidance: idle SMs share a long cache, a short one is not split
    assert [plans.att_split(64, 40, s, N_SMS) for s in (592, 1535, 1536, 4608)] == [1, 1, 2, 2]
    assert [plans.att_split(64, 20, s, N_SMS) for s in (592, 1536, 4608)] == [1, 2, 4]
    assert [plans.att_split(128, 64, s, N_SMS) for s in (511, 512, 2384)] == [1, 2, 2]


def test_tree_walk_parts(plans):
    for vocab in (1, 64, 2048, 4096, 8191, 8192, 10000, 16383, 16384, 65536, 1 << 23):
        for n_images in (1, 2, 4, 8, 15, 16, 33, 34, 40, 74, 75, 500):
            s = plans.tree_parts(vocab, n_images, N_SMS)
            # small codebooks stay with one CTA; otherwise all clusters find room at once (15 of eight CTAs, 33 of four)
            assert s == 1 if vocab < 8192 else s in (1, 2, 4, 8), (vocab, n_images, s)
            assert n_images <= {1: n_images, 2: 74, 4: 33, 8: 15}[s], (vocab, n_images, s)
    assert [plans.tree_parts(16384, b, N_SMS) for b in (1, 15, 16, 33, 34, 75)] == [8, 8, 4, 4, 2, 1]
