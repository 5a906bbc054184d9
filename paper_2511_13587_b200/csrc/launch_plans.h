// How calls are dealt to CTAs: arithmetic on sizes, no CUDA, so that it can be checked on any host.
#pragma once

#include <stddef.h>
#include <stdint.h>

namespace vvs {

// ---- projections with folded epilogues, proj_tc.cu -----------------------------------------------
namespace proj {
constexpr int kMaxStages = 12;
constexpr int kMaxThreads = 512;
constexpr int kMaxTok = 128;              // tokens per pass
constexpr int kPairTok = 160;             // the same, gate/up on CTA pairs
constexpr uint32_t kTileRows = 128;       // weight rows per tile = MMA M
constexpr uint32_t kBlockK = 64;          // bf16 elements per smem row = one 128-byte swizzle row
constexpr uint32_t kATileBytes = kTileRows * kBlockK * 2;
constexpr int kFewTok = 96;               // proj_few.cu: tokens of a call,
constexpr int kFewStages = 12;            // stages of a ring,
constexpr int kFewSmem = 226 * 1024;      // dynamic shared memory of a CTA
}  // namespace proj

struct ProjPlan {
  int nt, passes, tiles, kb_total, splits, stages, alias, recv_off, smem_bytes, tmem_cols, threads;
  int tiles_on_z;              // grid (passes, slices, tiles) in the place of (tiles, slices, passes)
};

// partial sums of squares per token an ADD projection writes (at most d / 16 rounded up to tiles)
inline int proj_ss_parts(const ProjPlan& pl) {
  using namespace proj;
  const int rpr = (int)kTileRows / pl.splits;
  return pl.tiles * (int)kTileRows / (rpr < 32 ? rpr : 32);
}

// Token passes, K splits and ring of one projection.
//
// Up to 20 MB of weights (a step's layers then fit in L2 together, see the prefetch) a projection is bound by the chain
// of one CTA, one CTA per SM: k-blocks x the slower of filling shared memory (55 bytes per clock and SM, measured from
// L2) and issuing (280 cycles per issuer and k-block), then the exchange (a fixed 2000 cycles, 25 per token, three times
// that with two accumulators, 1500 for the barrier of one that lies over the stages, 400 per epilogue item) or, unsplit,
// the epilogue (47 per token); 1500 cycles per further wave.  The cheapest of all pass counts and splits is taken.  At the
// XL shape (d 1280): 18 tokens 1 pass x 4 (QKV, gate/up) or 8 (O, down) slices, 972 us per step against 1054 with as many
// small slices as make two CTAs per SM; 288 tokens unsplit passes of 64-80 tokens for QKV and gate/up, 1.95 ms against
// 3.01 ms with the same rule.  (With eight warps an exchanged token cost 60 cycles; 25 chooses a split QKV at 54 tokens,
// 1183 -> 1152 us, and split O at 108 and 180, 1452 -> 1415 and 1615 -> 1551 us.)
// A larger one is bound by HBM: two CTAs per SM keep more of the stream in flight (7B shape, d 4096, 18 tokens: 3.13 ms
// per step against 3.29 with one), and a split deals the rows out evenly over the SMs.
// Where several passes of 32 tokens or more give nearly every SM one CTA with 32 k-blocks or more to stream, a deep ring
// for each does better still (d 2048, 72 tokens 1415 -> 1383 us per step, 126 tokens 1667 -> 1525; 7B down projection,
// 32 tiles x 4, 3049 -> 3028).
// Beyond 64 MB the weights do not stay in L2 from one pass to the next.  Up to 128 tokens one pass streams them once (four
// layers of the 7B shape, 128 tokens 514 us, two passes of 64 595).  More take passes of up to 64, as few as there can be, and
// the passes of a tile run side by side, grid x, so that all but one of them find its weights in L2: 180 tokens 1084 us with
// two passes of 96 one behind the other, 734 with three of 64, 730 with these side by side; 288 tokens 1455, 1191 and 1102;
// 576 tokens 2602, 1981 and 1859.  (Smaller ones stay in L2 and lose by it: d 2048, 72 tokens 430 -> 435.)
// A cluster needs its CTAs' room inside one GPC: of 148 SMs 132 take clusters of four and 120 clusters of eight at one
// CTA per SM, 284 and 264 of 296 at two.
inline ProjPlan plan_proj(int m, int n, int k, bool dual, int n_sms) {
  using namespace proj;
  ProjPlan pl{};
  const int nacc = dual ? 2 : 1;
  pl.tiles = (n + (int)kTileRows - 1) / (int)kTileRows;
  pl.kb_total = (k + (int)kBlockK - 1) / (int)kBlockK;
  const size_t bytes = (size_t)n * k * 2 * nacc;
  const bool large = bytes > ((size_t)20 << 20), huge = bytes > ((size_t)64 << 20);
  // (64: two CTAs' accumulators and their shared memory, below, fit on an SM)
  const int most = large && !(huge && m <= kMaxTok) ? 64 : kMaxTok;
  auto room = [&](int sp, int per_sm) {
    return per_sm == 1 ? (sp == 8 ? n_sms * 30 / 37 : sp == 4 ? n_sms * 33 / 37 : n_sms)
                       : (sp == 8 ? n_sms * 66 / 37 : sp == 4 ? n_sms * 71 / 37 : 2 * n_sms);
  };
  auto ring = [&](int passes, int nt, int sp, int* alias) {
    const int stage_bytes = (int)kATileBytes * nacc + nt * (int)kBlockK * 2, per_cta = (pl.kb_total + sp - 1) / sp;
    const int recv = sp > 1 ? nacc * (nt / 4) * (int)kTileRows * 16 : 0;
    // one CTA per SM: as deep as it gets if nothing is exchanged (XL shape, 288 tokens: 160 KB 1851, 200 KB 1839 us per step)
    // or HBM is the bound, else 160 KB, which leave room for the attention kernel's first CTAs beside it; two: 108 KB
    const int kb = pl.tiles * passes * sp > room(sp, 1) ? 108 : sp == 1 || large ? 200 : 160, budget = kb * 1024 - 1024;
    // a ring that is used again: every stage must always belong to the same issuer (they take turns), or one that is a
    // lap ahead would find the other's unfinished phase
    auto usable = [&](int room_for) {
      int st = room_for < kMaxStages ? room_for : kMaxStages;
      if (st < per_cta && !dual) st &= ~1;
      return st < per_cta ? st : per_cta;
    };
    int stages = usable((budget - recv) / stage_bytes);
    // too shallow beside the exchange's buffer: the exchange lies over the drained stages (costs a cluster barrier: XL shape,
    // 54 tokens, down projection with 4 stages or with 6 and the barrier 1128, 1152 us per step)
    *alias = stages < per_cta && stages < (dual ? 2 : 4);
    if (*alias) stages = usable(budget / stage_bytes);
    if (stages < 2 && per_cta > 1) stages = 2;
    if (*alias && stages * stage_bytes + recv <= budget) *alias = 0;
    // one stage fewer than k-blocks where that is even: the next kernel's first CTAs then fit beside more of this one's
    // (18 tokens 958 -> 940 us, 28 tokens 1004 -> 988; with 16 or 64 tokens a pass they do not, and it costs 1 %)
    if (!dual && sp > 1 && nt == 32 && stages == per_cta && per_cta >= 5 && (per_cta & 1)) stages = per_cta - 1;
    return stages;
  };
  double best = -1.0;
  bool deep = false;                          // the plan taken is one of the deep rings described above
  int S = 1;
  for (int passes = (m + most - 1) / most; passes <= (m + 15) / 16; ++passes) {
    const int nt = ((m + passes - 1) / passes + 15) / 16 * 16;
    if (nt > most || (m + nt - 1) / nt != passes) continue;
    if (huge && pl.passes > 0) break;         // (the weights do not stay in L2 from one pass to the next)
    const int tok = nt < m ? nt : m;
    for (int sp = 1; sp <= 8 && sp <= pl.kb_total; sp *= 2) {
      const int ctas = pl.tiles * passes * sp, kb = (pl.kb_total + sp - 1) / sp, fit = room(sp, large && nt <= 64 ? 2 : 1);
      const int waves = (ctas + fit - 1) / fit;
      int alias;
      ring(passes, nt, sp, &alias);
      const double fill = (kATileBytes * nacc + 2.0 * kBlockK * (nt < 32 ? 32 : nt)) / 55.0, issue = 280.0 * nacc;
      double t = kb * (fill > issue ? fill : issue);
      t += sp > 1 ? 2000.0 + 25.0 * tok * (dual ? 3 : 1) + 1500.0 * alias + 400.0 * ((tok + 3) / 4 * ((int)kTileRows / sp) / 256 + 1)
                  : 47.0 * tok;
      t = t * waves + 1500.0 * (waves - 1);
      // (of several such the one of the fewest passes and slices, i.e. the longest streams: the estimate knows no HBM)
      const bool d = large && kb >= 32 && (huge || nt >= 32) && ctas <= room(sp, 1) && ctas * 20 >= n_sms * 17;
      if (!deep && (d || best < 0.0 || t < best)) {
        deep = d;
        best = t;
        pl.passes = passes;
        pl.nt = nt;
        S = sp;
      }
    }
  }
  pl.splits = S;
  pl.tiles_on_z = huge && pl.passes > 1;
  int alias;
  const int stages = ring(pl.passes, pl.nt, S, &alias);
  const int stage_bytes = (int)kATileBytes * nacc + pl.nt * (int)kBlockK * 2;
  const int recv = S > 1 ? nacc * (pl.nt / 4) * (int)kTileRows * 16 : 0;
  // Eight warps are two per scheduler, and an epilogue item (a row's four tokens: ~250 dependent instructions) then takes
  // 0.9 us: from two items per thread on there are sixteen (XL shape, 288 tokens 2015 -> 1970 us per step, 54 tokens 1243
  // -> 1224; 7B shape 3172 -> 3134).  With fewer, starting eight more warps only costs (18 tokens 958 -> 976).
  pl.threads = (S > 1 ? pl.nt / 4 * (int)kTileRows / S : pl.nt * 8) > 256 ? kMaxThreads : 256;
  pl.stages = stages;
  pl.alias = alias;
  pl.recv_off = alias ? 0 : stages * stage_bytes;
  pl.smem_bytes = (alias ? (stages * stage_bytes > recv ? stages * stage_bytes : recv) : stages * stage_bytes + recv) + 1024;
  if (S == 1 && pl.smem_bytes < pl.nt * 272 + 1024) pl.smem_bytes = pl.nt * 272 + 1024;   // the finished tile, token-major
  int cols = 32;
  while (cols < pl.nt * 2) cols <<= 1;        // two accumulators
  pl.tmem_cols = cols;
  // CTAs of a cluster wait for one another, so none may wait for tensor memory that a waiting one holds: each takes at
  // least as large a share of an SM's shared memory as of its tensor memory, whatever shares the SM with it
  const int share = (int)((228u * 1024u * (unsigned)cols + 511u) / 512u) - 1024;          // (1 KB per CTA is the system's)
  if (pl.smem_bytes < share) pl.smem_bytes = share;
  return pl;
}

// ---- the same for few tokens, proj_few.cu ----------------------------------------------------------
struct ProjFewPlan {
  int nt, tiles, kb_total, splits, group, stages, ring, recv_off, smem_bytes, tmem_cols;    // stages of `group` k-blocks
  int parts;                   // slices of plan_proj's per slice, whose sums are kept apart; 0: sums of its own
  int acc_ld;                  // columns of tensor memory from one accumulator to the next
};

// partial sums of squares per token an ADD projection writes: one per tile and slice, rounded up to whole float4
inline int proj_ss_parts(const ProjFewPlan& pl) { return (pl.tiles * pl.splits + 3) & ~3; }

// A CTA's part of a later projection's weights, which it requests into L2 in pieces of 4 KB: where it begins (CTA x every) and how
// much of it is requested.  An SM requests some 160 KB a microsecond, and the kernel behind waits for it: where a gate/up of narrow
// d_ff has few CTAs for a whole QKV matrix, most of that matrix is left to its own kernel.  18 layers, everything / at most 256 KB a
// CTA (64 to 512 KB are alike): d_model 2304, d_ff 64, 18 tokens 2282 / 483 us; 2048, 512, 18 tokens 512 / 429, 54 tokens 649 / 554;
// 2048, 832, 54 tokens 618 / 569; XL shape (at most 147 KB a CTA) 362 / 361.
struct AheadShare { uint32_t every, bytes; };
inline AheadShare ahead_share(uint32_t bytes, uint32_t n_cta) {
  const uint32_t every = ((bytes + n_cta - 1) / n_cta + 4095u) & ~4095u, most = 256u << 10;
  return {every, every < most ? every : most};
}

// One pass of at most kFewTok tokens, k a multiple of 64; no stages: proj_tc.cu has to take it.  K slices: proj_few.cu has the
// measurements; fewer than eight k-blocks are not worth an exchange.
// in_l2: the model's weights are requested into L2 ahead and a CTA takes as much shared memory as its K range fills.  All CTAs have to
// fit at once here too: a second wave of a few repeats load, MMAs and epilogue in the open.  18 layers, two waves / proj_tc.cu for that
// projection, 18 and 90 tokens: d_model 1024, d_ff 5120 (gate/up 160 CTAs) 414 / 406 and 632 / 573 us; 1600, 2048 (QKV 150) 432 / 428
// and 660 / 586; 1792, 1664 (QKV 168) 445 / 422 and 691 / 607 (around 54 tokens gate/up loses 2 %: 1088, 5120 554 / 564).
// Weights that come from HBM need all CTAs on the device at once, and those of the next projection beside them as they leave: one,
// two or three CTAs per SM, as many as it takes, rings of stages of two k-blocks.  And such models are large and deep: any other order
// of the sums moves their features by 2.4e-3 (24 layers of d_model 2048) to 5.7e-3 (7B shape) and guided probabilities by more than
// the 1e-2 that two correct calls may differ by, so the partial sums of plan_proj's slices are kept apart and added in proj_tc.cu's
// order: the same bits from either kernel.  Hence this kernel takes a projection whose slices each hold whole ones of that plan, an
// output or down projection only where its four ranks of 16 rows are that plan's eight of 128.  Step with proj_tc.cu alone / with sums of
// its own, for all projections / so: 7B shape 18 tokens 2851 / 2473 / 2570 us, 64 tokens 3359 / 3154 / 3231; d_model 2048, 24
// layers, 18 tokens 996 / 792 / 869, 64 tokens 1197 / 928 / 1038, 90 tokens 1396 / 1106 / 1318; four layers of d_model 5120, 18 tokens
// 541 / 475 / 500, 80 tokens 667 / 621 / 627 (96 tokens lost with sums of its own, hence 80 for matrices beyond 64 MB).  (proj_tc.cu with
// MMAs from a lone lane; from a converged warp 2 % less.)
// Which CTAs per SM, with sums of its own: 7B shape, QKV 384 CTAs, three per SM, 2886 us, 1 slice and two per SM 2894; gate/up 344, three
// 2875, two per SM, i.e. two waves, 2998; d_model 2048, 18 tokens 803, one CTA per SM and two waves 908, two per SM everywhere 838;
// stages of four k-blocks instead of two 858.  Where even three CTAs per SM are not enough (d_model 8192) proj_tc.cu takes it.
inline ProjFewPlan plan_proj_few(int m, int n, int k, bool dual, bool add, bool in_l2, int n_sms) {
  using namespace proj;
  ProjFewPlan pl{};
  pl.nt = (m + 7) / 8 * 8;
  pl.tiles = (n + (dual ? 31 : 63)) / (dual ? 32 : 64);
  pl.kb_total = k / (int)kBlockK;
  pl.splits = dual || pl.kb_total < 8 ? 1 : add ? 4 : 2;
  int q = 1;
  if (!in_l2) {
    const bool huge = (size_t)n * k * (dual ? 4 : 2) > (size_t)64 << 20;
    if (!add && pl.tiles <= 2 * n_sms && pl.tiles * pl.splits > 3 * n_sms) pl.splits = 1;
    const int ctas = pl.tiles * pl.splits, fit = pl.splits == 4 ? n_sms * 33 / 37 : n_sms;      // (clusters of four: as in plan_proj)
    while (q < 3 && ctas > q * fit) ++q;
    if (ctas > q * fit || (huge && m > 80)) return ProjFewPlan{};
    const int slices = plan_proj(m, n, k, dual, n_sms).splits;
    pl.parts = slices / pl.splits;
    if (pl.parts < 1 || (add && pl.parts * pl.splits != 8)) return ProjFewPlan{};    // (ADD: ranks of 16 rows, a sum of squares each)
  }
  pl.acc_ld = (pl.nt + 31) & ~31;
  const int n_acc = pl.parts * (dual ? 1 : 2) > 1 ? pl.parts * (dual ? 1 : 2) : 1;
  const int kb_bytes = 64 * (int)kBlockK * 2 + pl.nt * (int)kBlockK * 2, per_cta = (pl.kb_total + pl.splits - 1) / pl.splits;
  // the tile's rows on their way to the epilogue: unsplit they lie over the drained stages
  const int recv = (m + 3) / 4 * 64 * 16 * (pl.splits > 1 && pl.parts > 1 ? pl.parts : 1), beside = pl.splits > 1 ? recv : 0;
  const int most = q == 1 ? kFewSmem : 228 * 1024 / q - 2048, room = most - 1024 - beside;      // for stages (a CTA's fixed part and the system's: 2 KB)
  // All k-blocks at once where they fit, in stages of four, five or seven: as few blocks beyond the range as there can be, then as
  // few stages.
  auto fit = [&](int g) { return (per_cta + g - 1) / g * g * kb_bytes <= room; };
  pl.group = 4;
  for (int g = 5; g <= 7; g += 2)
    if (fit(g) && (per_cta + g - 1) / g * g <= (per_cta + pl.group - 1) / pl.group * pl.group) pl.group = g;
  if (!in_l2) pl.group = 2;
  const int stage_bytes = pl.group * kb_bytes, groups = (per_cta + pl.group - 1) / pl.group;
  pl.stages = room / stage_bytes;
  if (pl.stages > kFewStages) pl.stages = kFewStages;
  if (pl.stages > groups) pl.stages = groups;
  pl.ring = pl.stages < groups || pl.parts > 0;
  if (pl.stages < groups && pl.stages < 2) return ProjFewPlan{};
  pl.recv_off = beside ? pl.stages * stage_bytes : 0;
  pl.smem_bytes = pl.stages * stage_bytes + beside + 1024;
  if (pl.smem_bytes < recv + 1024) pl.smem_bytes = recv + 1024;
  pl.tmem_cols = 32;
  while (pl.tmem_cols < (n_acc > 1 ? pl.acc_ld * n_acc : pl.nt)) pl.tmem_cols <<= 1;
  // as in plan_proj, less the fixed part too: of at most sixteen CTAs the half kilobyte that may be missing from each is less than
  // 32 columns' share
  const int share = (int)((228u * 1024u * (unsigned)pl.tmem_cols + 511u) / 512u) - 2048;
  if (pl.smem_bytes < share) pl.smem_bytes = share;
  if (in_l2) {
    const int fit = pl.smem_bytes > 112 * 1024 ? 1 : 228 * 1024 / (pl.smem_bytes + 2048), per_sm = fit < 3 ? fit : 3;
    if (pl.tiles * pl.splits > per_sm * (pl.splits == 4 ? n_sms * 33 / 37 : n_sms)) return ProjFewPlan{};
  }
  return pl.smem_bytes <= most ? pl : ProjFewPlan{};
}

// ---- gate/up of many tokens on CTA pairs, gateup_pair.cu --------------------------------------------
struct GateupPairPlan {
  int pairs, passes, nt, kb_total, sub, stages, smem_bytes, tmem_cols;  // kb_total: stages' worth of sub k-blocks; pairs 0: proj_tc.cu takes it
};

// Where proj_tc.cu's plan is an unsplit one, of up to 20 MB of weights, and a CTA of a pair stages at most nine tenths of the bytes: the
// fewest tokens per pass (a multiple of 32, an MMA's on a pair) that leave no second wave.  How many that may be: a pass has about twice
// the tokens of proj_tc.cu's, and its epilogue the time they take, which short K ranges do not earn back.  18 layers, steps against
// proj_tc.cu, 337 calls of 97 to 1200 tokens in chains of 9, 16 and 18 rows, 100 and 300 cached: up to 64 tokens a pass -0.4 to -5 % at every
// width; 96 and 128 from 18 k-blocks on -0.3 to -3.6 %, at 16 of them (d_model 1024) -1.5 to +1.0 %, 0 on average; 160 where weights x k-blocks
// reach 270 MB (MB x blocks of 64: d_model 1280, d_ff 3456 338; 1536, 2048 288; below 1280, 2560 250; 1024, 4096 256) -2.7 to 0 %, below
// +0.1 to +2.6 %.  Of what this takes 1280, 3456 with passes of 160 loses while caches are short: 288 tokens, 20 cached +0.2 to +0.8 %, 100
// -0.2 to +0.4, 300 -1.6 to 0, 550 -1.2 to -0.6.
inline GateupPairPlan plan_gateup_pair(int m, int ff, int k, int n_sms) {
  using namespace proj;
  GateupPairPlan pl{};
  const ProjPlan one = plan_proj(m, ff, k, true, n_sms);
  if (one.splits > 1 || one.tiles_on_z || k % (int)kBlockK || (size_t)ff * k * 4 > (size_t)20 << 20) return pl;
  const int pairs = (ff + 127) / 128, blocks = k / (int)kBlockK;
  const int most = (size_t)ff * k * 4 * blocks >= (size_t)270 << 20 ? kPairTok : blocks >= 18 ? 128 : 64;
  for (int passes = (m + most - 1) / most; passes * pairs <= n_sms / 2; ++passes) {
    const int nt = ((m + passes - 1) / passes + 31) / 32 * 32;
    if ((m + nt - 1) / nt != passes || (pl.passes > 0 && nt >= pl.nt)) continue;
    pl.passes = passes;
    pl.nt = nt;
  }
  if (pl.passes == 0 || (128 + pl.nt / 2) * 10 > (256 + one.nt) * 9) return pl;       // (rows of a k-block that a CTA stages)
  // (220 KB: a fifth stage of two k-blocks with 96 tokens a pass, 144 tokens 628.0 -> 623.0 us a step of 18 layers of the XL shape)
  const int kb_bytes = (int)kATileBytes + pl.nt * (int)kBlockK, room = 220 * 1024;
  pl.sub = 5 * 2 * kb_bytes <= room ? 2 : 1;
  pl.kb_total = (k / (int)kBlockK + pl.sub - 1) / pl.sub;
  const int stage_bytes = pl.sub * kb_bytes;
  pl.stages = room / stage_bytes;
  if (pl.stages > pl.kb_total) pl.stages = pl.kb_total;
  if (pl.stages > kMaxStages) pl.stages = kMaxStages;
  pl.smem_bytes = pl.stages * stage_bytes + 1024;
  if (pl.smem_bytes < pl.nt * 144 + 1024) pl.smem_bytes = pl.nt * 144 + 1024;         // the finished tile, token-major
  pl.tmem_cols = pl.nt <= 32 ? 32 : pl.nt <= 64 ? 64 : pl.nt <= 128 ? 128 : 256;
  // (as in plan_proj: as large a share of an SM's shared memory as of its tensor memory)
  const int share = (int)((228u * 1024u * (unsigned)pl.tmem_cols + 511u) / 512u) - 1024;
  if (pl.smem_bytes < share) pl.smem_bytes = share;
  pl.pairs = pairs;
  return pl;
}

// ---- block-vs-cache attention, attention_block.cu -------------------------------------------------
// CTAs (a cluster) per (sequence, head) item.  The keys of an item are split where the items leave SMs idle and the cache can
// be long enough to pay for the exchange: by its capacity s_max, since the fill levels are known to the GPU only.  Heads of 64
// keep 16 warps on an item, which take 256 keys a turn; of 128, 8 warps and 128 keys.  XL shape (40 items of 64-wide heads,
// 18 layers, 18 tokens), one CTA an item / two: 592 slots, 300 filled 473 / 477 us; 2304 slots, 64 filled 462 / 472, 2200
// filled 626 / 558; 4608 slots, 4500 filled 819 / 656.  20 items, 4608 slots, two / four: 100 filled 448 / 466, 2000 filled
// 511 / 497, 4500 filled 612 / 560.  7B shape (64 items of 128-wide heads, 8 layers), one / two: 60 filled 735 / 735, 450
// filled 762 / 749, 2300 filled 864 / 816; 32 items, 4500 filled, two / four 837 / 785.
inline int attention_split(int hd, long long items, int s_max, int n_sms) {
  const int slots = hd == 128 ? 512 : 1536;
  int split = 1;
  while (split < 4 && items * split * 2 <= n_sms && s_max >= slots * split) split *= 2;
  return split;
}

// ---- QKV and attention of few tokens and few sequences, qkv_attention_few.cu ----------------------
struct QkvAttentionPlan {
  ProjFewPlan proj;
  int per_item;                // CTAs of a cluster that share an item; 0: two kernels
  int part_off, recv_off, new_off, smem_bytes;
};

// qkv: the projection's plan, in two slices with all k-blocks in shared memory (tiles of 64 rows: a head's q, k or v).  Heads of 64 whose
// items have a CTA each in attention_block.cu; one to three sequences, since the sixteen warps' parts of an item need two CTAs; and all
// clusters have to fit at once (of 148 SMs 22 take clusters of six: 132).  A token has at most 128 sums of squares (d / 16 of them).
inline QkvAttentionPlan plan_qkv_attention(const ProjFewPlan& qkv, int n_heads, int hd, int d, int n_rows, int t_len, int s_max, int n_sms) {
  using namespace proj;
  QkvAttentionPlan pl{};
  pl.proj = qkv;
  if (hd != 64 || n_heads * hd != d || d > 2048 || n_rows > 3 || t_len > 32 || qkv.stages < 1 || qkv.splits != 2 || qkv.ring || qkv.parts > 0) return pl;
  if (n_heads * 6 > n_sms * 33 / 37 || attention_split(hd, (long long)n_heads * n_rows, s_max, n_sms) > 1) return pl;
  const int per_item = 6 / n_rows, slots = (16 + per_item - 1) / per_item, ld_t = t_len < 16 ? t_len : 16;
  const int stages = qkv.stages * qkv.group * (64 * (int)kBlockK * 2 + qkv.nt * (int)kBlockK * 2), recv = (qkv.nt + 3) / 4 * 64 * 16;
  // the keys and, in the CTA that folds, the parts lie over the stages
  pl.part_off = slots * 8192;
  const int attention = pl.part_off + 16 * ld_t * (100 + 2) * 4;
  pl.recv_off = ((stages > attention ? stages : attention) + 1023) & ~1023;
  pl.new_off = pl.recv_off + ((recv + 1023) & ~1023);
  pl.smem_bytes = pl.new_off + 3 * t_len * 128 + 1024;
  if (pl.smem_bytes < qkv.smem_bytes) pl.smem_bytes = qkv.smem_bytes;
  if (pl.smem_bytes <= kFewSmem) pl.per_item = per_item;
  return pl;
}

// ---- walk of a candidate tree, kernels_tree.cu ---------------------------------------------------
// CTAs (a cluster) per image, each with a part of the codes: what a part saves on each residual has to outweigh the cluster's
// barriers, also where most drafts are accepted and there are few residuals.  26 nodes, one image, most accepted / most
// rejected: 4096 codes 9.2 / 22.9 us with one CTA, 10.4 / 19.6 with four; 8192 codes 10.8 / 34.4, 10.8 / 23.0, eight 10.9 /
// 21.2; 16384 codes, four images 17.4 / 65.6, 13.1 / 28.5, 13.3 / 24.2.  And all clusters run at once: of clusters of eight
// (one CTA per SM) 15 fit, of four 33 (16 images x 16384 codes, most rejected: 39 us with eight each, 29 with four; 40
// images, all accepted: 38 with eight, 24 with two).
inline int tree_walk_parts(int vocab, int n_images, int n_sms) {
  int S = vocab < 8192 ? 1 : vocab < 16384 ? 4 : 8;
  while (S > 1 && (long long)n_images * S > (S == 8 ? n_sms * 30 / 37 : S == 4 ? n_sms * 33 / 37 : n_sms)) S /= 2;
  return S;
}

}  // namespace vvs
