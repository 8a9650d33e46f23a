// Tile, thread split and work split of the float32 MTTKRP (simt_mttkrp.cu): host
// arithmetic on the shape, the rank and the scratch size alone.
#pragma once

#include <algorithm>

#include "nncp_internal.cuh"

namespace nncp {

namespace {

constexpr int kBK = 32;        // contraction elements per step
constexpr int kThreadsMax = 256;  // computing threads; the feeder warp comes after them
constexpr int kStages = 3;
constexpr int kTM = 4;         // output rows per thread
constexpr int kTabs = 4;       // step descriptors in flight
constexpr int kSmemMax = 232448;  // 227 KB per CTA on sm_103a
constexpr int kSmemSM = 233472;   // 228 KB per SM, 1 KB of it reserved per CTA
constexpr int kStaticSmem = 512; // descriptors (checked below)

struct SimtArgs {
  const float* X;
  long long L, I, K;
  int R, RP, ld;          // rank columns; padded to whole groups of eight; row stride of H and out
  int CG, RGH, KG;        // rank groups, row groups, splits of a step
  int bm_log2;            // BM = 32 RGH
  int tl;                 // threads that load: the most whole pairs of computing warps
  int b_all;              // the computing threads load the factor rows too
  int gsh;                // 2^gsh lanes copy a factor row (all of it in one go when vecb)
  int fk, fc;             // threads / (RP / 4) and the remainder
  int vecx, vecb, veco, evict;
  int nm;                 // contracted modes, fastest first
  int dim[kMaxModes];     // their lengths
  int dstep, mag0, magl;  // 32 mod dim[0]; ceil(2^16 / dim[0]) and / L below 32, else 0
  long long rstep;        // 32 / dim[0]
  const float* H[kMaxModes];
  long long lstep, qstep;  // 32 mod L, 32 / L
  int nrest_max;           // rest rows a stage has room for
  int red_pairs;           // column pairs per round of the KG sums (1, 2 or 4)
  int x_floats, stage_floats;
  long long nk;            // steps per whole tile
  long long whole;         // tiles taken whole
  long long U2;            // steps of the tiles cut into runs
  int G2, two;             // runs; partial slots per run (1 or 2)
  float* out;
  float* slots;
  long long slot_floats;   // min(BM, I) x R
  int seg;                 // steps per segment of a long unsplit run (0: the whole run)
};

inline long long cdiv(long long a, long long b) { return (a + b - 1) / b; }

struct SimtPlan {
  SimtArgs a;
  int BM, threads, grid;
  size_t smem;
  double cost;  // work of the busiest SM
};

// The plan with tiles of 32 RGH = 32 << c rows, from `base`, which holds the fields
// that no tile height changes; false: it does not fit.
inline bool plan_tile(const SimtPlan& base, int c, size_t cap, int num_sms, SimtPlan* t) {
  *t = base;
  SimtArgs& b = t->a;
  b.RGH = 1 << c;
  b.bm_log2 = 5 + c;
  t->BM = 32 << c;
  if (8 * b.RGH * b.CG > kThreadsMax) return false;
  // splitting a step further than over four warps only shortens each one's
  // share of it: 301 x 257 x 199, R = 20, 72 us at eight warps against 68
  b.KG = 1;
  while (b.KG < 8 && 8 * b.RGH * b.CG * b.KG * 2 <= kThreadsMax / 2) b.KG *= 2;
  const int computing = 8 * b.RGH * b.CG * b.KG;
  t->threads = (computing + 31) / 32 * 32;
  b.tl = t->threads / 64 * 64;
  const int rest = (b.nm - 1) * b.nrest_max;
  // more copies of factor rows than a warp issues in a step's time
  b.b_all = (kBK + rest) * (b.R % 4 == 0 ? b.R / 4 : b.R) > 32 * 16;
  b.fk = t->threads / (b.RP / 4);
  b.fc = t->threads % (b.RP / 4);
  b.x_floats = t->BM * kBK;
  b.stage_floats = b.x_floats + (kBK + rest) * b.RP;
  b.red_pairs = 4;
  while (b.red_pairs > 1 && computing / 2 * b.red_pairs * kTM * 2 > b.stage_floats) b.red_pairs /= 2;
  t->smem = (size_t)kStages * b.stage_floats * sizeof(float);
  if (t->smem > (size_t)(kSmemMax - kStaticSmem)) return false;
  // CTAs per SM at once: shared memory, and the registers of five warps (96 a
  // thread) on each of its four schedulers
  const int occ = std::max(1, std::min((int)(kSmemSM / (t->smem + kStaticSmem + 1024)),
                                       20 / (t->threads / 32 + 1)));
  const long long G = (long long)num_sms * occ, gx = cdiv(b.I, t->BM);
  long long left = gx % G;
  if (left * 10 >= G * 9) left = 0;  // a wave nine tenths full is left whole
  b.whole = gx - left;
  b.slot_floats = std::min<long long>(t->BM, b.I) * b.R;
  if (left > 0) {
    // at least four steps per run; one slot per run where runs end with tiles
    long long g2 = std::max(left, std::min(G, left * b.nk / 4));
    const long long slots = (long long)(cap / (size_t)b.slot_floats);
    if (g2 % left != 0 && 2 * g2 > slots) g2 = left * (g2 / left);
    if (g2 % left == 0 && g2 > slots) g2 = left * std::max(1LL, slots / left);
    if (g2 <= left) {
      b.whole = gx;
    } else {
      b.U2 = left * b.nk;
      b.G2 = (int)g2;
      b.two = g2 % left != 0;
    }
  }
  t->grid = (int)std::max<long long>(std::min(G, b.whole), b.G2);
  const long long run = std::max(b.whole ? b.nk : 0, b.G2 ? std::min(b.nk, cdiv(b.U2, b.G2)) : 0);
  // A run is one chain of float32 additions per output (KG of them where steps are split),
  // whose error grows with the square root of its length.  The kernel before this one cut
  // the contraction into `parts` chunks; whole runs of more than 1.25 times that length
  // were up to 1.95 times as far from float64 (301 x 257 x 199 at R = 20, root -> {2, 3}:
  // 2.6e-7, 1.3e-7 in segments of 160).  Others stay whole, since the form with segments
  // costs more than its flushes where a thread copies 16 bytes along the contraction:
  // 512^3 at R = 32, root -> {2, 3} 250 -> 270 us, 40000 x 48 x 40 at R = 16 92 -> 105;
  // 301 x 257 x 199 45.3 -> 45.5.
  const long long tiles = cdiv(b.I, 128) * cdiv(b.R, 32);
  const long long parts = std::max(1LL, std::min(cdiv(4LL * num_sms, tiles), cdiv(b.K, 256)));
  const long long chain = std::min(b.K, run * kBK);
  if (b.KG == 1 && run > 5 && tiles < 4LL * num_sms && (double)chain * parts > 1.25 * b.K) b.seg = run > 32 ? 10 : 5;
  const double steps = (double)cdiv(b.whole, G) * b.nk + (b.G2 ? (double)cdiv(b.U2, b.G2) : 0.0);
  // each whole tile ends with log2(KG) rounds of sums over its rows: with four steps a
  // tile (4000 x 21 x 8 x 14 at R = 8, root -> {1, 2}) eight splits of 32 rows take
  // 47.8 us, one of 256 rows 18.8
  double rounds = 0.0;
  for (int k = 1; k < b.KG; k *= 2) rounds += (double)cdiv(b.whole, G);
  t->cost = (steps * (t->BM + 24) + rounds * t->BM) * (double)cdiv(t->grid, num_sms) * (occ == 1 ? 1.15 : 1.0);
  return true;
}

// The plan of one MTTKRP; cap: floats of scratch for partial tiles.
inline bool plan_simt(int64_t L, int64_t I, int64_t Q, const KrpDesc& KL, const KrpDesc& KQ, int R,
                      size_t cap, int num_sms, SimtPlan* pl) {
  SimtPlan base = {};
  SimtArgs& a = base.a;
  a.L = L;
  a.I = I;
  a.K = (long long)L * Q;
  a.R = R;
  a.nk = cdiv(a.K, kBK);
  for (const KrpDesc* d : {&KL, &KQ})
    for (int m = 0; m < d->nm; ++m) {
      if (a.nm == kMaxModes) return false;
      a.dim[a.nm] = (int)d->dim[m];
      a.H[a.nm++] = d->H[m];
    }
  if (a.nm < 1) return false;
  a.dstep = kBK % a.dim[0];
  a.rstep = kBK / a.dim[0];
  a.mag0 = a.dim[0] < kBK ? (65535 + a.dim[0]) / a.dim[0] : 0;
  a.magl = L < kBK ? (int)((65535 + L) / L) : 0;
  a.lstep = kBK % L;
  a.qstep = kBK / L;
  a.nrest_max = a.nm > 1 ? std::min(kBK, (kBK - 1) / a.dim[0] + 2) : 0;
  a.CG = (R + 7) / 8;
  a.RP = 8 * a.CG;
  // tile rows: the least work for the busiest SM, a step costing its rows plus the
  // part that does not depend on them (24)
  bool found = false;
  for (int c = 0; c < 4; ++c) {
    SimtPlan t;
    if (!plan_tile(base, c, cap, num_sms, &t)) break;
    if (!found || t.cost < pl->cost) *pl = t;
    found = true;
  }
  return found;
}

// Scratch (floats) that a context sets aside for the partial tiles of one MTTKRP: chunks
// of at least 256 elements for four tiles of 128 rows x 32 ranks per SM.  Outputs of few
// rows leave most of the GPU idle unless they are cut finely, and their partials are
// small: fine, chunks of 128 elements for four tiles of 128 rows per SM.  (Longer outputs
// lose with what finer cuts they have room for: 1205 x 34 x 219 at R = 67, root -> {1, 2},
// 78.5 us whole and 94 in runs.  11 rows of 41 x 64 x 14 x 11 at R = 81: 100 us in coarse
// chunks, 34 in fine ones.)
constexpr long long kFewRows = 512;
inline size_t scratch_floats(long long K, long long I, int R, int num_sms, bool fine) {
  if (fine && I > kFewRows) return 0;
  const long long tiles = cdiv(I, 128) * (fine ? 1 : cdiv(R, 32)), target = 4LL * num_sms;
  if (tiles >= target) return 0;
  const long long C = std::min(cdiv(target, tiles), cdiv(K, fine ? 128 : 256));
  return C > 1 ? (size_t)C * I * R : 0;
}

}  // namespace

}  // namespace nncp
