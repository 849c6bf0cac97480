// Host side of the few-row pair forward: which calls it serves, its split of the
// work and its tensor maps.
#include <atomic>
#include <cmath>
#include <cstdlib>
#include <cstring>

#include "pair_fr_kernel.cuh"

namespace zoact {

namespace pairfr {
int dispatch_fr_bf16(Ctx* ctx, bool gated, const TmaSet& tm, const Params& p, const FrArgs& fr, int smem);
int dispatch_fr_fp16(Ctx* ctx, bool gated, const TmaSet& tm, const Params& p, const FrArgs& fr, int smem);
int dispatch_fr_w4(Ctx* ctx, bool gated, const TmaSet& tm, const Params& p, const FrArgs& fr, int smem);
int fr_max_clusters(int size, int smem);
}  // namespace pairfr

namespace {

constexpr int SM_SMEM = 228 * 1024;            // shared memory of an SM, 1 KB of it reserved per CTA
using pairfr::CTA_SMEM;
constexpr int FR_TOK = 256;                    // most accumulator columns (the MMA's N)

int64_t round16(int64_t v) { return (v + 15) / 16 * 16; }

// Clusters of `size` CTAs that the device runs at once, per_sm (1 or 2) CTAs on an SM: what it answers for one CTA per SM
// (asked once per device); two per SM fit twice as many, or a cluster takes half its SMs.
int64_t clusters_at_once(const Ctx* ctx, int size, int per_sm) {
  constexpr int DEVICES = 64;
  static std::atomic<int> known[DEVICES][pairfr::MAX_SPLITS + 1];
  auto one = [&](int n) {
    const bool keep = ctx->device >= 0 && ctx->device < DEVICES;
    int v = keep ? known[ctx->device][n].load(std::memory_order_relaxed) : 0;
    if (v == 0) {
      v = pairfr::fr_max_clusters(n, SM_SMEM / 2 + 1024);
      if (keep) known[ctx->device][n].store(v, std::memory_order_relaxed);
    }
    return (int64_t)v;
  };
  if (per_sm == 1) return one(size);
  const int64_t twice = 2 * one(size), half = one((size + 1) / 2);
  return twice > half ? twice : half;
}

// Tiles, stages and K ranges of a call.
struct FrPlan {
  pairfr::FrArgs fr;
  int per_sm, smem;
  int64_t tiles;
};

FrPlan fr_plan(const Ctx* ctx, const PairArgs& a) {
  using namespace pairfr;
  const bool w4 = a.wtype == ZOACT_DT_INT4_G128, gated = a.W2 != nullptr;
  const int nw = gated ? 2 : 1;
  FrPlan p{};
  FrArgs& fr = p.fr;
  fr.tpad = (int)round16(a.T);
  fr.tok = a.nb * fr.tpad;
  fr.out32 = a.ydtype == ZOACT_DT_FP32;
  fr.tmem_cols = 32;
  while (fr.tmem_cols < nw * fr.tok) fr.tmem_cols *= 2;
  fr.lr_mats = gated && a.P2 != a.P ? 2 : 1;
  fr.lr_groups = fr.lr_mats * ((a.r + LR_RANKS - 1) / LR_RANKS);
  const int num_k = (a.d_in + BKF - 1) / BKF;

  // Two CTAs per SM where their TMEM (256 columns each) and rings fit twice; a CTA that must not share an SM takes
  // more than half of its shared memory, so that no CTA of this launch ever waits for another one's TMEM.
  const int stage = nw * W_TILE + fr.tok * BKF * 2, raw = w4 ? nw * RAW_TILE : 0;
  const int most = w4 ? 4 : MAX_STAGES;                 // INT4: the rest goes to the packed rows in flight
  auto fit = [&](int budget) {
    budget -= FR_BARS;
    fr.stages = (budget - 4 * raw) / stage;
    if (fr.stages > most) fr.stages = most;
    fr.raw_slots = w4 ? (budget - fr.stages * stage) / raw / 2 * 2 : 0;   // an even number (see the kernel)
    if (fr.raw_slots > MAX_RAW) fr.raw_slots = MAX_RAW;
  };
  p.per_sm = 2;
  fit(SM_SMEM / 2 - 1024);
  // Two stages only where one CTA per SM would leave a second wave of tiles (fp16 5120 -> 20480, 200 rows, 160 tiles:
  // 99.0 us a call with one CTA per SM and 3 stages, 90.2 with two CTAs and 2).
  p.tiles = (a.d_out + WR - 1) / WR;
  const bool second_wave = p.tiles > ctx->sm_count && p.tiles <= 2 * ctx->sm_count;
  if (fr.tmem_cols > 256 || fr.stages < (second_wave ? 2 : 3)) {
    p.per_sm = 1;
    fit(CTA_SMEM);                                      // at least 3 stages of at most 64 KB, and 4 packed slots of 8 KB
  }
  const int ring = fr.stages * stage + fr.raw_slots * raw;
  p.smem = FR_BARS + ring;
  if (p.per_sm == 1 && p.smem <= SM_SMEM / 2) p.smem = SM_SMEM / 2 + 1024;
  fr.chunk = ring / (nw * WR * 4) / 16 * 16;
  if (fr.chunk > fr.tok) fr.chunk = fr.tok;
  // K ranges: as many as fill the chip's CTA slots once, each at least four K-blocks, at most a portable cluster.  More
  // would add waves, whose prologues and epilogues nothing hides (4096 -> 14336 gated, 128 rows: 59 us a call with one
  // range per tile, 81 with two, 93 with four; 14336 -> 4096, 32 rows: 50 with two, 34 with four, 33 with eight).
  // A cluster lies within a GPC, so fewer than slots / S clusters of S run at once, and those left over are a second
  // wave: fp16 5120 -> 5120, 64 rows (40 tiles) takes 30.2 us with 7 ranges, 20.8 with 6; INT4 4096 -> 5120, 48 rows
  // 34.0 and 24.3; gated 4096 -> 2560, 80 rows (20 tiles) 33.7 and 21.0.
  int64_t splits = (int64_t)p.per_sm * ctx->sm_count / p.tiles;
  if (splits > num_k / 4) splits = num_k / 4;
  if (splits > MAX_SPLITS) splits = MAX_SPLITS;
  while (splits > 1 && p.tiles > clusters_at_once(ctx, (int)splits, p.per_sm)) --splits;
  fr.splits = (int)(splits < 1 ? 1 : splits);
  return p;
}

// Padded rows that fit one tile, and types that the kernel takes.
bool fr_supported(const PairArgs& a) {
  if (a.rows <= 0 || a.nseg > 1 || a.fuse_loss || a.in_scale || a.out_sumsq) return false;
  if (a.xdtype != ZOACT_DT_BF16 && a.xdtype != ZOACT_DT_FP16) return false;
  if (a.T > FR_TOK || a.nb * round16(a.T) > FR_TOK || a.rows >= FEW_ROWS) return false;
  return a.wtype == ZOACT_DT_INT4_G128 ? a.xdtype == ZOACT_DT_BF16 : a.wtype == a.xdtype;
}

// The other route for few rows, one-CTA tiles of 128 rows (INT4: on W expanded to bf16), in what its time depends on.
struct OneCta {
  bool stacked;               // the low-rank term as K columns of stacked rows (above rank 32 a shared input is copied)
  int64_t rows;               // of the stacked X, or of the shared one
  int slots, ka, nw;
  int64_t table_rows;         // of B_aug, both matrices
};
OneCta one_cta(const PairArgs& a) {
  OneCta o{};
  o.nw = a.W2 ? 2 : 1;
  o.stacked = !a.shared || a.r > 32;
  o.rows = o.stacked ? a.nb * a.T : a.T;
  const int64_t tile = o.rows >= FEW_ROWS ? 256 : 128;        // (copies of 256 rows go to CTA pairs)
  const int64_t span = o.stacked && a.T % tile != 0 ? (tile - 1) / a.T + 2 : 1;
  o.slots = (int)(span < a.nb ? span : a.nb);
  o.ka = aug_cols(a.r) * (a.W2 && a.P2 != a.P ? 2 : 1);
  o.table_rows = (int64_t)o.nw * (o.stacked ? a.nb : 1) * a.d_out;
  return o;
}

// Estimates of a call's time (its projection apart) by this kernel and by the other route, in us on a GB300: sums of the
// main loop or the read of W, whichever is longer (a fourth-power mean), the low-rank K-blocks or table elements, and the
// epilogue, fitted to 6000 calls drawn over d_in 64 .. 20480, d_out 8 .. 20480, 2 to 17 blocks, ranks 1 .. 256, gated ones
// (rms 8% for this kernel, 15% for the other), and to 800 without scratch.  This kernel is behind where W is small and the
// low-rank K-blocks, 1 to 2 us each to write, or the partials of many rows are most of its work: two signs of 127 rows,
// 512 -> 512, rank 4 25.5 us against 10.7, and nine blocks of 7 rows, 256 -> 1024 gated, rank 256 595 against 154.  It is
// ahead on wide layers: 32 / 128 / 240 rows, projection included, bf16 4096 -> 4096 16 / 21 / 32 against 33 / 36 / 37 us,
// gated 4096 -> 14336 52 / 59 / 70 against 65 / 68 / 84, INT4 14336 -> 4096 (r = 32) 41 / 48 / 66 against 69 / 80 / 98.
// Of 3908 16-bit calls (2092 INT4 ones) the estimates choose a slower kernel by more than 3% in 2%; they take 0.851
// (0.866) of this kernel's time alone, against 0.846 (0.864) by the better one of each.
double longer(double a, double b) {
  a *= a;
  b *= b;
  return std::sqrt(std::sqrt(a * a + b * b));
}
double fr_us(const Ctx* ctx, const PairArgs& a, const FrPlan& p) {
  const bool w4 = a.wtype == ZOACT_DT_INT4_G128;
  const pairfr::FrArgs& fr = p.fr;
  const int nw = a.W2 ? 2 : 1, S = fr.splits;
  const int64_t slots = (int64_t)p.per_sm * ctx->sm_count;
  const double waves = (double)((p.tiles * S + slots - 1) / slots), tok = fr.tok / 64.0;
  const double nm = ((a.d_in + pairfr::BKF - 1) / pairfr::BKF + S - 1) / S, nl = a.nb * ((fr.lr_groups + S - 1) / S);
  const double mb = (w4 ? 0.5e-6 : 2e-6) * a.d_out * (double)a.d_in * nw;
  const double block = w4 ? (p.per_sm == 1 ? 0.24 * nw + 0.11 * tok : 0.37 * nw + 0.16 * tok)
                          : (p.per_sm == 1 ? 0.13 * nw + 0.093 * tok : 0.18 * nw + 0.17 * tok);
  const double lr = 1.1 + (nw == 2 && fr.lr_mats == 1 ? 0.54 : 0.0) + 0.2 * ((fr.tpad + 63) / 64) + (a.r % 4 ? 0.15 : 0.0);
  const double out = S == 1 ? tok * nw : 6.4 * tok * nw / S + 1.8 * ((fr.tok + fr.chunk - 1) / fr.chunk);
  return (w4 ? 2.8 : 1.2) + longer(waves * nm * block, (w4 ? 0.76 : 0.15) * mb) + waves * (nl * lr + out);
}
double one_cta_us(const Ctx* ctx, const PairArgs& a, const OneCta& o) {
  const int bn = o.nw == 2 ? 128 : 256, num_k = (a.d_in + 63) / 64;
  const int64_t tiles = (o.rows + 127) / 128 * ((a.d_out + bn - 1) / bn);
  const double waves = (double)((tiles + ctx->sm_count - 1) / ctx->sm_count);
  const double cols = a.d_out < bn ? (double)a.d_out / bn : 1.0;
  const double rt = a.r <= 4 ? 4 : a.r <= 8 ? 8 : a.r <= 16 ? 16 : 32, mb = 2e-6 * a.d_out * (double)a.d_in * o.nw;
  if (!ctx->may_allocate) return 3.5 + 0.27 * waves * num_k + waves * rt * (0.35 * cols + 0.03) + 0.06 * mb;
  const double main = (o.nw == 2 ? 0.33 : 0.3) * waves * (num_k + o.slots * (o.ka / 64));
  double us = 5.6 + 0.9 * waves * cols + longer(main, 0.2 * mb) + (a.r % 4 ? 0.62e-5 : 0.12e-5) * o.table_rows * o.ka +
              2.4e-5 * o.rows * o.slots * o.ka;
  if (!o.stacked) us += waves * ((a.nb + 1) / 2) * (1.6 + rt * cols * (o.nw == 2 ? 0.57 : 0.35));
  if (a.shared && o.stacked) us += 2.7 * a.nb;                     // copies of X and P
  if (a.wtype == ZOACT_DT_INT4_G128) us += 0.3 * mb + 0.7 * o.nw;
  return us;
}

}  // namespace

// ZOACT_PAIR_KERNEL=few / =1cta: this kernel wherever it can run / never; ZOACT_INT4=staged: not on INT4 weights.
bool pair_fr_possible(const PairArgs& a) {
  if (!fr_supported(a)) return false;
  const char* sel = std::getenv("ZOACT_PAIR_KERNEL");
  if (sel && std::strcmp(sel, "1cta") == 0) return false;
  const char* isel = std::getenv("ZOACT_INT4");
  return !(a.wtype == ZOACT_DT_INT4_G128 && isel && std::strcmp(isel, "staged") == 0);
}

bool pair_fr_chosen(const Ctx* ctx, const PairArgs& a) {
  if (!pair_fr_possible(a)) return false;
  const char* sel = std::getenv("ZOACT_PAIR_KERNEL");
  if (sel && std::strcmp(sel, "few") == 0) return true;
  // fp32 outputs keep this kernel's three-part low-rank term: the other route's two parts leave out 2^-16 of |T||P|, which
  // a 16-bit output cannot show (its form without scratch sums in fp32)
  if (a.ydtype == ZOACT_DT_FP32 && ctx->may_allocate) return true;
  const OneCta o = one_cta(a);
  // (0.9: about as many calls lose by an error of the estimates one way as the other)
  return one_cta_us(ctx, a, o) >= 0.9 * fr_us(ctx, a, fr_plan(ctx, a)) || !tile_route_ready(ctx, a);
}

// The sizes are launch_pair_tc's.
bool tile_route_ready(const Ctx* ctx, const PairArgs& a) {
  if (!ctx->may_allocate) return true;                              // (its form without scratch)
  const OneCta o = one_cta(a);
  int queries = 0;                                                  // distinct ones of the perturbed blocks
  for (int b = 0; b < a.nb; ++b) {
    bool seen = a.coef[b] == 0.f;
    for (int i = 0; i < b; ++i) seen = seen || (a.coef[i] != 0.f && a.qry[i] == a.qry[b]);
    queries += !seen;
  }
  const bool one_p = !a.W2 || a.P2 == a.P, pairs_of_ctas = o.rows >= FEW_ROWS;
  const bool blocks16 = pairs_of_ctas && !o.stacked && a.nb >= 2 && dtype_size(a.ydtype) == 2;
  const bool mirror = blocks16 && a.nb == 2 && a.qry[0] == a.qry[1] && a.coef[1] == -a.coef[0] && a.coef[0] != 0.f;
  const int rt = a.r <= 4 ? 4 : a.r <= 8 ? 8 : a.r <= 16 ? 16 : 32;
  const size_t z = blocks16 && !mirror && one_p ? z_table_words(rt, a.d_out) : (size_t)a.r * a.d_out;
  const size_t copy = (size_t)a.T * a.d_in * 2 + (size_t)(one_p ? 1 : 2) * a.T * a.r * sizeof(float);
  const size_t w_bytes = a.wtype == ZOACT_DT_INT4_G128 ? (size_t)a.d_out * a.d_in * 2 : 0;
  bool ok = scratch_ready(ctx, SLOT_AUG_A, (size_t)o.rows * o.slots * o.ka * 2) &&
            scratch_ready(ctx, SLOT_AUG_B, (size_t)o.table_rows * o.ka * 2) &&
            (o.stacked || scratch_ready(ctx, SLOT_AUG_Z, o.nw * queries * z * sizeof(float))) &&
            (!(a.shared && o.stacked) || scratch_ready(ctx, SLOT_STACKED_X, a.nb * copy + 1024)) &&
            scratch_ready(ctx, SLOT_WDQ0, w_bytes) && (!a.W2 || scratch_ready(ctx, SLOT_WDQ1, w_bytes));
  if (pairs_of_ctas) {                                              // a split tail's partials
    const int64_t pairs = ctx->sm_count / 2, bn = a.W2 ? 128 : 256;
    const int64_t rem = (o.rows + 255) / 256 * ((a.d_out + bn - 1) / bn) % pairs;
    const int64_t split = rem > 0 ? (pairs / rem < 4 ? pairs / rem : 4) : 0;
    if (split >= 2 && ((a.d_in + 63) / 64 + o.slots * (o.ka / 64)) / split >= 4)
      ok = ok && scratch_ready(ctx, SLOT_SK_PART, (size_t)pairs * 2 * 128 * 256 * sizeof(float));
  }
  return ok;
}

int launch_pair_fr(Ctx* ctx, const PairArgs& a) {
  using namespace pairfr;
  const bool w4 = a.wtype == ZOACT_DT_INT4_G128, gated = a.W2 != nullptr;
  if (a.ydtype != a.xdtype && a.ydtype != ZOACT_DT_FP32) return ZOACT_ERR_UNSUPPORTED;
  const FrPlan plan = fr_plan(ctx, a);
  const FrArgs& fr = plan.fr;
  const int smem = plan.smem;

  TmaSet tm;
  int st = encode_tmap_2d_16bit(&tm.a, a.X, a.xdtype, a.rows, a.d_in, fr.tpad);
  if (st) return st;
  if (w4) {
    st = encode_tmap_2d_int(&tm.b, a.W, 1, a.d_out, a.d_in / 2, BKF / 2, WR);
    if (!st && gated) st = encode_tmap_2d_int(&tm.b2, a.W2, 1, a.d_out, a.d_in / 2, BKF / 2, WR);
  } else {
    st = encode_tmap_2d_16bit(&tm.b, a.W, a.wtype, a.d_out, a.d_in, WR);
    if (!st && gated) st = encode_tmap_2d_16bit(&tm.b2, a.W2, a.wtype, a.d_out, a.d_in, WR);
  }
  if (st) return st;
  if (!gated) tm.b2 = tm.b;
  tm.aa = tm.ba = tm.ba2 = tm.y = tm.y16 = tm.s = tm.s2 = tm.a;   // not used

  Params p{};
  p.P = a.P; p.C = a.C; p.P2 = a.P2; p.C2 = a.C2; p.Y = a.Y;
  p.rows = a.rows; p.T = a.T; p.d_in = a.d_in; p.d_out = a.d_out; p.r = a.r;
  p.shared = a.shared; p.act = a.act; p.seed = a.seed;
  p.nb = a.nb;
  for (int b = 0; b < a.nb; ++b) { p.coef[b] = a.coef[b]; p.qry[b] = a.qry[b]; }
  p.layer_id = a.layer_id; p.layer_id2 = a.layer_id2;
  p.num_k = (a.d_in + BKF - 1) / BKF;
  p.Ws = static_cast<const __half*>(a.w_scales);
  p.Ws2 = static_cast<const __half*>(a.w_scales2);
  p.status = ctx->d_status;
  auto al16 = [](const void* q) { return ((uintptr_t)q & 15u) == 0; };
  p.vec_ok = al16(a.C) && al16(a.C2) && al16(a.P) && al16(a.P2);

  st = timing_begin(ctx);
  if (st) return st;
  st = w4 ? dispatch_fr_w4(ctx, gated, tm, p, fr, smem)
          : a.xdtype == ZOACT_DT_BF16 ? dispatch_fr_bf16(ctx, gated, tm, p, fr, smem)
                                      : dispatch_fr_fp16(ctx, gated, tm, p, fr, smem);
  if (st) return st;
  return timing_end(ctx);
}

}  // namespace zoact
