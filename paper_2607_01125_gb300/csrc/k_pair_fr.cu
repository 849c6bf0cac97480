// Host side of the few-row pair forward: which calls it serves, its split of the
// work and its tensor maps.
#include <atomic>
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

}  // namespace

// Few rows: fewer than 256, and every block's rows padded to 16 within one MMA's 256 columns.  The 128-row one-CTA kernel
// takes what is left (17 blocks of 20 rows, say).  A call (projection included) on 32 / 128 / 240 rows, this kernel
// against that one: bf16 4096 -> 4096 16 / 21 / 32 against 33 / 36 / 37 us, bf16 gated 4096 -> 14336 52 / 59 / 70 against
// 65 / 68 / 84, fp16 5120 -> 20480 (r = 32) 55 / 67 / 93 against 70 / 76 / 102.  INT4 14336 -> 4096 (r = 32): 41 / 48 / 66
// against 69 / 80 / 98 with W expanded to bf16 first.
bool pair_fr_supported(const PairArgs& a) {
  if (a.rows <= 0 || a.nseg > 1 || a.fuse_loss || a.in_scale || a.out_sumsq) return false;
  if (a.xdtype != ZOACT_DT_BF16 && a.xdtype != ZOACT_DT_FP16) return false;
  if (a.T > FR_TOK || a.nb * round16(a.T) > FR_TOK || a.rows >= FEW_ROWS) return false;
  const char* sel = std::getenv("ZOACT_PAIR_KERNEL");
  if (sel && std::strcmp(sel, "1cta") == 0) return false;
  if (a.wtype == ZOACT_DT_INT4_G128) {
    const char* isel = std::getenv("ZOACT_INT4");
    return a.xdtype == ZOACT_DT_BF16 && !(isel && std::strcmp(isel, "staged") == 0);
  }
  return a.wtype == a.xdtype;
}

int launch_pair_fr(Ctx* ctx, const PairArgs& a) {
  using namespace pairfr;
  const bool w4 = a.wtype == ZOACT_DT_INT4_G128, gated = a.W2 != nullptr;
  if (a.ydtype != a.xdtype && a.ydtype != ZOACT_DT_FP32) return ZOACT_ERR_UNSUPPORTED;
  const int nw = gated ? 2 : 1;
  FrArgs fr{};
  fr.tpad = (int)round16(a.T);
  fr.tok = a.nb * fr.tpad;
  fr.out32 = a.ydtype == ZOACT_DT_FP32;
  fr.tmem_cols = 32;
  while (fr.tmem_cols < nw * fr.tok) fr.tmem_cols *= 2;
  fr.lr_mats = gated && a.P2 != a.P ? 2 : 1;
  fr.lr_groups = fr.lr_mats * ((a.r + LR_RANKS - 1) / LR_RANKS);

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
  int per_sm = 2;
  fit(SM_SMEM / 2 - 1024);
  // Two stages only where one CTA per SM would leave a second wave of tiles (fp16 5120 -> 20480, 200 rows, 160 tiles:
  // 99.0 us a call with one CTA per SM and 3 stages, 90.2 with two CTAs and 2).
  const int64_t tiles = (a.d_out + WR - 1) / WR;
  const bool second_wave = tiles > ctx->sm_count && tiles <= 2 * ctx->sm_count;
  if (fr.tmem_cols > 256 || fr.stages < (second_wave ? 2 : 3)) {
    per_sm = 1;
    fit(CTA_SMEM);                                      // at least 3 stages of at most 64 KB, and 4 packed slots of 8 KB
  }
  const int ring = fr.stages * stage + fr.raw_slots * raw;
  int smem = FR_BARS + ring;
  if (per_sm == 1 && smem <= SM_SMEM / 2) smem = SM_SMEM / 2 + 1024;
  fr.chunk = ring / (nw * WR * 4) / 16 * 16;
  if (fr.chunk > fr.tok) fr.chunk = fr.tok;
  // K ranges: as many as fill the chip's CTA slots once, each at least four K-blocks, at most a portable cluster.  More
  // would add waves, whose prologues and epilogues nothing hides (4096 -> 14336 gated, 128 rows: 59 us a call with one
  // range per tile, 81 with two, 93 with four; 14336 -> 4096, 32 rows: 50 with two, 34 with four, 33 with eight).
  // A cluster lies within a GPC, so fewer than slots / S clusters of S run at once, and those left over are a second
  // wave: fp16 5120 -> 5120, 64 rows (40 tiles) takes 30.2 us with 7 ranges, 20.8 with 6; INT4 4096 -> 5120, 48 rows
  // 34.0 and 24.3; gated 4096 -> 2560, 80 rows (20 tiles) 33.7 and 21.0.
  int64_t splits = (int64_t)per_sm * ctx->sm_count / tiles;
  if (splits > p.num_k / 4) splits = p.num_k / 4;
  if (splits > MAX_SPLITS) splits = MAX_SPLITS;
  while (splits > 1 && tiles > clusters_at_once(ctx, (int)splits, per_sm)) --splits;
  fr.splits = (int)(splits < 1 ? 1 : splits);

  st = timing_begin(ctx);
  if (st) return st;
  st = w4 ? dispatch_fr_w4(ctx, gated, tm, p, fr, smem)
          : a.xdtype == ZOACT_DT_BF16 ? dispatch_fr_bf16(ctx, gated, tm, p, fr, smem)
                                      : dispatch_fr_fp16(ctx, gated, tm, p, fr, smem);
  if (st) return st;
  return timing_end(ctx);
}

}  // namespace zoact
