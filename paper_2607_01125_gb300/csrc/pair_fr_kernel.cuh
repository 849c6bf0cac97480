// Pair forward of few rows (up to 256 padded rows: short sequences), 16-bit or
// INT4 weights: the same computation as pair_tc_kernel with the roles of the
// operands exchanged.
//
// With few rows the frozen weight is all there is to read, so the kernel is
// bound by HBM (INT4: by the dequantisation) and every SM has to stream its share
// of W.  A tile is 128 rows of W (the MMA's M) by every output row (its N: the
// blocks' T rows, each block padded to 16; a shared input is loaded once per
// block): W is read once, X's few rows come from L2, and the accumulator's TMEM
// lanes are output columns.  K is split over the S CTAs of a cluster, so that 32
// tiles (4096 outputs) still fill the chip; each CTA leaves its fp32 partial in
// its own shared memory and CTA c adds the S partials of its share of the rows
// over distributed shared memory, in K order (the result does not depend on
// scheduling, and needs no scratch).
//
// The low-rank term (C + c_b Z_b) p goes through the same MMAs as extra K-blocks
// whose operands the idle epilogue warps write into ring stages, so no launch
// prepares them: with v = hi + mid + lo in bf16 (24 bits), a K-block holds eight
// ranks' products T_hi P_hi, T_hi P_mid, T_mid P_hi, T_hi P_lo, T_lo P_hi and
// T_mid P_mid, which leave out 2^-24 of |T||P| -- fp32's own rounding.  Block b's
// K-blocks are multiplied into its own accumulator columns only.  The CTAs of a
// cluster share them out, each after its first LR_AT K-blocks of W (the ring's
// first loads are then under way while Z is drawn).
//
// Warp 0 loads X (and 16-bit W) by TMA into a ring of 64-wide K-blocks, warp 1
// issues the MMAs, warps 2-9 write the low-rank operands and run the epilogue.
// INT4: warp 10 loads packed rows by TMA into a ring of their own, and warps 2-9
// turn each K-block into the 128-byte-swizzled bf16 tile (q s exact in fp32,
// rounded once).  Two CTAs share an SM where the rings fit twice (more bytes in
// flight, and one CTA's epilogue beside the other's main loop).
//
// Measured on GB300, calls with their projection, against the kernel that served these calls before (128 x 256 tiles,
// no K split, INT4 dequantised by four warps that kept 8 KB in flight):
//   bf16 4096 -> 4096, 32 rows, r = 16              35.3 -> 16.0 us
//   bf16 gated 4096 -> 14336, 200 rows, r = 16      83.9 -> 66.9 us
//   INT4 14336 -> 4096, 128 rows, r = 32             396 -> 48.1 us
// A read of 117 MB (14336 -> 4096, 32 rows) takes 33 us with its projection, of which ~26 are what a plain read of as
// much takes.  INT4 is bound by the hand-over of dequantised stages, not by its arithmetic: a form with a third fewer
// ALU instructions measured the same.  The low-rank term as fp32 dot products in the epilogue took 57 us more at 200
// gated rows; prefetching W into L2, before the dependency wait or 8 .. 32 K-blocks ahead, gained nothing or lost.
#pragma once
#include <type_traits>

#include "pair_tc2_kernel.cuh"

namespace zoact {
namespace pairfr {

using pairtc::Params;
using pairtc::TmaSet;

constexpr int WR = 128;                        // W rows per tile (per matrix)
constexpr int BKF = 64;                        // K columns per block
constexpr int W_TILE = WR * BKF * 2;           // 16-bit W tile of one K-block
constexpr int RAW_TILE = WR * BKF / 2;         // packed INT4 W tile of one K-block
constexpr int MAX_STAGES = 8, MAX_RAW = 12;
constexpr int WORK_WARPS = 8, WORK_THREADS = 32 * WORK_WARPS;
constexpr int WORK_BAR = 1;                    // named barrier of the work warps
constexpr int FR_BARS = 512;                   // shared-memory bytes kept for FrShared
constexpr int LR_RANKS = 8;                    // ranks per low-rank K-block (six products each: 48 of 64 columns)
constexpr int LR_AT = 4;                       // K-blocks of W that a CTA takes ahead of its low-rank ones
constexpr int MAX_SPLITS = 8;                  // a portable cluster
constexpr int CTA_SMEM = 232448;               // most shared memory that one CTA may use
__host__ __device__ constexpr int fr_threads(bool w4) { return 64 + WORK_THREADS + (w4 ? 32 : 0); }

struct FrArgs {
  int tpad;         // rows of one block padded to a multiple of 16
  int tok;          // nb * tpad: the MMA's N
  int splits;       // CTAs per cluster (K ranges)
  int stages, raw_slots;
  int chunk;        // accumulator columns whose partials fit in shared memory at once (a multiple of 16)
  int tmem_cols;    // power of two >= matrices * tok
  int lr_mats;      // 2: gate and up have their own projections (a low-rank K-block serves one of them)
  int lr_groups;    // low-rank K-blocks of one evaluation block
  int out32;        // Y is fp32
};

struct FrShared {
  uint64_t full[MAX_STAGES], empty[MAX_STAGES];
  uint64_t raw_full[MAX_RAW], raw_empty[MAX_RAW];
  uint64_t done;
  uint32_t tmem_base;
  int abort_flag;
  int lr_ok;
};
static_assert(sizeof(FrShared) <= FR_BARS, "barrier block outgrew its shared-memory slot");

__device__ __forceinline__ float ld_dsmem(uint32_t saddr, uint32_t rank) {
  float v;
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(pairtc::tc2::map_to(saddr, rank)) : "memory");
  return v;
}
__device__ __forceinline__ void mbar_arrive_n(uint32_t bar, uint32_t n) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(n) : "memory");
}
__device__ __forceinline__ void st_shared_v2(uint32_t addr, uint2 v) {
  asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(addr), "r"(v.x), "r"(v.y) : "memory");
}

// Low-rank K-block i of a CTA whose first group is g0: evaluation block, matrix (own projections only) and first
// rank.  A group is the K-blocks of all evaluation blocks for the same ranks: a CTA takes whole groups, so that every
// block's sums run in the same order (two signs with eps = 0 stay bit-identical).
struct LowrankBlock {
  int b, mat, j0;
};
__device__ __forceinline__ LowrankBlock lowrank_block(int nb, int r, int g0, int i) {
  const int per = (r + LR_RANKS - 1) / LR_RANKS;
  const int g = g0 + i / nb;
  LowrankBlock l;
  l.b = i % nb;
  l.mat = g / per;
  l.j0 = (g - l.mat * per) * LR_RANKS;
  return l;
}

// Four consecutive ranks' operand columns of row `row`: the six products' parts of v at columns 8 term + 4 quad
// (W side: hi hi mid hi lo mid; X side: hi mid hi lo hi mid), and this quad's share of the zero columns 48 .. 63.
__device__ __forceinline__ void write_lowrank(uint32_t tile, int row, int quad, const float* v, bool w_side) {
  __nv_bfloat16 h[4], m[4], l[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    h[i] = __float2bfloat16_rn(v[i]);
    const float rest = v[i] - __bfloat162float(h[i]);          // exact
    m[i] = __float2bfloat16_rn(rest);
    l[i] = __float2bfloat16_rn(rest - __bfloat162float(m[i]));
  }
  auto pack = [](const __nv_bfloat16* a) {
    return make_uint2((uint32_t)__bfloat16_as_ushort(a[0]) | ((uint32_t)__bfloat16_as_ushort(a[1]) << 16),
                      (uint32_t)__bfloat16_as_ushort(a[2]) | ((uint32_t)__bfloat16_as_ushort(a[3]) << 16));
  };
  const uint2 hi = pack(h), mid = pack(m), lo = pack(l);
  auto at = [&](int term) { return tile + pairtc::sw128_off(row, term) + 8u * (uint32_t)quad; };
  st_shared_v2(at(0), hi);
  st_shared_v2(at(1), w_side ? hi : mid);
  st_shared_v2(at(2), w_side ? mid : hi);
  st_shared_v2(at(3), w_side ? hi : lo);
  st_shared_v2(at(4), w_side ? lo : hi);
  st_shared_v2(at(5), mid);
  st_shared_v2(at(6), make_uint2(0u, 0u));
  st_shared_v2(at(7), make_uint2(0u, 0u));
}

// T = C + c Z of ranks j .. j + 3 of output column n (zero past r or d_out).
__device__ __forceinline__ void table_quad(float* t, const float* __restrict__ C, uint32_t layer, int64_t n, bool ok,
                                           int j, int r, uint64_t seed, float c, uint64_t q, bool vec) {
#pragma unroll
  for (int i = 0; i < 4; ++i) t[i] = 0.f;
  if (!ok) return;
  const int64_t e = n * r + j;
  if (vec && (r & 3) == 0) {
    if (j >= r) return;
    const float4 cv = *reinterpret_cast<const float4*>(C + e);
    float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
    if (c != 0.f) z = z_normals4(seed, layer, q, (uint64_t)(e >> 2));
    t[0] = fmaf(c, z.x, cv.x); t[1] = fmaf(c, z.y, cv.y); t[2] = fmaf(c, z.z, cv.z); t[3] = fmaf(c, z.w, cv.w);
    return;
  }
#pragma unroll 1
  for (int i = 0; i < 4 && j + i < r; ++i) {
    const float z = c != 0.f ? z_select(z_normals4(seed, layer, q, (uint64_t)((e + i) >> 2)), (int)((e + i) & 3)) : 0.f;
    const float v = fmaf(c, z, C[e + i]);
    if (i == 0) t[0] = v; else if (i == 1) t[1] = v; else if (i == 2) t[2] = v; else t[3] = v;
  }
}

// The operands of one low-rank K-block into a ring stage, by the work threads: T's 128 rows (gate, up), and the
// block's padded rows of P.
template <bool GATED>
__device__ __forceinline__ void fill_lowrank(const Params& prm, const FrArgs& fr, const LowrankBlock& l, uint32_t sw,
                                             uint32_t sx, int n0, int wt) {
  const int quad = wt & 1, j = l.j0 + 4 * quad, r = prm.r;
  const bool vec = prm.vec_ok != 0;
  const float c = prm.coef[l.b];
  const uint64_t q = prm.qry[l.b];
  {
    const int row = wt >> 1;
    const int64_t n = n0 + row;
    const bool ok = n < prm.d_out;
    float t[4];
    if (!GATED || fr.lr_mats == 1 || l.mat == 0) {
      table_quad(t, prm.C, prm.layer_id, n, ok, j, r, prm.seed, c, q, vec);
      write_lowrank(sw, row, quad, t, true);
    }
    if (GATED && (fr.lr_mats == 1 || l.mat == 1)) {
      table_quad(t, prm.C2, prm.layer_id2, n, ok, j, r, prm.seed, c, q, vec);
      write_lowrank(sw + W_TILE, row, quad, t, true);
    }
  }
  const float* P = l.mat ? prm.P2 : prm.P;
  const int64_t row0 = prm.shared ? 0 : (int64_t)l.b * prm.T;
  for (int t = wt >> 1; t < fr.tpad; t += WORK_THREADS / 2) {
    float p[4] = {0.f, 0.f, 0.f, 0.f};
    if (t < prm.T) {
      const float* src = P + (row0 + t) * r + j;
      if (vec && (r & 3) == 0) {
        if (j < r) {
          const float4 v = *reinterpret_cast<const float4*>(src);
          p[0] = v.x; p[1] = v.y; p[2] = v.z; p[3] = v.w;
        }
      } else {
#pragma unroll
        for (int i = 0; i < 4; ++i)
          if (j + i < r) p[i] = src[i];
      }
    }
    write_lowrank(sx, l.b * fr.tpad + t, quad, p, false);
  }
}

// The bf16 parts of an INT4 scale (fp16): s = hi + lo exactly (11 bits = 8 + 3).  A non-finite scale keeps lo = 0, so
// that its products stay what hi gives.
__device__ __forceinline__ void split_scale(float s, __nv_bfloat162& hi, __nv_bfloat162& lo) {
  const __nv_bfloat16 h = __float2bfloat16_rn(s);
  const float rest = s - __bfloat162float(h);
  hi = __halves2bfloat162(h, h);
  const __nv_bfloat16 l = __float2bfloat16_rn(isfinite(rest) ? rest : 0.f);
  lo = __halves2bfloat162(l, l);
}

// Eight INT4 elements of a word (element j in bits 4j .. 4j + 3, two's complement) times s = hi + lo, in K order as 8
// bf16, each q s rounded once: v = 128 + 8 + q is exact in bf16 (0x4300 | nibble ^ 8), q = v - 136 too, q lo has at
// most 7 bits, so the one rounding is that of fma(q, hi, q lo).  In 16-bit pairs throughout: the fp32 form of the
// CTA-pair kernel needs five more conversions per word.
__device__ __forceinline__ uint4 dequant8_bf16(uint32_t w, __nv_bfloat162 hi, __nv_bfloat162 lo) {
  const uint32_t x = w ^ 0x88888888u;
  const __nv_bfloat162 c136 = __floats2bfloat162_rn(136.0f, 136.0f);
  uint32_t p[4];                                       // elements (i, i + 4)
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const uint32_t v = ((x >> (4 * i)) & 0x000F000Fu) | 0x43004300u;
    const __nv_bfloat162 q = __hsub2(*reinterpret_cast<const __nv_bfloat162*>(&v), c136);
    const __nv_bfloat162 r = __hfma2(q, hi, __hmul2(q, lo));
    p[i] = *reinterpret_cast<const uint32_t*>(&r);
  }
  return make_uint4(__byte_perm(p[0], p[1], 0x5410), __byte_perm(p[2], p[3], 0x5410),
                    __byte_perm(p[0], p[1], 0x7632), __byte_perm(p[2], p[3], 0x7632));
}

// T16: the 16-bit activation type (and 16-bit output type).
template <typename T16, bool GATED, bool W4>
__global__ void __launch_bounds__(fr_threads(W4), 2)
pair_fr_kernel(const __grid_constant__ TmaSet tm, const __grid_constant__ Params prm, const FrArgs fr) {
  constexpr int NW = GATED ? 2 : 1;
  constexpr int AB = std::is_same<T16, __nv_bfloat16>::value ? 1 : 0;
  // A stage's arrivals: the producer's, and those of the warps that dequantise it (INT4) or write its low-rank operands
  // (16-bit W's K-blocks: one more by the producer).  The producer arrives on every stage, so that none is freed before
  // it has waited for it: every waiter then sees each phase of a barrier that it waits on, or the one before.
  constexpr int WORK_ARRIVALS = W4 ? WORK_WARPS / 2 : 1;
  static_assert(!W4 || AB == 1, "INT4 weights come with bf16 activations");
  extern __shared__ __align__(1024) uint8_t smem[];
  if (tc::smem_u32(smem) & 1023u) {       // the swizzled tiles need it; uniform over the launch
    if (threadIdx.x == 0) record_error(prm.status, ZOACT_ERR_UNSUPPORTED);
    return;
  }
  const int x_bytes = fr.tok * BKF * 2;
  const int stage_bytes = NW * W_TILE + x_bytes;       // a multiple of 1024 (tok a multiple of 16)
  uint8_t* raw = smem + fr.stages * stage_bytes;
  FrShared* ss = reinterpret_cast<FrShared*>(raw + (W4 ? fr.raw_slots * NW * RAW_TILE : 0));
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  volatile int* abort_flag = &ss->abort_flag;
  const int S = fr.splits;
  const int rank = (int)pairtc::tc2::cluster_rank();
  const int n0 = (int)(blockIdx.x / S) * WR;
  // this CTA's K-blocks of W [m0, m0 + nm) (the host leaves each CTA at least one) and low-rank ones (groups g0 ..); in
  // order: `at` of W (no more than the ring holds: the work warps enter it there), the low-rank ones, the rest of W
  const int m0 = (int)((int64_t)rank * prm.num_k / S), nm = (int)((int64_t)(rank + 1) * prm.num_k / S) - m0;
  const int g0 = rank * fr.lr_groups / S, nl = prm.nb * ((rank + 1) * fr.lr_groups / S - g0);
  const int at = min(min(LR_AT, nm), fr.stages), steps = nm + nl;
  auto is_lr = [&](int i) { return i >= at && i < at + nl; };
  auto k_of = [&](int i) { return m0 + (i < at ? i : i - nl); };

  if (threadIdx.x == 0) {
    for (int s = 0; s < fr.stages; ++s) {
      tc::mbar_init(tc::smem_u32(&ss->full[s]), 1 + WORK_ARRIVALS);
      tc::mbar_init(tc::smem_u32(&ss->empty[s]), 1);
    }
    if (W4)
      for (int s = 0; s < fr.raw_slots; ++s) {
        tc::mbar_init(tc::smem_u32(&ss->raw_full[s]), 1);
        tc::mbar_init(tc::smem_u32(&ss->raw_empty[s]), WORK_WARPS / 2);
      }
    tc::mbar_init(tc::smem_u32(&ss->done), 1);
    ss->abort_flag = 0;
    tc::fence_mbar_init();
    tc::prefetch_tmap(&tm.a);
    tc::prefetch_tmap(&tm.b);
    if (GATED) tc::prefetch_tmap(&tm.b2);
  }
  if (warp == 1) {
    tc::tmem_alloc(tc::smem_u32(&ss->tmem_base), (uint32_t)fr.tmem_cols);
    tc::tmem_relinquish();
  }
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  const uint32_t tmem = ss->tmem_base;
  const uint32_t up_col = (uint32_t)(fr.tmem_cols / 2);
  pdl_wait();                             // X, P and C are visible
  pdl_trigger();

  const bool worker = warp >= 2 && warp < 2 + WORK_WARPS;
  const int wt = threadIdx.x - 64;
  bool ok = true;                         // this thread's waits succeeded
  if (warp == 0) {
    // ---------------- TMA producer: X, and 16-bit W ----------------
    if (lane == 0) {
      uint32_t issued = 0, parity = 0, phase = 0;
      int stage = 0;
      for (int i = 0; i < steps; ++i) {
        if (!tc::mbar_wait(tc::smem_u32(&ss->empty[stage]), phase ^ 1u, abort_flag, prm.status)) break;
        const uint32_t full = tc::smem_u32(&ss->full[stage]);
        if (is_lr(i)) {
          tc::mbar_arrive(full);
        } else {
          const uint32_t sw = tc::smem_u32(smem + stage * stage_bytes), sx = sw + NW * W_TILE;
          const int kx = k_of(i) * BKF;
          tc::mbar_arrive_expect_tx(full, (uint32_t)(x_bytes + (W4 ? 0 : NW * W_TILE)));
          if (!W4) {
            tc::mbar_arrive(full);
            tc::tma_load_2d(sw, &tm.b, kx, n0, full);
            if (GATED) tc::tma_load_2d(sw + W_TILE, &tm.b2, kx, n0, full);
          }
          for (int b = 0; b < prm.nb; ++b)
            tc::tma_load_2d(sx + (uint32_t)(b * fr.tpad * BKF * 2), &tm.a, kx, prm.shared ? 0 : b * (int)prm.T, full);
          issued |= 1u << stage;
          parity = (parity & ~(1u << stage)) | (phase << stage);
        }
        if (++stage == fr.stages) { stage = 0; phase ^= 1u; }
      }
      if (*abort_flag)                    // give our copies in flight time to land
        for (int s = 0; s < fr.stages; ++s)
          if (issued & (1u << s))
            tc::mbar_wait_drain(tc::smem_u32(&ss->full[s]), (parity >> s) & 1u, 100000000ull);
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer ----------------
    if (lane == 0) {
      const uint32_t idesc_main = tc::idesc_f16(WR, fr.tok, AB);
      const uint32_t idesc_lr = tc::idesc_f16(WR, fr.tpad, 1);   // low-rank K-blocks are bf16, one block's columns
      int stage = 0;
      uint32_t phase = 0;
      bool any = false;
      for (int i = 0; i < steps; ++i) {
        if (!tc::mbar_wait(tc::smem_u32(&ss->full[stage]), phase, abort_flag, prm.status)) break;
        tc::tc_fence_after();
        const uint32_t sw = tc::smem_u32(smem + stage * stage_bytes);
        uint32_t sx = sw + NW * W_TILE, dcol = 0u, idesc = idesc_main;
        bool gate = true, up = GATED;
        if (is_lr(i)) {
          const LowrankBlock l = lowrank_block(prm.nb, prm.r, g0, i - at);
          sx += (uint32_t)(l.b * fr.tpad * BKF * 2);
          dcol = (uint32_t)(l.b * fr.tpad);
          idesc = idesc_lr;
          if (GATED && fr.lr_mats == 2) { gate = l.mat == 0; up = l.mat == 1; }
        }
#pragma unroll
        for (int k = 0; k < BKF / 16; ++k) {
          const uint32_t acc = (i | k) != 0 ? 1u : 0u;   // the first K-block is W's: it sets every column
          const uint64_t xd = tc::sdesc_k_sw128(sx + k * 32);
          if (gate) tc::mma_f16(tmem + dcol, tc::sdesc_k_sw128(sw + k * 32), xd, idesc, acc);
          if (up) tc::mma_f16(tmem + up_col + dcol, tc::sdesc_k_sw128(sw + W_TILE + k * 32), xd, idesc, acc);
        }
        tc::mma_commit(tc::smem_u32(&ss->empty[stage]));
        any = true;
        if (++stage == fr.stages) { stage = 0; phase ^= 1u; }
      }
      if (any) {
        tc::mma_commit(tc::smem_u32(&ss->done));
        tc::mbar_wait_drain(tc::smem_u32(&ss->done), 0, 100000000ull);
      } else {
        tc::mbar_arrive(tc::smem_u32(&ss->done));
      }
    }
  } else if (W4 && warp == 2 + WORK_WARPS) {
    // ---------------- packed INT4 rows ----------------
    if (lane == 0) {
      int slot = 0;
      uint32_t phase = 0, issued = 0, parity = 0;
      for (int kb = m0; kb < m0 + nm; ++kb) {
        if (!tc::mbar_wait(tc::smem_u32(&ss->raw_empty[slot]), phase ^ 1u, abort_flag, prm.status)) break;
        const uint32_t bar = tc::smem_u32(&ss->raw_full[slot]);
        const uint32_t dst = tc::smem_u32(raw + slot * NW * RAW_TILE);
        tc::mbar_arrive_expect_tx(bar, NW * RAW_TILE);
        tc::tma_load_2d(dst, &tm.b, kb * (BKF / 2), n0, bar);
        if (GATED) tc::tma_load_2d(dst + RAW_TILE, &tm.b2, kb * (BKF / 2), n0, bar);
        issued |= 1u << slot;
        parity = (parity & ~(1u << slot)) | (phase << slot);
        if (++slot == fr.raw_slots) { slot = 0; phase ^= 1u; }
      }
      if (*abort_flag)
        for (int s = 0; s < fr.raw_slots; ++s)
          if (issued & (1u << s))
            tc::mbar_wait_drain(tc::smem_u32(&ss->raw_full[s]), (parity >> s) & 1u, 100000000ull);
    }
  } else {
    // ---------------- work warps: low-rank operands, INT4 dequantisation ----------------
    // INT4: two groups of four warps take alternate K-blocks, so that one group's writes, proxy fence and hand-over
    // overlap the other's work (the packed ring has an even number of slots: a slot's blocks are all one group's, which
    // so sees every phase of its barrier); a thread turns half a row (32 weights) into bf16, for rows row and row + 64.
    const int grp = wt >> 7, row = (wt & 127) >> 1, hf = wt & 1;
    const uint32_t gran = (uint32_t)(((4 * hf) ^ (row & 7)) << 4);   // swizzled offset of granule 4 hf + c: gran ^ 16 c
    const int64_t groups = prm.d_in / 128;
    const __half* src_s[2 * NW];
    float next[2 * NW];
    bool valid[2] = {false, false};
    if (W4) {
      const int kb = m0 + ((m0 ^ grp) & 1);          // this group's K-blocks have parity grp: one scale group each
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        valid[h] = n0 + row + 64 * h < prm.d_out;
#pragma unroll
        for (int w = 0; w < NW; ++w) {
          src_s[h * NW + w] = (w ? prm.Ws2 : prm.Ws) + (int64_t)(n0 + row + 64 * h) * groups;
          next[h * NW + w] = valid[h] && kb < prm.num_k ? __half2float(src_s[h * NW + w][kb / 2]) : 0.f;
        }
      }
    }
    int stage = 0, slot = 0;
    uint32_t phase = 0, rphase = 0;
    for (int i = W4 ? 0 : at; i < (W4 ? steps : at + nl); ++i) {
      if (!W4 && i == at) {                          // the stage and phase of step `at`
        stage = at % fr.stages;
        phase = (uint32_t)(at / fr.stages) & 1u;
      }
      // a work warp whose wait gave up stays in the loop without working, so that every named barrier below is
      // reached by all of them
      if (is_lr(i)) {
        if (wt == 0) ss->lr_ok = ok && tc::mbar_wait(tc::smem_u32(&ss->empty[stage]), phase ^ 1u, abort_flag, prm.status);
        tc::named_bar_sync(WORK_BAR, WORK_THREADS);
        ok = ok && *reinterpret_cast<volatile int*>(&ss->lr_ok) != 0;
        if (ok) {
          const uint32_t sw = tc::smem_u32(smem + stage * stage_bytes);
          fill_lowrank<GATED>(prm, fr, lowrank_block(prm.nb, prm.r, g0, i - at), sw, sw + NW * W_TILE, n0, wt);
          tc::fence_proxy_async_smem();              // generic writes -> the tensor core's reads
        }
        tc::named_bar_sync(WORK_BAR, WORK_THREADS);
        if (wt == 0 && ok) mbar_arrive_n(tc::smem_u32(&ss->full[stage]), WORK_ARRIVALS);
      } else if (W4) {
        const int kb = k_of(i);
        float sc[2 * NW];
        if (ok && ((kb ^ grp) & 1) == 0) {
#pragma unroll
          for (int q = 0; q < 2 * NW; ++q) {
            sc[q] = next[q];
            if (valid[q / NW] && kb + 2 < prm.num_k) next[q] = __half2float(src_s[q][kb / 2 + 1]);
          }
          if (lane == 0)
            ok = tc::mbar_wait(tc::smem_u32(&ss->raw_full[slot]), rphase, abort_flag, prm.status) &&
                 tc::mbar_wait(tc::smem_u32(&ss->empty[stage]), phase ^ 1u, abort_flag, prm.status);
          ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
        }
        if (ok && ((kb ^ grp) & 1) == 0) {
          const uint32_t src = tc::smem_u32(raw + slot * NW * RAW_TILE) + (uint32_t)(row * 32 + hf * 16);
          const uint32_t dst = tc::smem_u32(smem + stage * stage_bytes);
          uint4 q[2 * NW];
#pragma unroll
          for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int w = 0; w < NW; ++w) q[h * NW + w] = tc::ld_shared_v4(src + w * RAW_TILE + h * 64 * 32);
          __syncwarp();
          if (lane == 0) tc::mbar_arrive(tc::smem_u32(&ss->raw_empty[slot]));
#pragma unroll
          for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int w = 0; w < NW; ++w)
            {
              __nv_bfloat162 hi, lo;
              split_scale(sc[h * NW + w], hi, lo);
              const uint4 qq = q[h * NW + w];
              const uint32_t wd[4] = {qq.x, qq.y, qq.z, qq.w};
              const uint32_t rowp = dst + w * W_TILE + (uint32_t)((row + 64 * h) * 128);
#pragma unroll
              for (int c = 0; c < 4; ++c) tc::st_shared_v4(rowp + (gran ^ (16u * c)), dequant8_bf16(wd[c], hi, lo));
            }
          tc::fence_proxy_async_smem();
          __syncwarp();
          if (lane == 0) tc::mbar_arrive(tc::smem_u32(&ss->full[stage]));
        }
        if (++slot == fr.raw_slots) { slot = 0; rphase ^= 1u; }
      }
      if (++stage == fr.stages) { stage = 0; phase ^= 1u; }
    }
    // every MMA of this CTA has completed: its accumulators are whole and its rings free
    if (lane == 0) ok = tc::mbar_wait(tc::smem_u32(&ss->done), 0, abort_flag, prm.status) && ok;
    ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
    tc::tc_fence_after();
  }
  __syncwarp();

  // ---------------- partials, their sums, and the outputs (warps 2-9) ----------------
  const int quad = warp & 3, half = (warp - 2) >> 2;
  const int col = quad * 32 + lane;                  // TMEM lane = output column within the tile
  const int64_t n = n0 + col;
  const uint32_t t_lane = tmem + ((uint32_t)(quad * 32) << 16);
  auto put = [&](int b, int tb, float g, float u) {  // row tb of block b, this thread's output column
    if (tb >= prm.T || n >= prm.d_out) return;
    const float v = GATED ? pairtc::silu_fast(g) * u : apply_act(g, prm.act);
    const int64_t e = ((int64_t)b * prm.T + tb) * prm.d_out + n;
    if (fr.out32) static_cast<float*>(prm.Y)[e] = v;
    else static_cast<T16*>(prm.Y)[e] = from_f32<T16>(v);
  };
  const uint32_t inv = (65535u + (uint32_t)fr.tpad) / (uint32_t)fr.tpad;   // t / tpad = t inv >> 16 for t < 256
  if (S == 1) {
    if (worker && ok) {
      for (int c = 16 * half; c < fr.tok; c += 32) {
        const int b = (int)((uint32_t)c * inv >> 16);  // 16 columns lie in one block
        float g[16], u[16];
        tc::tmem_ld16(t_lane + (uint32_t)c, g);
        if (GATED) tc::tmem_ld16(t_lane + up_col + (uint32_t)c, u);
#pragma unroll
        for (int i = 0; i < 16; ++i) put(b, c - b * fr.tpad + i, g[i], GATED ? u[i] : 0.f);
      }
    }
  } else {
    float* part = reinterpret_cast<float*>(smem);    // [chunk columns][NW][128]: the rings are done with
    const uint32_t part_s = tc::smem_u32(part);
    for (int c0 = 0; c0 < fr.tok; c0 += fr.chunk) {
      const int cn = min(fr.chunk, fr.tok - c0);     // a multiple of 16
      if (worker && ok) {
        for (int c = 16 * half; c < cn; c += 32) {
          float v[16];
#pragma unroll
          for (int w = 0; w < NW; ++w) {
            tc::tmem_ld16(t_lane + (w ? up_col : 0u) + (uint32_t)(c0 + c), v);
#pragma unroll
            for (int i = 0; i < 16; ++i) part[((c + i) * NW + w) * WR + col] = v[i];
          }
        }
      }
      __syncwarp();
      pairtc::tc2::cluster_sync();
      if (worker && ok) {
        const int per = (cn + S - 1) / S;
        const int t0 = min(rank * per, cn), t1 = min(t0 + per, cn);
#pragma unroll 2
        for (int t = t0 + half; t < t1; t += 2) {
          float sum[NW];
#pragma unroll
          for (int w = 0; w < NW; ++w) {
            const uint32_t a = part_s + (uint32_t)(((t * NW + w) * WR + col) * 4);
            float v[MAX_SPLITS];
#pragma unroll
            for (int s = 0; s < MAX_SPLITS; ++s) v[s] = s < S ? ld_dsmem(a, (uint32_t)s) : 0.f;
            sum[w] = v[0];
#pragma unroll
            for (int s = 1; s < MAX_SPLITS; ++s)
              if (s < S) sum[w] += v[s];
          }
          const int b = (int)((uint32_t)(c0 + t) * inv >> 16);
          put(b, c0 + t - b * fr.tpad, sum[0], sum[NW - 1]);
        }
      }
      __syncwarp();
      pairtc::tc2::cluster_sync();                   // the peers have read this chunk's partials
    }
  }
  tc::tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    __syncwarp();
    tc::tc_fence_after();
    tc::tmem_dealloc(tmem, (uint32_t)fr.tmem_cols);
  }
}

}  // namespace pairfr
}  // namespace zoact
