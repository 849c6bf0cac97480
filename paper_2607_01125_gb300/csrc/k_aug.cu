// Operands of the low-rank term on the tensor cores (Section 3: the factor
// (X V_r)(B + mu Z) of the perturbed forward pass as extra K columns of the
// pair-forward MMA).
//
// The low-rank term of an output element is sum_j P[t, j] T[n, j] with P = X U
// (fp32) and T = C + c_b Z_b (fp32).  Both factors are split into 16-bit
// parts, v = hi + lo with hi = bf16(v) and lo = bf16(v - hi), and the three
// largest products are laid out as 3r extra K columns (padded with zeros to
// whole 64-column K-blocks):
//     A_aug row t = [ P_hi | P_hi | P_lo | 0 ]      B_aug row n = [ T_hi | T_lo | T_hi | 0 ]
// so the MMA adds P_hi T_hi + P_hi T_lo + P_lo T_hi, which differs from P T by
// the dropped P_lo T_lo and the rounding of the lo parts: below 2^-15 sum_j
// |P_j| |T_j|.  For a gated pair whose gate and up projections differ, A_aug
// holds both ([gate parts | up parts]) and each B_aug zero-fills the other half.
// B_aug holds one table per evaluation block when the whole term goes to the
// tensor cores (LOWRANK_ALL_ON_TC: T = C + c_b Z_b, Z_b from the same Philox
// stream as every other kernel; when a tile's rows span up to S blocks, A_aug
// has S K slots and row t fills slot block(t) mod S, so each slot meets the
// table of the tile's block congruent to it), and the single table T = C otherwise.  With C
// on the tensor cores the epilogue still adds c_b Z_b p: for it this kernel
// also writes Z of every distinct query, so the pair kernel copies its tile's
// columns instead of regenerating them per tile: transposed, Zt[q][j][n] (fp32),
// or, where several blocks' terms go on the epilogue's matrix instruction, in its
// operand order and three bf16 parts.
// Purely memory-bound and small (rows x r and d_out x r inputs).
#include "internal.h"
#include "philox.cuh"

namespace zoact {
namespace {

struct AugBlocks {
  float coef[ZOACT_MAX_EVAL_BLOCKS];
  uint64_t qry[ZOACT_MAX_EVAL_BLOCKS];
  uint64_t zq[ZOACT_MAX_EVAL_BLOCKS];   // distinct queries whose Z is written
  int nzq;
  // layers run as one (B rows only): row n of the table belongs to layer s with seg_off[s] <= n <
  // seg_off[s + 1]; its T = C_s + c_b Z_b takes C_s and Z from that layer's own rows and Philox stream
  int nseg;
  int seg_off[ZOACT_MAX_GROUP + 1];
  const float* seg_C[ZOACT_MAX_GROUP];
  uint32_t seg_lid[ZOACT_MAX_GROUP];
};

// v = hi + lo (+ what bf16 cannot hold): hi = bf16(v), lo = bf16(v - hi); v - hi is exact in fp32.
__device__ __forceinline__ void split16(float v, __nv_bfloat16& hi, __nv_bfloat16& lo) {
  hi = __float2bfloat16_rn(v);
  lo = __float2bfloat16_rn(v - __bfloat162float(hi));
}

__device__ __forceinline__ uint32_t pack_bf16x2(__nv_bfloat16 a, __nv_bfloat16 b) {
  return (uint32_t)__bfloat16_as_ushort(a) | ((uint32_t)__bfloat16_as_ushort(b) << 16);
}

// The split parts of four consecutive ranks j0..j0+3 of one source row: hi
// (want_lo false) or lo, packed as bf16 pairs.
__device__ __forceinline__ uint2 split_quad(float4 v, bool want_lo) {
  __nv_bfloat16 h[4], l[4];
  split16(v.x, h[0], l[0]);
  split16(v.y, h[1], l[1]);
  split16(v.z, h[2], l[2]);
  split16(v.w, h[3], l[3]);
  const __nv_bfloat16* o = want_lo ? l : h;
  return make_uint2(pack_bf16x2(o[0], o[1]), pack_bf16x2(o[2], o[3]));
}

// Transposed Z tables: Zt[q][j][n] for each distinct query (gate, then up); one thread per (matrix, query, group of 4
// ranks, column n), columns fastest so that the stores coalesce.
__device__ __forceinline__ void write_z_tables(const AugBlocks& blk, int d_out, int r, uint64_t seed, uint32_t lid,
                                               uint32_t lid2, float* __restrict__ Zt, float* __restrict__ Zt2) {
  const int groups = (r + 3) / 4;
  const int n_mat = Zt2 ? 2 : 1;
  const int64_t items = (int64_t)n_mat * blk.nzq * groups * d_out;
  for (int64_t it = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; it < items;
       it += (int64_t)gridDim.x * blockDim.x) {
    const int n = (int)(it % d_out);
    int64_t rest = it / d_out;
    const int jg = (int)(rest % groups);
    rest /= groups;
    const int qi = (int)(rest % blk.nzq);
    const int mat = (int)(rest / blk.nzq);
    float* dst = (mat ? Zt2 : Zt) + (int64_t)qi * r * d_out;
    const uint32_t layer = mat ? lid2 : lid;
    if ((r & 3) == 0) {
      // the four ranks are one Philox group
      const float4 z = z_normals4(seed, layer, blk.zq[qi], (uint64_t)(((int64_t)n * r + 4 * jg) >> 2));
      dst[(int64_t)(4 * jg) * d_out + n] = z.x;
      dst[(int64_t)(4 * jg + 1) * d_out + n] = z.y;
      dst[(int64_t)(4 * jg + 2) * d_out + n] = z.z;
      dst[(int64_t)(4 * jg + 3) * d_out + n] = z.w;
    } else {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int j = 4 * jg + i;
        if (j < r) {
          const int64_t e = (int64_t)n * r + j;
          dst[(int64_t)j * d_out + n] =
              z_select(z_normals4(seed, layer, blk.zq[qi], (uint64_t)(e >> 2)), (int)(e & 3));
        }
      }
    }
  }
}

// The Z tables in operand order (see z_chunk_words): one thread per (matrix, query, 16 columns, lanes l and l + 1 with l
// even): its two columns and, of each group of eight, four ranks -- one Philox group where the rank is a multiple of
// four -- of which it writes 32 H bytes a part.
template <int H>
__device__ __forceinline__ void write_z_operands(const AugBlocks& blk, int d_out, int r, uint64_t seed, uint32_t lid,
                                                 uint32_t lid2, uint32_t* __restrict__ Zt, uint32_t* __restrict__ Zt2) {
  constexpr int CHUNK = 3 * 32 * 2 * H, G = H > 2 ? 4 : 2 * H;
  const int chunks = (d_out + 63) / 64 * 4;
  const int64_t items = (int64_t)(Zt2 ? 2 : 1) * blk.nzq * chunks * 16;
  for (int64_t it = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; it < items;
       it += (int64_t)gridDim.x * blockDim.x) {
    const int l = 2 * (int)(it & 15);
    int64_t rest = it >> 4;
    const int ch = (int)(rest % chunks);
    rest /= chunks;
    const int qi = (int)(rest % blk.nzq), mat = (int)(rest / blk.nzq);
    const uint32_t layer = mat ? lid2 : lid;
    float z[2][H][4];                                 // [8 columns][group][rank]
#pragma unroll
    for (int nt = 0; nt < 2; ++nt) {
      const int n = ch * 16 + nt * 8 + l / 4;
#pragma unroll
      for (int h = 0; h < H; ++h) {
        const int j0 = 8 * h + 4 * ((l >> 1) & 1);
        const int64_t e = (int64_t)n * r + j0;
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (n < d_out && j0 < r && (r & 3) == 0) v = z_normals4(seed, layer, blk.zq[qi], (uint64_t)(e >> 2));
        z[nt][h][0] = v.x; z[nt][h][1] = v.y; z[nt][h][2] = v.z; z[nt][h][3] = v.w;
        if (n < d_out && j0 < r && (r & 3) != 0) {
          // four ranks in at most two Philox groups
          const int at = (int)(e & 3), ranks = min(4, r - j0);
          const float4 a = z_normals4(seed, layer, blk.zq[qi], (uint64_t)(e >> 2));
          float4 b = a;
          if (at + ranks > 4) b = z_normals4(seed, layer, blk.zq[qi], (uint64_t)(e >> 2) + 1);
#pragma unroll
          for (int i = 0; i < 4; ++i)
            if (i < ranks) z[nt][h][i] = at + i < 4 ? z_select(a, at + i) : z_select(b, at + i - 4);
        }
      }
    }
    uint32_t* dst = (mat ? Zt2 : Zt) + ((int64_t)qi * chunks + ch) * CHUNK;
#pragma unroll
    for (int part = 0; part < 3; ++part) {
      uint32_t w[2][2 * H];                           // [lane][8 columns, group]
#pragma unroll
      for (int nt = 0; nt < 2; ++nt)
#pragma unroll
        for (int h = 0; h < H; ++h) {
          w[0][nt * H + h] = next_part_bf16x2(z[nt][h][0], z[nt][h][1]);
          w[1][nt * H + h] = next_part_bf16x2(z[nt][h][2], z[nt][h][3]);
        }
#pragma unroll
      for (int g = 0; g < 2 * H / G; ++g) {
        uint32_t* d = dst + part * (CHUNK / 3) + g * 32 * G + l * G;
#pragma unroll
        for (int i = 0; i < 2 * G; i += 4)
          *reinterpret_cast<uint4*>(d + i) = make_uint4(w[i / G][g * G + i % G], w[(i + 1) / G][g * G + (i + 1) % G],
                                                        w[(i + 2) / G][g * G + (i + 2) % G],
                                                        w[(i + 3) / G][g * G + (i + 3) % G]);
      }
    }
  }
}

// Z's tables, transposed or (OPS; a kernel of its own, the others need fewer registers) in operand order.
template <bool OPS>
__device__ __forceinline__ void write_z(int z_rt, const AugBlocks& blk, int d_out, int r, uint64_t seed, uint32_t lid,
                                        uint32_t lid2, float* __restrict__ Zt, float* __restrict__ Zt2) {
  if (!Zt || blk.nzq == 0) return;
  if constexpr (OPS) {
    uint32_t* z1 = reinterpret_cast<uint32_t*>(Zt);
    uint32_t* z2 = reinterpret_cast<uint32_t*>(Zt2);
    if (z_rt <= 8) write_z_operands<1>(blk, d_out, r, seed, lid, lid2, z1, z2);
    else if (z_rt == 16) write_z_operands<2>(blk, d_out, r, seed, lid, lid2, z1, z2);
    else write_z_operands<4>(blk, d_out, r, seed, lid, lid2, z1, z2);
  } else {
    write_z_tables(blk, d_out, r, seed, lid, lid2, Zt, Zt2);
  }
}

// Any rank (the quad kernel below serves ranks that are multiples of 4 with 16-byte aligned sources): one thread per
// 16-byte chunk (8 K columns) of an output row: rows [0, nA) of A_aug, then the nB rows of B_aug (block b, column n),
// then those of B_aug2.  Each column k of a row maps to (slot, half, part, rank j); the chunk is built from the source
// values it needs (P or P2 for A rows, T = C + c_b Z_b for B rows; source rows are re-read from L1/L2 by the row's
// chunks).
template <bool OPS>
__global__ void __launch_bounds__(256)
aug_prep_kernel(const float* __restrict__ P, const float* __restrict__ P2, const float* __restrict__ C,
                const float* __restrict__ C2, __nv_bfloat16* __restrict__ A, __nv_bfloat16* __restrict__ B,
                __nv_bfloat16* __restrict__ B2, int64_t rows, int d_out, int r, int ka, int distinct, int full,
                int nb, const __grid_constant__ AugBlocks blk, uint64_t seed, uint32_t lid, uint32_t lid2,
                float* __restrict__ Zt, float* __restrict__ Zt2, int z_rt, int slots, int64_t T) {
  pdl_wait();                                         // P and C written by the previous kernels
  pdl_trigger();
  const int ka_row = distinct ? 2 * ka : ka;          // columns of one slot (= B_aug row width)
  const int cA = slots * ka_row / 8, cB = ka_row / 8; // 16-byte chunks per A / B row
  const int nbB = full ? nb : 1;
  const int64_t nB = (int64_t)nbB * d_out;
  const int64_t itA = rows * cA;
  const int64_t items = itA + (B2 ? 2 : 1) * nB * cB;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t it = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; it < items; it += stride) {
    const bool is_a = it < itA;
    bool up = false;
    int64_t orow;
    int c;
    if (is_a) {
      orow = it / cA;
      c = (int)(it - orow * cA);
    } else {
      const int64_t ib = it - itA;
      const int64_t rb = ib / cB;
      c = (int)(ib - rb * cB);
      up = rb >= nB;
      orow = up ? rb - nB : rb;                      // b * d_out + n
    }
    int my_slot = 0, n = 0;
    float cb = 0.f;
    uint64_t q = 0;
    uint32_t layer = up ? lid2 : lid;
    const float* Cs = up ? C2 : C;      // the coefficients row n indexes (a grouped layer's own)
    if (is_a) {
      if (slots > 1) my_slot = (int)((orow / T) % slots);
    } else {
      const int b = (int)(orow / d_out);
      n = (int)(orow - (int64_t)b * d_out);
      if (full) { cb = blk.coef[b]; q = blk.qry[b]; }
      if (blk.nseg > 1) {
        int sg = 0;
        while (sg + 1 < blk.nseg && n >= blk.seg_off[sg + 1]) ++sg;
        n -= blk.seg_off[sg];
        Cs = blk.seg_C[sg];
        layer = blk.seg_lid[sg];
      }
    }
    uint32_t w[4];
#pragma unroll
    for (int h4 = 0; h4 < 2; ++h4) {
      {
        __nv_bfloat16 e4[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int k = 8 * c + 4 * h4 + i;
          const int slot = k / ka_row;
          const int kk = k - slot * ka_row;
          const int half = kk >= ka ? 1 : 0, kq = kk - half * ka;
          const int part = kq / r, j = kq - part * r;
          const bool live = part < 3 && slot == my_slot && (is_a || !distinct || half == (up ? 1 : 0));
          __nv_bfloat16 hi = __float2bfloat16_rn(0.f), lo = hi;
          if (live) {
            float v;
            if (is_a) {
              v = (distinct && half ? P2 : P)[orow * r + j];
            } else {
              const int64_t e = (int64_t)n * r + j;
              v = Cs[e];
              if (cb != 0.f) v = fmaf(cb, z_select(z_normals4(seed, layer, q, (uint64_t)(e >> 2)), (int)(e & 3)), v);
            }
            split16(v, hi, lo);
          }
          e4[i] = live ? ((is_a ? part == 2 : part == 1) ? lo : hi) : __float2bfloat16_rn(0.f);
        }
        w[2 * h4] = pack_bf16x2(e4[0], e4[1]);
        w[2 * h4 + 1] = pack_bf16x2(e4[2], e4[3]);
      }
    }
    __nv_bfloat16* dst = is_a ? A : (up ? B2 : B);
    const int64_t row_w = 8 * (int64_t)(is_a ? cA : cB);
    *reinterpret_cast<uint4*>(dst + orow * row_w + 8 * c) = make_uint4(w[0], w[1], w[2], w[3]);
  }
  write_z<OPS>(z_rt, blk, d_out, r, seed, lid, lid2, Zt, Zt2);
}

// The same tables for ranks that are multiples of 4 with aligned sources: one thread per four ranks of a row, which
// forms their values once -- a Philox call serves the three parts and, where two evaluation blocks share a query (the
// two signs), both of them -- and writes 8 bytes to each part and its share of the row's zeros.  A chunk per thread drew
// every Z three times: 20480 x 32, two signs, 666 rows 20.3 us there, 6.0 here; gated 14336 x 16, two signs, 8192
// rows 15.6 and 5.6.  I: 32-bit item indexes where they fit.
// ZEROS: the zeros of A's rows or of both as items of their own (zeros; see spread_zeros).  A kernel of its own: its
// branches cost the others 1.5 us at 20480 x 32.
constexpr int SPREAD_A = 1, SPREAD_B = 2;
template <typename I, bool OPS, bool ZEROS>
__global__ void __launch_bounds__(256, ZEROS ? 4 : 0)
aug_quad_kernel(const float* __restrict__ P, const float* __restrict__ P2, const float* __restrict__ C,
                const float* __restrict__ C2, __nv_bfloat16* __restrict__ A, __nv_bfloat16* __restrict__ B,
                __nv_bfloat16* __restrict__ B2, int64_t rows, int d_out, int r, int ka, int distinct, int full,
                int nb, const __grid_constant__ AugBlocks blk, uint64_t seed, uint32_t lid, uint32_t lid2,
                float* __restrict__ Zt, float* __restrict__ Zt2, int z_rt, int slots, int64_t T, int zeros) {
  const int spread = ZEROS ? zeros : 0;
  pdl_wait();                                         // P and C written by the previous kernels
  pdl_trigger();
  const int rq = r / 4, kq = ka / 4, halves = distinct ? 2 : 1;
  const int row_q = halves * kq;                      // quads of one slot (= B_aug row)
  const int nbB = full ? nb : 1, pairs = (nbB + 1) / 2;
  const I itA = (I)rows * (I)(halves * rq);
  const I itB = (I)pairs * (I)d_out * (I)rq;
  const I items = itA + itB * (B2 ? 2 : 1);
  // the zeros of A's and of B's rows as items of their own, two quads (16 bytes) each over whole rows
  const I pa = (I)(slots * row_q / 2), pb = (I)(row_q / 2);
  const I zA = spread & SPREAD_A ? (I)rows * pa : 0, zB = spread & SPREAD_B ? (I)nbB * (I)d_out * pb : 0;
  const I total = items + zA + zB * (B2 ? 2 : 1);
  const uint2 zero = make_uint2(0u, 0u);
  // one half of one slot: this quad's three parts (live), and, unless they are spread, its share of the zeros
  auto put = [&](uint2* half_q, int g, float4 v, bool is_a, bool live) {
    if (live) {
      const uint2 hi = split_quad(v, false), lo = split_quad(v, true);
      half_q[g] = hi;
      half_q[rq + g] = is_a ? hi : lo;
      half_q[2 * rq + g] = is_a ? lo : hi;
    }
    if (spread & (is_a ? SPREAD_A : SPREAD_B)) return;
    for (int z = (live ? 3 * rq : 0) + g; z < kq; z += rq) half_q[z] = zero;
  };
  const I stride = (I)gridDim.x * blockDim.x;
  for (I it = (I)blockIdx.x * blockDim.x + threadIdx.x; it < total; it += stride) {
    if (it < itA) {
      const I rh = it / (I)rq;
      const int g = (int)(it - rh * (I)rq);
      const int h = distinct ? (int)(rh & 1) : 0;
      const int64_t row = distinct ? (int64_t)(rh >> 1) : (int64_t)rh;
      const float4 v = *reinterpret_cast<const float4*>((h ? P2 : P) + row * r + 4 * g);
      const int mine = slots > 1 ? (int)((row / T) % slots) : 0;
      uint2* q = reinterpret_cast<uint2*>(A) + row * ((int64_t)slots * row_q) + h * kq;
      if (spread & SPREAD_A) put(q + mine * row_q, g, v, true, true);
      else
        for (int s = 0; s < slots; ++s) put(q + s * row_q, g, v, true, s == mine);
    } else if (it < items) {
      I ib = it - itA;
      const bool up = ib >= itB;
      if (up) ib -= itB;
      const I bn = ib / (I)rq;
      const int g = (int)(ib - bn * (I)rq);
      const int bp = (int)(bn / (I)d_out);
      const int n_all = (int)(bn - (I)bp * (I)d_out);
      int n = n_all;
      uint32_t layer = up ? lid2 : lid;
      const float* Cs = up ? C2 : C;                  // the coefficients row n indexes (a grouped layer's own)
      if (blk.nseg > 1) {
        int sg = 0;
        while (sg + 1 < blk.nseg && n >= blk.seg_off[sg + 1]) ++sg;
        n -= blk.seg_off[sg];
        Cs = blk.seg_C[sg];
        layer = blk.seg_lid[sg];
      }
      const int64_t e = (int64_t)n * r + 4 * g;
      const float4 c = *reinterpret_cast<const float4*>(Cs + e);
      float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
      uint64_t drawn = 0;
      bool have = false;
      for (int b = 2 * bp; b < min(2 * bp + 2, nbB); ++b) {
        float4 v = c;
        const float cb = full ? blk.coef[b] : 0.f;
        if (cb != 0.f) {
          if (!have || blk.qry[b] != drawn) z = z_normals4(seed, layer, blk.qry[b], (uint64_t)(e >> 2));
          have = true;
          drawn = blk.qry[b];
          v.x = fmaf(cb, z.x, v.x); v.y = fmaf(cb, z.y, v.y);
          v.z = fmaf(cb, z.z, v.z); v.w = fmaf(cb, z.w, v.w);
        }
        uint2* q = reinterpret_cast<uint2*>(up ? B2 : B) + ((int64_t)b * d_out + n_all) * row_q;
        // distinct: gate rows fill the first half, up rows the second
        for (int h = 0; h < halves; ++h) put(q + h * kq, g, v, false, !distinct || h == (up ? 1 : 0));
      }
    } else {
      I ib = it - items;
      const bool is_a = ib < zA;
      if (!is_a) ib -= zA;
      const bool up = !is_a && ib >= zB;
      if (up) ib -= zB;
      const I row = ib / (is_a ? pa : pb);
      const int q0 = 2 * (int)(ib - row * (is_a ? pa : pb)), s = q0 / row_q, h = (q0 - s * row_q) / kq;
      const int z0 = q0 - s * row_q - h * kq;         // quad of the half (kq is even)
      const bool live = is_a ? slots == 1 || s == (int)(((int64_t)row / T) % slots) : !distinct || h == (up ? 1 : 0);
      uint2* q = reinterpret_cast<uint2*>(is_a ? A : up ? B2 : B) + 2 * (int64_t)ib;
      if (!live || z0 >= 3 * rq) *reinterpret_cast<uint4*>(q) = make_uint4(0u, 0u, 0u, 0u);
      else if (z0 + 1 >= 3 * rq) q[1] = zero;
    }
  }
  write_z<OPS>(z_rt, blk, d_out, r, seed, lid, lid2, Zt, Zt2);
}

bool aligned16_or_null(const void* p) { return ((uintptr_t)p & 15u) == 0; }

// Whose zeros are items of their own.  A quad's thread writes its share of them beside its three parts while these are
// few: zero to five stores for ranks from 12 in one or two slots.  Ranks 4 and 8 have one or two threads a row, and rows
// of several slots many zeros a thread.  Calls on 256 columns, their zeros by the quads' threads, spread, and with a thread
// per chunk for everything: rank 4, two signs of 2048 rows on 14336 outputs 98.1, 69.4, 69.7 us; rank 8 70.2, 67.0, 69.8;
// rank 12, 333 rows each on 256 outputs 9.4, 9.2, 9.3; 17 blocks of 14 rows (11 slots), rank 24 25.2, 23.6, 24.4.  The
// other way: rank 16, 333 rows each on 4096 outputs (two slots) 11.1 and 11.5; B's rows, which the two threads' stores
// fill whole, gate and up with a projection each, 17 blocks on 14336 outputs, rank 16 68.6 and 96.4.
// Rank 8's B rows only while the quads' threads leave SMs idle (eight queries, 512 tokens each through an MLP block: 530
// us a step with B's zeros spread too, 525 so).
int spread_zeros(int slots, int row_q, int rq, int distinct, bool few_b) {
  if (rq <= 2) return SPREAD_A | (rq == 1 || few_b ? SPREAD_B : 0);
  return slots * row_q / ((distinct ? 2 : 1) * rq) - 3 > 6 ? SPREAD_A : 0;
}

}  // namespace

int launch_aug_prep(Ctx* ctx, const PairArgs& a, int mode, int ka, int distinct, int slots, void* A_aug,
                    void* B_aug, void* B_aug2, float* Zt, float* Zt2, const uint64_t* zq, int nzq, int z_rt) {
  AugBlocks blk{};
  for (int b = 0; b < a.nb; ++b) { blk.coef[b] = a.coef[b]; blk.qry[b] = a.qry[b]; }
  blk.nseg = a.nseg > 1 ? a.nseg : 0;
  for (int g = 0; g < blk.nseg; ++g) {
    blk.seg_off[g] = a.seg_off[g];
    blk.seg_C[g] = a.seg_C[g];
    blk.seg_lid[g] = a.seg_lid[g];
  }
  blk.seg_off[blk.nseg] = a.d_out;
  // the operand rows of a grouped launch come from the layers' own coefficients (Z tables: one layer only)
  if (blk.nseg > 1 && (Zt || B_aug2)) return ZOACT_ERR_UNSUPPORTED;
  for (int i = 0; i < nzq; ++i) blk.zq[i] = zq[i];
  blk.nzq = Zt ? nzq : 0;
  const int full = mode == LOWRANK_ALL_ON_TC;
  const int ka_row = distinct ? 2 * ka : ka;
  const int64_t nbB = full ? a.nb : 1;
  const int64_t items = a.rows * (slots * ka_row / 8) + (B_aug2 ? 2 : 1) * nbB * a.d_out * (ka_row / 8);
  const int64_t z_each = z_rt ? (int64_t)(a.d_out + 63) / 64 * 64 : (int64_t)((a.r + 3) / 4) * a.d_out;
  const int64_t z_items = Zt ? (Zt2 ? 2 : 1) * blk.nzq * z_each : 0;
  const int64_t work = items > z_items ? items : z_items;
  int64_t grid = (work + 255) / 256;
  const int64_t cap = (int64_t)ctx->sm_count * 32;
  if (grid > cap) grid = cap;
  if (grid < 1) grid = 1;
  // float4 source loads need 16-byte aligned rows: r a multiple of 4 and aligned bases (null: unused)
  bool quad = a.r % 4 == 0 && aligned16_or_null(a.P) && aligned16_or_null(distinct ? a.P2 : nullptr) &&
              aligned16_or_null(a.C) && aligned16_or_null(a.C2);
  for (int g = 0; g < blk.nseg; ++g) quad = quad && aligned16_or_null(a.seg_C[g]);
  if (quad) {
    const int rq = a.r / 4, row_q = ka_row / 4;
    const int64_t itA = a.rows * ((distinct ? 2 : 1) * rq), itB = (B_aug2 ? 2 : 1) * ((nbB + 1) / 2) * a.d_out * (int64_t)rq;
    const int spread = spread_zeros(slots, row_q, rq, distinct, itB < 512 * (int64_t)ctx->sm_count);
    const int64_t q_items = itA + itB + (spread & SPREAD_A ? a.rows * (slots * row_q / 2) : 0) +
                            (spread & SPREAD_B ? (B_aug2 ? 2 : 1) * nbB * a.d_out * (int64_t)(row_q / 2) : 0);
    const int64_t q_work = q_items > z_items ? q_items : z_items;
    grid = (q_work + 255) / 256;
    if (grid > cap) grid = cap;
    if (grid < 1) grid = 1;
    // (a grid-stride step past the last item must fit too)
    const bool narrow = q_items + grid * 256 < ((int64_t)1 << 31);
    auto pick = [&](auto index) {
      using I = decltype(index);
      return spread ? (z_rt ? aug_quad_kernel<I, true, true> : aug_quad_kernel<I, false, true>)
                    : (z_rt ? aug_quad_kernel<I, true, false> : aug_quad_kernel<I, false, false>);
    };
    auto quad_kern = narrow ? pick(uint32_t{}) : pick(int64_t{});
    ZOACT_CUDA_TRY(launch_pdl(ctx, quad_kern, dim3((unsigned)grid), dim3(256), 0, a.P, distinct ? a.P2 : nullptr, a.C,
                              a.C2, static_cast<__nv_bfloat16*>(A_aug), static_cast<__nv_bfloat16*>(B_aug),
                              static_cast<__nv_bfloat16*>(B_aug2), a.rows, a.d_out, a.r, ka, distinct, full, a.nb, blk,
                              a.seed, a.layer_id, a.layer_id2, Zt, Zt2, z_rt, slots, a.T, spread));
  } else {
    ZOACT_CUDA_TRY(launch_pdl(ctx, z_rt ? aug_prep_kernel<true> : aug_prep_kernel<false>, dim3((unsigned)grid), dim3(256),
                              0, a.P, distinct ? a.P2 : nullptr, a.C, a.C2, static_cast<__nv_bfloat16*>(A_aug),
                              static_cast<__nv_bfloat16*>(B_aug), static_cast<__nv_bfloat16*>(B_aug2), a.rows, a.d_out,
                              a.r, ka, distinct, full, a.nb, blk, a.seed, a.layer_id, a.layer_id2, Zt, Zt2, z_rt, slots,
                              a.T));
  }
  ++ctx->n_launch;
  ZOACT_CHECK_LAUNCH();
  return ZOACT_OK;
}

}  // namespace zoact
