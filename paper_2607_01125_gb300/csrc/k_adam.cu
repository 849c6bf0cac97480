// ZO-Adam and ZO-SGD over the flat coefficient arenas (Section 3: Adam on the
// estimated coefficient gradient; Table 1 "Full SGD"; Appendix B: weight decay 0).
//
//   g = (1/q) sum_j a_j Z(seed, layer_id, query_j)   (Z regenerated, never stored;
//                                                      q = 1, a = a_pair: the two-sided g = a Z)
//   m = b1 m + (1 - b1) g ;  v = b2 v + (1 - b2) g^2
//   C -= (lr / (1 - b1^t)) * m / (sqrt(v) / sqrt(1 - b2^t) + adam_eps)
//
// Purely HBM-bound: each coefficient costs 24 bytes (read and write C, m, v).
// A thread owns groups of 4 consecutive elements: one Philox call yields the 4
// normals, and C, m, v move as 16-byte vectors, those of two groups loaded before
// either's normals are drawn (the draw, ~200 instructions, covers their latency).
// The layer table (offsets, layer ids) travels in the kernel parameters.  A block
// walks a contiguous range of groups, so that it searches the table once and then
// only steps to the next layer (a grid stride over the arena searched eight levels
// for every group).  22.0 M coefficients, 224 layers: 105 us (5.0 TB/s) with the
// search per group and loads after the draw, 86.6 (6.1 TB/s) here.  a is read from device memory (the loss kernel's output), so a whole
// ZO step runs without a host synchronisation.  With q queries every group
// draws q Philox groups (one per query) and sums a_j z_j in query order.
#include "internal.h"
#include "philox.cuh"

#include <cmath>

namespace zoact {
namespace {

constexpr int ADAM_TABLE = 256;  // layers per launch

struct QueryList {
  uint64_t q[ZOACT_MAX_EVAL_BLOCKS];
};

struct AdamTable {
  int64_t begin[ADAM_TABLE];
  int64_t end[ADAM_TABLE];
  uint32_t layer_id[ADAM_TABLE];
  int n;
};

__device__ __forceinline__ int find_block(const AdamTable& t, int64_t e) {
  int lo = 0, hi = t.n - 1;
  while (lo < hi) {                  // last block with begin <= e
    const int mid = (lo + hi + 1) >> 1;
    if (t.begin[mid] <= e) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// The gradient estimate of one group: (1/q) sum_j a_j z_j.
__device__ __forceinline__ float4 zo_gradient4(const double* __restrict__ a_dev, float a0, int nq, float inv_q,
                                               const QueryList& qs, uint64_t seed, uint32_t layer, uint64_t group) {
  float4 g = z_normals4(seed, layer, qs.q[0], group);
  g.x *= a0; g.y *= a0; g.z *= a0; g.w *= a0;
  if (nq > 1) {
    for (int j = 1; j < nq; ++j) {
      const float aj = (float)a_dev[j];
      const float4 z = z_normals4(seed, layer, qs.q[j], group);
      g.x = fmaf(aj, z.x, g.x); g.y = fmaf(aj, z.y, g.y);
      g.z = fmaf(aj, z.z, g.z); g.w = fmaf(aj, z.w, g.w);
    }
    g.x *= inv_q; g.y *= inv_q; g.z *= inv_q; g.w *= inv_q;
  }
  return g;
}

// ADAM_UNROLL: groups of a thread whose loads are in flight together: two where a block has two rounds, else one (65536
// coefficients after their loss: 18.1 us with the search per group, 16.5 so; 40 registers, as that had, spill: 18.2).
template <bool SGD, int ADAM_UNROLL>
__global__ void __launch_bounds__(256)
zo_update_kernel(float* __restrict__ C, float* __restrict__ m, float* __restrict__ v, const __grid_constant__ AdamTable tab,
                 int64_t g_begin, int64_t g_end, int64_t per_block, const double* __restrict__ a_dev, int nq,
                 const __grid_constant__ QueryList qs, float lr, float b1, float b2, float adam_eps, float step_size,
                 float inv_sqrt_bc2, uint64_t seed, int* __restrict__ status) {
  pdl_wait();                              // a (the loss kernel's output) is visible
  pdl_trigger();
  bool finite = true;
  for (int j = 0; j < nq; ++j) finite = finite && isfinite(a_dev[j]);
  if (!finite) {
    if (blockIdx.x == 0 && threadIdx.x == 0) record_error(status, ZOACT_ERR_NONFINITE);
    return;
  }
  const float a0 = (float)a_dev[0];
  const float inv_q = 1.0f / (float)nq;
  const int64_t first = g_begin + blockIdx.x * per_block;
  const int64_t last = first + per_block < g_end ? first + per_block : g_end;
  if (first >= last) return;
  int b = find_block(tab, 4 * first);
  for (int64_t g0 = first + threadIdx.x; g0 < last; g0 += ADAM_UNROLL * 256) {
    int lay[ADAM_UNROLL], left[ADAM_UNROLL];             // layer, and elements of the group inside it (0: none)
    float4 c4[ADAM_UNROLL], m4[ADAM_UNROLL], v4[ADAM_UNROLL];
#pragma unroll
    for (int u = 0; u < ADAM_UNROLL; ++u) {
      const int64_t e = 4 * (g0 + u * 256);
      c4[u] = m4[u] = v4[u] = make_float4(0.f, 0.f, 0.f, 0.f);
      left[u] = 0;
      if (g0 + u * 256 < last) {
        if (b + 1 < tab.n && tab.begin[b + 1] <= e) {    // the next layer, or (many short ones) a search
          ++b;
          if (b + 1 < tab.n && tab.begin[b + 1] <= e) b = find_block(tab, e);
        }
        const int64_t rest = tab.end[b] - e;             // <= 0: a gap between blocks
        left[u] = rest >= 4 ? 4 : rest > 0 ? (int)rest : 0;
      }
      lay[u] = b;
      if (left[u] == 4) {
        c4[u] = *reinterpret_cast<const float4*>(C + e);
        if (!SGD) {
          m4[u] = *reinterpret_cast<const float4*>(m + e);
          v4[u] = *reinterpret_cast<const float4*>(v + e);
        }
      } else if (left[u] > 0) {
        float* cp = &c4[u].x;
        float* mp = &m4[u].x;
        float* vp = &v4[u].x;
#pragma unroll
        for (int i = 0; i < 3; ++i)
          if (i < left[u]) {
            cp[i] = C[e + i];
            if (!SGD) { mp[i] = m[e + i]; vp[i] = v[e + i]; }
          }
      }
    }
#pragma unroll
    for (int u = 0; u < ADAM_UNROLL; ++u) {
      if (left[u] == 0) continue;
      const int64_t e = 4 * (g0 + u * 256);
      const int64_t local = e - tab.begin[lay[u]];       // element index inside the layer's [d_out, r]
      const float4 g4 = zo_gradient4(a_dev, a0, nq, inv_q, qs, seed, tab.layer_id[lay[u]], (uint64_t)(local >> 2));
      const float gz[4] = {g4.x, g4.y, g4.z, g4.w};
      float cv[4] = {c4[u].x, c4[u].y, c4[u].z, c4[u].w};
      float mv[4] = {m4[u].x, m4[u].y, m4[u].z, m4[u].w};
      float vv[4] = {v4[u].x, v4[u].y, v4[u].z, v4[u].w};
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        if (SGD) {
          cv[i] -= lr * gz[i];
        } else {
          mv[i] = b1 * mv[i] + (1.0f - b1) * gz[i];
          vv[i] = b2 * vv[i] + (1.0f - b2) * gz[i] * gz[i];
          const float denom = sqrtf(vv[i]) * inv_sqrt_bc2 + adam_eps;
          cv[i] = cv[i] - step_size * (mv[i] / denom);
        }
      }
      if (left[u] == 4) {
        *reinterpret_cast<float4*>(C + e) = make_float4(cv[0], cv[1], cv[2], cv[3]);
        if (!SGD) {
          *reinterpret_cast<float4*>(m + e) = make_float4(mv[0], mv[1], mv[2], mv[3]);
          *reinterpret_cast<float4*>(v + e) = make_float4(vv[0], vv[1], vv[2], vv[3]);
        }
      } else {
#pragma unroll
        for (int i = 0; i < 3; ++i)
          if (i < left[u]) {
            C[e + i] = cv[i];
            if (!SGD) { m[e + i] = mv[i]; v[e + i] = vv[i]; }
          }
      }
    }
  }
}

}  // namespace

int launch_adam(Ctx* ctx, float* C, float* m, float* v, const zoact_coeff_block* blocks, int n_blocks,
                const double* a, int q, const uint64_t* queries, float lr, float b1, float b2, float adam_eps,
                int64_t step, uint64_t seed, int sgd) {
  if (q < 1 || q > ZOACT_MAX_EVAL_BLOCKS) return ZOACT_ERR_INVALID_ARG;
  QueryList qs{};
  for (int j = 0; j < q; ++j) qs.q[j] = queries[j];
  const double bc1 = 1.0 - std::pow((double)b1, (double)step);
  const double bc2 = 1.0 - std::pow((double)b2, (double)step);
  const float step_size = sgd ? 0.f : (float)((double)lr / bc1);
  const float inv_sqrt_bc2 = sgd ? 0.f : (float)(1.0 / std::sqrt(bc2));
  for (int base = 0; base < n_blocks; base += ADAM_TABLE) {
    AdamTable tab;
    tab.n = n_blocks - base < ADAM_TABLE ? n_blocks - base : ADAM_TABLE;
    int64_t lo = INT64_MAX, hi = 0;
    for (int i = 0; i < tab.n; ++i) {
      const zoact_coeff_block& bl = blocks[base + i];
      tab.begin[i] = bl.offset;
      tab.end[i] = bl.offset + (int64_t)bl.d_out * bl.r;
      tab.layer_id[i] = bl.layer_id;
      if (tab.begin[i] < lo) lo = tab.begin[i];
      if (tab.end[i] > hi) hi = tab.end[i];
    }
    if (hi <= lo) continue;
    const int64_t g_begin = lo / 4, g_end = (hi + 3) / 4;
    // a block's range: whole rounds of its threads (one group each), eight blocks per SM.  With several queries the draws
    // are the time, and few rounds go to rather more blocks, which the SMs take as they come, than to ranges that leave
    // some SM a round ahead (1310720 elements, 8 queries: 28.2 us in 640 blocks of two rounds, 26.1 in 1280 of one; with
    // one query, where a thread's two groups in flight count, 7.4 and 7.7).
    const int64_t groups = g_end - g_begin, cap = (int64_t)ctx->sm_count * 8;
    int64_t rounds = (groups + 255) / 256 / cap;
    if (q < 4 || rounds >= 8) rounds = (groups + cap * 256 - 1) / (cap * 256);
    const int64_t per_block = 256 * (rounds < 1 ? 1 : rounds), nb = (groups + per_block - 1) / per_block;
    auto kern = per_block > 256 ? (sgd ? zo_update_kernel<true, 2> : zo_update_kernel<false, 2>)
                                : (sgd ? zo_update_kernel<true, 1> : zo_update_kernel<false, 1>);
    ZOACT_CUDA_TRY(launch_pdl(ctx, kern, dim3((unsigned)nb),
                              dim3(256), 0, C, m, v, tab, g_begin, g_end, per_block, a, q, qs, lr, b1, b2, adam_eps, step_size,
                              inv_sqrt_bc2, seed, ctx->d_status));
    ++ctx->n_launch;
  }
  return ZOACT_OK;
}

}  // namespace zoact
