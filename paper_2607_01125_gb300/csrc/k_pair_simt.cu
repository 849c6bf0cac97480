// Pair / multi-point forward on CUDA cores for fp32 weights and activations
// (Section 3; Algorithm 2):
//   y_b = W x + (C + c_b Z_b)(U^T x)      for the evaluation blocks b
// fp32 inputs have no dense tensor-core path with fp32 accuracy (tf32 keeps a
// 10-bit mantissa), so this kernel serves the fp32 workloads (the 256-wide toy
// graph), which are latency-bound: what counts is how many SMs take part and how
// many round trips to L2 a block makes.  A block of 256 threads owns a
// (16 TM) x (16 TM) output tile, TM x TM outputs per thread; X and W come by 16-byte
// cp.async into a ring of 32-wide K chunks (STAGES of them in flight at once: all of
// a 256-wide layer for the smallest tile), and each output is one chain of FMAs in
// ascending k, whatever the tile.
// While the first chunks are under way the block builds the table C + c_b Z_b of
// its columns (32 ranks at a time, Z from the shared Philox generator) and takes its
// rows of P to shared memory; the low-rank term is added in fp32 at the end: stacked
// rows use their own block, shared rows are written once per block.
//
// Tile: the largest whose blocks fill half of the SMs, else 16 x 16.  64 rows x 256 x
// 256, both signs written (ncu): 64.9 us on four 64 x 64 blocks with 16-wide chunks and
// scalar loads, 8.1 on 64 of 16 x 16; the toy ZO step (64 tokens) 152 -> 56 us, its launches then paced by the host.
#include "internal.h"
#include "philox.cuh"

namespace zoact {
namespace {

constexpr int SKC = 32;          // K chunk
constexpr int SLD = SKC + 4;     // row stride of a chunk in shared memory (floats): 16-byte rows, spread over the banks
constexpr int SR = 32;           // ranks per epilogue table chunk

struct EvalBlocks {
  int nb;
  float coef[ZOACT_MAX_EVAL_BLOCKS];
  uint64_t qry[ZOACT_MAX_EVAL_BLOCKS];
};

__host__ __device__ constexpr int simt_stages(int tm) { return tm == 1 ? 8 : tm == 2 ? 6 : 4; }

__device__ __forceinline__ void cp_async16(float* dst, const float* src, bool ok) {
  const uint32_t s = (uint32_t)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(s), "l"(src), "r"(ok ? 16 : 0) : "memory");
}

template <int TM>
__host__ __device__ constexpr int simt_smem() {
  const int b = 16 * TM;
  return (simt_stages(TM) * 2 * b * SLD + 2 * b * (SR + 1)) * 4;
}

template <int TM>
__global__ void __launch_bounds__(256)
pair_simt_kernel(const float* __restrict__ X, const float* __restrict__ W, const float* __restrict__ P,
                 const float* __restrict__ Cg, float* __restrict__ Y, int64_t rows, int64_t T, int d_in,
                 int d_out, int r, int shared_in, int act, const __grid_constant__ EvalBlocks blk, uint64_t seed,
                 uint32_t layer_id) {
  constexpr int B = 16 * TM, ST = simt_stages(TM);
  extern __shared__ __align__(16) float sm[];
  float* Tt = sm + ST * 2 * B * SLD;                 // [B][SR + 1] table
  float* Ps = Tt + B * (SR + 1);                     // [B][SR + 1] projections
  const int tid = threadIdx.x;
  const int tx = tid % 16, ty = tid / 16;
  const int64_t m0 = (int64_t)blockIdx.y * B;
  const int n0 = blockIdx.x * B;
  const int n_chunks = (d_in + SKC - 1) / SKC;
  pdl_wait();                                        // X, P and C written by the previous kernels
  pdl_trigger();

  // chunk c into its stage: 16-byte pieces of the tile's X rows, then of its W rows; zero outside
  auto load = [&](int c) {
    if (c < n_chunks) {
      float* st = sm + (c % ST) * 2 * B * SLD;
      for (int v = tid; v < 2 * B * (SKC / 4); v += 256) {
        const int row = v / (SKC / 4), k = c * SKC + (v % (SKC / 4)) * 4;
        const bool is_w = row >= B;
        const int64_t g = is_w ? n0 + row - B : m0 + row;
        const bool ok = k < d_in && g < (is_w ? (int64_t)d_out : rows);   // (d_in is a multiple of 4)
        cp_async16(st + row * SLD + (v % (SKC / 4)) * 4, (is_w ? W : X) + (ok ? g * d_in + k : 0), ok);
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
#pragma unroll
  for (int c = 0; c < ST - 1; ++c) load(c);

  // blocks this tile's rows touch (all of them when the input is shared)
  int b_first = 0, b_last = blk.nb - 1;
  if (!shared_in) {
    const int64_t last = (m0 + B < rows ? m0 + B : rows) - 1;
    b_first = (int)(m0 / T);
    b_last = (int)(last / T);
  }
  const int n_cols = min(B, d_out - n0);
  // ranks [jc, jc + rc) of the table of block b (and of P, whose rows do not depend on b)
  auto build = [&](int b, int jc, int rc, bool with_p) {
    const float cb = blk.coef[b];
    if ((r & 3) == 0) {                              // whole Philox groups: jc and rc are multiples of 4
      for (int v = tid; v < n_cols * (rc / 4); v += 256) {
        const int c = v / (rc / 4), j = (v % (rc / 4)) * 4;
        const int64_t e = (int64_t)(n0 + c) * r + jc + j;
        float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
        if (cb != 0.f) z = z_normals4(seed, layer_id, blk.qry[b], (uint64_t)(e >> 2));
        float* t = Tt + c * (SR + 1) + j;
        t[0] = fmaf(cb, z.x, Cg[e]);
        t[1] = fmaf(cb, z.y, Cg[e + 1]);
        t[2] = fmaf(cb, z.z, Cg[e + 2]);
        t[3] = fmaf(cb, z.w, Cg[e + 3]);
      }
    } else {
      for (int v = tid; v < n_cols * rc; v += 256) {
        const int c = v / rc, j = v % rc;
        const int64_t e = (int64_t)(n0 + c) * r + jc + j;
        const float z = cb != 0.f ? z_select(z_normals4(seed, layer_id, blk.qry[b], (uint64_t)(e >> 2)), (int)(e & 3))
                                  : 0.f;
        Tt[c * (SR + 1) + j] = fmaf(cb, z, Cg[e]);
      }
    }
    if (with_p)
      for (int v = tid; v < B * rc; v += 256) {
        const int rr = v / rc, j = v % rc;
        Ps[rr * (SR + 1) + j] = m0 + rr < rows ? P[(m0 + rr) * r + jc + j] : 0.f;
      }
  };
  build(b_first, 0, min(SR, r), true);               // the main loop's barriers order it before its use

  // outputs (ty + 16 i, tx + 16 j) of the tile
  float acc[TM][TM] = {};
  for (int c = 0; c < n_chunks; ++c) {
    load(c + ST - 1);
    asm volatile("cp.async.wait_group %0;" ::"n"(ST - 1) : "memory");
    __syncthreads();
    const float* Xs = sm + (c % ST) * 2 * B * SLD;
    const float* Ws = Xs + B * SLD;
#pragma unroll
    for (int k = 0; k < SKC; k += 4) {
      float4 a[TM], w[TM];
#pragma unroll
      for (int i = 0; i < TM; ++i) {
        a[i] = *reinterpret_cast<const float4*>(Xs + (ty + 16 * i) * SLD + k);
        w[i] = *reinterpret_cast<const float4*>(Ws + (tx + 16 * i) * SLD + k);
      }
#pragma unroll
      for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TM; ++j) {
          acc[i][j] = fmaf(a[i].x, w[j].x, acc[i][j]);
          acc[i][j] = fmaf(a[i].y, w[j].y, acc[i][j]);
          acc[i][j] = fmaf(a[i].z, w[j].z, acc[i][j]);
          acc[i][j] = fmaf(a[i].w, w[j].w, acc[i][j]);
        }
    }
    __syncthreads();                                 // the stage is free for chunk c + ST
  }

  for (int b = b_first; b <= b_last; ++b) {
    float sl[TM][TM] = {};
    for (int jc = 0; jc < r; jc += SR) {
      const int rc = min(SR, r - jc);
      if (b != b_first || jc > 0) {
        __syncthreads();
        build(b, jc, rc, r > SR);
        __syncthreads();
      }
      for (int jj = 0; jj < rc; ++jj) {
        float pj[TM], t[TM];
#pragma unroll
        for (int i = 0; i < TM; ++i) {
          pj[i] = Ps[(ty + 16 * i) * (SR + 1) + jj];
          t[i] = Tt[(tx + 16 * i) * (SR + 1) + jj];
        }
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
          for (int j = 0; j < TM; ++j) sl[i][j] = fmaf(t[j], pj[i], sl[i][j]);
      }
    }
#pragma unroll
    for (int i = 0; i < TM; ++i) {
      const int64_t m = m0 + ty + 16 * i;
      if (m >= rows || (!shared_in && m / T != b)) continue;
      const int64_t row = shared_in ? (int64_t)b * T + m : m;
#pragma unroll
      for (int j = 0; j < TM; ++j) {
        const int n = n0 + tx + 16 * j;
        if (n < d_out) Y[row * d_out + n] = apply_act(acc[i][j] + sl[i][j], act);
      }
    }
  }
}

template <int TM>
int launch_simt(Ctx* ctx, const PairArgs& a, const EvalBlocks& blk) {
  constexpr int B = 16 * TM;
  auto kern = pair_simt_kernel<TM>;
  ZOACT_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, simt_smem<TM>()));
  const dim3 grid((unsigned)((a.d_out + B - 1) / B), (unsigned)((a.rows + B - 1) / B));
  ZOACT_CUDA_TRY(launch_pdl(ctx, kern, grid, dim3(256), simt_smem<TM>(), static_cast<const float*>(a.X),
                            static_cast<const float*>(a.W), a.P, a.C, static_cast<float*>(a.Y), a.rows, a.T, a.d_in,
                            a.d_out, a.r, a.shared, a.act, blk, a.seed, a.layer_id));
  ++ctx->n_launch;
  ZOACT_CHECK_LAUNCH();
  return ZOACT_OK;
}

}  // namespace

int launch_pair_simt(Ctx* ctx, const PairArgs& a) {
  if (a.nseg > 1) return ZOACT_ERR_UNSUPPORTED;     // layers run as one: 16-bit activations only
  if (a.xdtype != ZOACT_DT_FP32 || a.wtype != ZOACT_DT_FP32 || a.ydtype != ZOACT_DT_FP32)
    return ZOACT_ERR_UNSUPPORTED;
  if (a.W2) return ZOACT_ERR_UNSUPPORTED;
  EvalBlocks blk{};
  blk.nb = a.nb;
  for (int b = 0; b < a.nb; ++b) { blk.coef[b] = a.coef[b]; blk.qry[b] = a.qry[b]; }
  auto blocks = [&](int tile) { return ((a.rows + tile - 1) / tile) * (int64_t)((a.d_out + tile - 1) / tile); };
  const int64_t enough = ctx->sm_count / 2;
  // (the grid's y dimension ends at 65535 row tiles: the smaller tiles are only taken where there are few)
  if (blocks(64) >= enough) return launch_simt<4>(ctx, a, blk);
  if (blocks(32) >= enough) return launch_simt<2>(ctx, a, blk);
  return launch_simt<1>(ctx, a, blk);
}

}  // namespace zoact
