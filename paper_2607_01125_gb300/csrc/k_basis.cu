// One-shot activation basis (Algorithm 1: top-r right singular vectors of the
// calibration activations X, i.e. the top-r eigenvectors of G = X^T X).
//
// Device pipeline (no host round trip, every step a kernel):
//   1. For 16-bit X, X is transposed into a zero-padded [d, n_pad] copy, and every
//      product G Q is X^T (X Q) on the tensor cores, in three 16-bit terms of the
//      fp32 factor.  Only with many more tokens than columns, and for fp32 X, is
//      G = X^T X formed (fp32; tcgen05 GEMM, or CUDA cores for fp32 X).
//   2. Omega [d, k] from the Z generator (seed, layer 0, query 0), k = r + oversample.
//   3. Q = orth(Omega); n_iter times Q = orth(G Q).  orth() is CholeskyQR2:
//      S = Y^T Y (64 x 64 output tiles; fp32 over 32-row slabs, fp64 or two floats
//      across slabs, fp64 across row chunks), R^-1 of the Cholesky factor S = R^T R (fp64),
//      Q = Y R^-1; done twice for orthogonality.
//   4. Rayleigh-Ritz: S = Q^T G Q (fp64), Jacobi (fp64): two-sided in one block's
//      shared memory for k <= 64, one-sided on the Cholesky factor over the whole
//      chip above; eigenpairs sorted by value, U = Q V[:, :r], each column flipped so
//      its largest-magnitude entry is positive (first index on ties).
//   k = r + oversample <= 512.
#include "internal.h"
#include "philox.cuh"

namespace zoact {
namespace {

constexpr int KMAX = 64;        // k handled by the shared-memory Cholesky and Jacobi; column tile of the rest
constexpr int KLIM = 512;       // largest k

// ---- X [n, d] (16-bit, d a multiple of 8, 16-byte aligned) -> Xt [d, n_pad], zero in columns n .. n_pad-1 ----
// 64 x 64 tiles, 16-byte loads and stores.  absmax (or null; zero before): max |X|, one atomic per block that raises it.
// 4096 x 5120 fp16: 111 us as 32 x 32 tiles of single elements with an atomic per warp (45 without), 22 here.
template <typename T>
__global__ void __launch_bounds__(256) transpose_pad_kernel(const T* __restrict__ X, T* __restrict__ Xt, int64_t n, int d,
                                                            int64_t n_pad, int* __restrict__ absmax) {
  __shared__ T tile[64][66];                         // [token][column]
  __shared__ int top_s;
  const int64_t t0 = (int64_t)blockIdx.x * 64;
  const int i0 = blockIdx.y * 64;
  if (threadIdx.x == 0) top_s = 0;
  __syncthreads();
  int top = 0;
  for (int v = threadIdx.x; v < 64 * 8; v += 256) {
    const int y = v >> 3, c = (v & 7) * 8;
    union { uint4 w; T e[8]; } u;
    u.w = make_uint4(0u, 0u, 0u, 0u);
    if (t0 + y < n && i0 + c < d) u.w = *reinterpret_cast<const uint4*>(X + (t0 + y) * d + i0 + c);
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      tile[y][c + e] = u.e[e];
      top = max(top, __float_as_int(fabsf(to_f32<T>(u.e[e]))));    // non-negative floats order as integers
    }
  }
  if (absmax) {
    top = __reduce_max_sync(0xffffffffu, top);
    if ((threadIdx.x & 31) == 0) atomicMax(&top_s, top);
  }
  __syncthreads();
  if (absmax && threadIdx.x == 0 && top_s > *reinterpret_cast<volatile int*>(absmax)) atomicMax(absmax, top_s);
  for (int v = threadIdx.x; v < 64 * 8; v += 256) {
    const int i = v & 63, y = (v >> 6) * 8;
    if (i0 + i < d && t0 + y < n_pad) {              // (n_pad is a multiple of 8)
      union { uint4 w; T e[8]; } u;
#pragma unroll
      for (int e = 0; e < 8; ++e) u.e[e] = tile[y + e][i];
      *reinterpret_cast<uint4*>(Xt + (int64_t)(i0 + i) * n_pad + t0 + y) = u.w;
    }
  }
}

// ---- G = X^T X for fp32 X [n, d] (CUDA cores, 64x64 tiles) ----
__global__ void __launch_bounds__(256) gram_f32_kernel(const float* __restrict__ X, float* __restrict__ G, int64_t n,
                                                       int d) {
  __shared__ float As[16][64 + 4];
  __shared__ float Bs[16][64 + 4];
  const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
  const int i0 = blockIdx.y * 64, j0 = blockIdx.x * 64;
  float acc[4][4] = {};
  for (int64_t t0 = 0; t0 < n; t0 += 16) {
    __syncthreads();
    for (int v = threadIdx.x; v < 16 * 64; v += 256) {
      const int kk = v / 64, c = v % 64;
      const int64_t t = t0 + kk;
      As[kk][c] = (t < n && i0 + c < d) ? X[t * d + i0 + c] : 0.f;
      Bs[kk][c] = (t < n && j0 + c < d) ? X[t * d + j0 + c] : 0.f;
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < 16; ++kk) {
      float a[4], b[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) { a[q] = As[kk][ty * 4 + q]; b[q] = Bs[kk][tx * 4 + q]; }
#pragma unroll
      for (int p = 0; p < 4; ++p)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[p][q] = fmaf(a[p], b[q], acc[p][q]);
    }
  }
  for (int p = 0; p < 4; ++p)
    for (int q = 0; q < 4; ++q) {
      const int i = i0 + ty * 4 + p, j = j0 + tx * 4 + q;
      if (i < d && j < d) G[(int64_t)i * d + j] = acc[p][q];
    }
}

// ---- Omega [d, k]: element i*k + j of the (seed, 0, 0) stream ----
__global__ void omega_kernel(float* __restrict__ Om, int64_t n, uint64_t seed) {
  pdl_wait();
  pdl_trigger();
  for (int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; 4 * g < n; g += (int64_t)gridDim.x * blockDim.x) {
    const float4 z = z_normals4(seed, 0u, 0ull, (uint64_t)g);
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (4 * g + i < n) Om[4 * g + i] = z_select(z, i);
  }
}

// ---- Y [d, k] = G [d, d] * Q [d, k] (fp32, 64-row x 64-column blocks, K staged in chunks of 32) ----
__global__ void __launch_bounds__(256) gemm_gq_kernel(const float* __restrict__ G, const float* __restrict__ Q,
                                                      float* __restrict__ Y, int d, int k) {
  const int c0 = blockIdx.y * KMAX;
  __shared__ float Gs[64][33];
  __shared__ __align__(16) float Qs[32][KMAX];
  const int cg = threadIdx.x % 16, rg = threadIdx.x / 16;  // 16 col groups x 16 row groups (4x4 each)
  const int64_t i0 = (int64_t)blockIdx.x * 64;
  float acc[4][4] = {};
  for (int k0 = 0; k0 < d; k0 += 32) {
    __syncthreads();
    for (int v = threadIdx.x; v < 64 * 32; v += 256) {
      const int rr = v / 32, kk = v % 32;
      Gs[rr][kk] = (i0 + rr < d && k0 + kk < d) ? G[(i0 + rr) * d + k0 + kk] : 0.f;
    }
    for (int v = threadIdx.x; v < 32 * KMAX; v += 256) {
      const int kk = v / KMAX, c = v % KMAX;
      Qs[kk][c] = (k0 + kk < d && c0 + c < k) ? Q[(int64_t)(k0 + kk) * k + c0 + c] : 0.f;
    }
    __syncthreads();
#pragma unroll 8
    for (int kk = 0; kk < 32; ++kk) {
      const float4 q = *reinterpret_cast<const float4*>(&Qs[kk][cg * 4]);
#pragma unroll
      for (int p = 0; p < 4; ++p) {
        const float g = Gs[rg * 4 + p][kk];
        acc[p][0] = fmaf(g, q.x, acc[p][0]);
        acc[p][1] = fmaf(g, q.y, acc[p][1]);
        acc[p][2] = fmaf(g, q.z, acc[p][2]);
        acc[p][3] = fmaf(g, q.w, acc[p][3]);
      }
    }
  }
  for (int p = 0; p < 4; ++p) {
    const int64_t i = i0 + rg * 4 + p;
    if (i >= d) continue;
    for (int c = 0; c < 4; ++c) {
      const int j = c0 + cg * 4 + c;
      if (j < k) Y[i * k + j] = acc[p][c];
    }
  }
}

// ---- partial S = A^T B over a chunk of rows, A, B [rows, k]: 64 x 64 output tiles per block (grid x, y), row chunks on
// grid z; fp32 products over 32-row slabs, added into fp64 per slab -- where there are several tiles (TILES), and the fp64
// adds of their many slabs would weigh twice their FMAs, into two floats that carry the rounding errors along (~46 bits;
// k = 272: 67 us a call with fp64 adds, 47 so; one tile, bound by latency: 9.4 with fp64, 11.8).  sym (A = B): tiles below the diagonal are left out.  A slab is a round
// trip to L2, so the rows are cut into as many chunks as give every SM two tiles: 7 blocks of 64 slabs took 296 us for
// 14336 x 32, 13 here (and 7 for the sum of the chunks).
template <bool TILES>
__global__ void __launch_bounds__(256) atb_partial_kernel(const float* __restrict__ A, const float* __restrict__ B,
                                                          double* __restrict__ part, int64_t rows, int k, int chunk,
                                                          int sym) {
  __shared__ float As[32][KMAX + 4];
  __shared__ float Bs[32][KMAX + 4];
  pdl_wait();
  pdl_trigger();
  const int p0 = blockIdx.y * KMAX, q0 = blockIdx.x * KMAX;
  if (sym && q0 < p0) return;
  const bool one = sym && q0 == p0;                  // one tile serves both sides
  const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
  const int64_t r_begin = (int64_t)blockIdx.z * chunk;
  const int64_t r_end = r_begin + chunk < rows ? r_begin + chunk : rows;
  const bool live = p0 + ty * 4 < k && q0 + tx * 4 < k;
  float acc[4][4] = {}, low[4][4] = {};
  double acc64[4][4] = {};
  for (int64_t s0 = r_begin; s0 < r_end; s0 += 32) {
    __syncthreads();
    for (int v = threadIdx.x; v < 32 * KMAX; v += 256) {
      const int rr = v / KMAX, c = v % KMAX;
      const int64_t row = s0 + rr;
      As[rr][c] = (row < r_end && p0 + c < k) ? A[row * k + p0 + c] : 0.f;
      if (!one) Bs[rr][c] = (row < r_end && q0 + c < k) ? B[row * k + q0 + c] : 0.f;
    }
    __syncthreads();
    if (live) {
      float (*Bt)[KMAX + 4] = one ? As : Bs;
      float a32[4][4] = {};
#pragma unroll 8
      for (int rr = 0; rr < 32; ++rr) {
        const float4 a = *reinterpret_cast<const float4*>(&As[rr][ty * 4]);
        const float4 b = *reinterpret_cast<const float4*>(&Bt[rr][tx * 4]);
        const float av[4] = {a.x, a.y, a.z, a.w}, bv[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j) a32[i][j] = fmaf(av[i], bv[j], a32[i][j]);
      }
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          if (!TILES) {
            acc64[i][j] += (double)a32[i][j];
            continue;
          }
          const float x = a32[i][j], t = __fadd_rn(acc[i][j], x), y = __fsub_rn(t, acc[i][j]);
          low[i][j] = __fadd_rn(low[i][j], __fadd_rn(__fsub_rn(acc[i][j], __fsub_rn(t, y)), __fsub_rn(x, y)));
          acc[i][j] = t;
        }
    }
  }
  if (!live) return;
  double* out = part + (int64_t)blockIdx.z * k * k;
  for (int i = 0; i < 4; ++i)
    for (int j = 0; j < 4; ++j) {
      const int p = p0 + ty * 4 + i, q = q0 + tx * 4 + j;
      if (p < k && q < k) out[(int64_t)p * k + q] = TILES ? (double)acc[i][j] + (double)low[i][j] : acc64[i][j];
    }
}

// S = the chunks' partials, eight strided slices of them per output added last; SYM: the upper triangle, mirrored; else
// (S + S^T) / 2, which the two roundings of Q^T (G Q) leave a little apart.
template <bool SYM>
__global__ void __launch_bounds__(256) sum_partials_kernel(const double* __restrict__ part, double* __restrict__ S,
                                                           int nchunk, int k) {
  __shared__ double red[SYM ? 1 : 2][8][32];
  pdl_wait();
  pdl_trigger();
  const int lane = threadIdx.x & 31, slice = threadIdx.x >> 5;
  const int o = blockIdx.x * 32 + lane, kk = k * k;
  const int i = o / k, j = o - i * k;
  const bool live = o < kk && !(SYM && i > j);
  double s = 0.0, t = 0.0;
  if (live)
#pragma unroll 4
    for (int b = slice; b < nchunk; b += 8) s += part[(int64_t)b * kk + o];
  red[0][slice][lane] = s;
  if constexpr (!SYM) {
    if (live)
#pragma unroll 4
      for (int b = slice; b < nchunk; b += 8) t += part[(int64_t)b * kk + j * k + i];
    red[1][slice][lane] = t;
  }
  __syncthreads();
  if (slice != 0 || !live) return;
#pragma unroll
  for (int w = 1; w < 8; ++w) s += red[0][w][lane];
  if constexpr (SYM) {
    S[o] = S[j * k + i] = s;
  } else {
#pragma unroll
    for (int w = 1; w < 8; ++w) t += red[1][w][lane];
    S[o] = 0.5 * (s + t);
  }
}

// ---- LDL^T of an n x n block in shared memory (n <= KMAX), with its inverse factor ----
// N: the upper triangle in, zeros below; out: row j of the eliminated matrix in the upper triangle (its diagonal D) and
// L^-1 (unit lower triangle) strictly below.  One block-wide barrier a column: while the other warps apply column j to
// the rows below, which they keep in registers until the row is the next but one, warp 0 finishes row j + 1 for its
// multipliers and for the step after (one or two columns a lane).
// A scheduler takes a warp's fp64 instruction in 68 cycles (whatever its active lanes), so a column's time is warp 0's
// chain, 710 to 810 cycles (nine such, five in the reciprocal; warps 4, 8, ... leave it the scheduler), or the other
// warps' row updates, 68 for each of the rows below over three schedulers, more beyond 32 columns.  With the rows in
// shared memory (three reads and a write an element), a comparison in the chain and a check of it every column: a factor
// of 32 columns with its inverse 23.6 us, 48 columns 43.6; 18.4 and 38.7 here.
// Returns false (to every thread) when a pivot is not positive.  f: 2 x KMAX doubles, bad: an int.
constexpr int LDL_ROWS = 6;                          // rows a warp may own: 64 over 12 warps, 32 over 6
__device__ bool ldl_shared(double* N, int ld, int n, double* f, int* bad) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
  const bool wide = n > 32, in0 = lane < n, in1 = lane + 32 < n;
  const int workers = warps - (warps + 3) / 4, mine = warp - 1 - warp / 4;
  const bool worker = (warp & 3) != 0;
  double x0 = 0.0, x1 = 0.0, f0 = 0.0, f1 = 0.0;     // warp 0: row j (1 in column j) and its multipliers
  bool fail = false;
  auto pivot = [&](int p, double a0, double a1) {    // warp 0: row p is eliminated: its multipliers
    const double d = __shfl_sync(0xffffffffu, p < 32 ? a0 : a1, p & 31);
    const double inv = 1.0 / d;
    double* fp = f + (p & 1) * KMAX;
    f0 = a0 * inv;
    fp[lane] = f0;
    if (wide) {
      f1 = a1 * inv;
      fp[lane + 32] = f1;
    }
    const long long bits = __double_as_longlong(d);  // (an fp64 comparison would be one more in the chain)
    fail = fail || bits <= 0 || bits > 0x7ff0000000000000ll;
    x0 = lane == p ? 1.0 : a0;
    x1 = lane + 32 == p ? 1.0 : a1;
  };
  // the other warps: columns 0 .. 31 of rows mine + s workers (r0), and from 32 on (r1) as many, or where they are at most
  // 16 those of two rows, one per half warp
  const bool two = n <= 48;
  const int c1 = 32 + (two ? lane & 15 : lane);
  auto row1 = [&](int s) { return mine + (two ? 2 * s + (lane >> 4) : s) * workers; };
  double r0[LDL_ROWS], r1[LDL_ROWS];
#pragma unroll
  for (int s = 0; s < LDL_ROWS; ++s) {
    const int p = mine + s * workers, q = row1(s);
    r0[s] = worker && p < n && in0 ? N[p * ld + lane] : 0.0;
    r1[s] = worker && q < n && c1 < n ? N[q * ld + c1] : 0.0;
  }
  if (warp == 0) pivot(0, in0 ? N[lane] : 0.0, in1 ? N[lane + 32] : 0.0);
  __syncthreads();
  for (int j = 0; j < n - 1; ++j) {
    if (warp == 0) {
      const int p = j + 1;
      double* row = N + p * ld;
      double a0 = in0 ? row[lane] : 0.0, a1 = in1 ? row[lane + 32] : 0.0;
      const double m = __shfl_sync(0xffffffffu, p < 32 ? f0 : f1, p & 31);
      a0 = fma(-m, x0, a0);                          // (columns 0 .. j and p .. n: all of them)
      if (in0) row[lane] = a0;
      if (wide) {
        a1 = fma(-m, x1, a1);
        if (in1) row[lane + 32] = a1;
      }
      pivot(p, a0, a1);
    } else if (worker) {
      const double* fj = f + (j & 1) * KMAX;
      double m[LDL_ROWS];
#pragma unroll
      for (int s = 0; s < LDL_ROWS; ++s) m[s] = fj[min(mine + s * workers, KMAX - 1)];
      const double y0 = lane == j ? 1.0 : in0 ? N[j * ld + lane] : 0.0;
#pragma unroll
      for (int s = 0; s < LDL_ROWS; ++s) {
        const int p = mine + s * workers;
        if (p > j + 1 && p < n) {                    // columns 0 .. j and from p on
          if (lane <= j || lane >= p) r0[s] = fma(-m[s], y0, r0[s]);
          if (p == j + 2 && in0) N[p * ld + lane] = r0[s];
        }
      }
      if (wide) {
#pragma unroll
        for (int s = 0; s < LDL_ROWS; ++s) m[s] = fj[min(row1(s), KMAX - 1)];
        const double y1 = c1 == j ? 1.0 : c1 < n ? N[j * ld + c1] : 0.0;
#pragma unroll
        for (int s = 0; s < LDL_ROWS; ++s) {
          const int p = row1(s);
          if (__any_sync(0xffffffffu, p > j + 1 && p < n)) {
            if (p > j + 1 && p < n && (c1 <= j || c1 >= p)) r1[s] = fma(-m[s], y1, r1[s]);
            if (p == j + 2 && c1 < n) N[p * ld + c1] = r1[s];
          }
        }
      }
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) *bad = fail;
  __syncthreads();
  return *bad == 0;
}

// The diagonal shift of attempt 0, 1, 2, ...: none, then 1e-12 of the trace, a thousand times more each time.
__device__ __forceinline__ double chol_shift(int attempt, double trace) {
  double s = attempt == 0 ? 0.0 : 1e-12 * trace;
  for (int i = 1; i < attempt; ++i) s *= 1e3;
  return s;
}
constexpr int CHOL_ATTEMPTS = 4;

// ---- R^-1 of the Cholesky factor S = R^T R (R upper), k <= KMAX: one block, everything in shared memory ----
// R^-1 = L^-T D^-1/2.  Bound by a column's chain (a row's update, a division, a barrier) and the fp64 pipe; k = 48:
// 228 us with the factor in global memory and a serial inverse per column, 39 here.
constexpr int CHOL_THREADS = 512;       // (half of it to 32 columns: as many rows a warp, fewer warps at the barrier)
constexpr int CHOL_SMEM = KMAX * (KMAX + 1) * 8;
__global__ void __launch_bounds__(CHOL_THREADS) chol_inv_kernel(const double* __restrict__ S, double* __restrict__ Rinv,
                                                                int k, int* status) {
  extern __shared__ double sm[];
  __shared__ double f[2 * KMAX], rs[KMAX], trace;
  __shared__ int bad;
  pdl_wait();
  pdl_trigger();
  const int ld = k + 1;
  bool ok = false;
  for (int attempt = 0; attempt < CHOL_ATTEMPTS && !ok; ++attempt) {
    __syncthreads();
    if (threadIdx.x == 0 && attempt == 1) {
      trace = 0.0;
      for (int i = 0; i < k; ++i) trace += S[i * k + i];
    }
    __syncthreads();
    const double shift = chol_shift(attempt, attempt ? trace : 0.0);
    for (int v = threadIdx.x; v < k * k; v += blockDim.x) {
      const int i = v / k, j = v % k;
      sm[i * ld + j] = j < i ? 0.0 : S[v] + (i == j ? shift : 0.0);
    }
    __syncthreads();
    ok = ldl_shared(sm, ld, k, f, &bad);
  }
  if (!ok) {
    if (threadIdx.x == 0) record_error(status, ZOACT_ERR_NONFINITE);
    return;
  }
  for (int i = threadIdx.x; i < k; i += blockDim.x) rs[i] = 1.0 / sqrt(sm[i * ld + i]);
  __syncthreads();
  for (int v = threadIdx.x; v < k * k; v += blockDim.x) {
    const int i = v / k, c = v % k;
    Rinv[v] = i > c ? 0.0 : (i == c ? 1.0 : sm[c * ld + i]) * rs[c];
  }
}

// ---- grid barrier of a cooperative launch: bounded (2 s); a barrier that gives up records ZOACT_ERR_TIMEOUT and
// releases the others through the abort word ----
constexpr int HJ_SWEEPS = 40;
struct GridSync {
  unsigned int count;             // arrivals since the launch
  int abort;
  int rotated[HJ_SWEEPS];         // large Jacobi: a sweep rotated something
};
__device__ __forceinline__ bool grid_barrier(GridSync* sy, unsigned int target, int* status) {
  __shared__ int give_up;
  __syncthreads();
  if (threadIdx.x == 0) {
    give_up = 0;
    // the block's writes, ordered before this thread by the barrier above, are released with the arrival
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(&sy->count) : "memory");
    unsigned int seen;
    uint64_t t0 = 0;
    for (unsigned int it = 0;; ++it) {
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(&sy->count) : "memory");
      if (seen >= target) break;
      if ((it & 63u) == 63u) {
        uint64_t now;
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(now));
        if (t0 == 0) t0 = now;
        if (*reinterpret_cast<volatile int*>(&sy->abort)) { give_up = 1; break; }
        if (now - t0 > 2000000000ull) {
          atomicExch(&sy->abort, 1);
          record_error(status, ZOACT_ERR_TIMEOUT);
          give_up = 1;
          break;
        }
      }
    }
  }
  __syncthreads();
  return give_up == 0;
}

// ---- R and R^-1 for k > KMAX: blocked LDL^T over the chip (cooperative) ----
// Panels of CB columns.  Every block factors the panel's diagonal block by itself (no barrier), the panel's rows of A
// and of M = L^-1 are multiplied by its inverse factor in 8-column strips, and after a barrier the rows below get their
// rank-CB update in 16 x 16 tiles.  Two barriers a panel; the columns' chain (as above) is most of the time.  k = 272:
// 5.6 ms in one block, 0.21 here.
constexpr int CB = 32;
constexpr int CHOLB_THREADS = 256;
constexpr int CHOLB_BLOCKS = 96;
struct CholBig {
  const double* S;
  double* A;          // S eliminated, then R
  double* M;          // L^-1
  double* Rinv;
  double* D;          // pivots
  double* shift;      // the shift taken
  GridSync* sync;
  int k;
  int any;            // S need not be positive: where those shifts fail, one that no symmetric matrix outweighs
  int* status;
};
__global__ void __launch_bounds__(CHOLB_THREADS) chol_big_kernel(CholBig w) {
  __shared__ double sN[CB * (CB + 1)], f[2 * KMAX], red[CHOLB_THREADS / 32], sum_s;
  __shared__ int bad;
  __shared__ double sx[CB][17], sf[CB][17], inv_d[CB];
  const int k = w.k, tid = threadIdx.x;
  const int64_t gtid = blockIdx.x * (int64_t)CHOLB_THREADS + tid, gthreads = (int64_t)gridDim.x * CHOLB_THREADS;
  unsigned int target = 0;
  auto sync = [&]() { target += gridDim.x; return grid_barrier(w.sync, target, w.status); };
  // the sum of the threads' values, the same in every block
  auto block_sum = [&](double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    __syncthreads();
    if ((tid & 31) == 0) red[tid >> 5] = v;
    __syncthreads();
    if (tid == 0) {
      sum_s = 0.0;
      for (int i = 0; i < CHOLB_THREADS / 32; ++i) sum_s += red[i];
    }
    __syncthreads();
    return sum_s;
  };
  double tr = 0.0;
  for (int i = tid; i < k; i += CHOLB_THREADS) tr += w.S[(int64_t)i * k + i];
  const double trace = block_sum(tr);
  bool ok = false;
  double shift = 0.0;
  for (int attempt = 0; attempt < CHOL_ATTEMPTS + w.any && !ok; ++attempt) {
    shift = chol_shift(attempt, trace);
    if (attempt == CHOL_ATTEMPTS) {
      // eigenvalues of at least |S|_F, at most three times that: as exact, relative to |S|_F, as without a shift
      double sq = 0.0;
      for (int64_t v = tid; v < (int64_t)k * k; v += CHOLB_THREADS) sq = fma(w.S[v], w.S[v], sq);
      shift = 2.0 * sqrt(block_sum(sq));
      if (shift == 0.0) shift = 1.0;
    }
    if (attempt > 0 && !sync()) return;              // every block has seen the failed pivot before A is rewritten
    for (int64_t v = gtid; v < (int64_t)k * k; v += gthreads) {
      const int i = (int)(v / k), j = (int)(v % k);
      __stcg(w.A + v, j >= i ? w.S[v] + (i == j ? shift : 0.0) : 0.0);
      __stcg(w.M + v, i == j ? 1.0 : 0.0);
    }
    if (!sync()) return;
    ok = true;
    for (int p0 = 0; p0 < k; p0 += CB) {
      const int nb = min(CB, k - p0), p1 = p0 + nb;
      for (int v = tid; v < nb * nb; v += CHOLB_THREADS)
        sN[(v / nb) * (CB + 1) + v % nb] = v % nb < v / nb ? 0.0 : __ldcg(w.A + (int64_t)(p0 + v / nb) * k + p0 + v % nb);
      __syncthreads();
      if (!ldl_shared(sN, CB + 1, nb, f, &bad)) { ok = false; break; }     // the same answer in every block
      if (tid < nb) inv_d[tid] = 1.0 / sN[tid * (CB + 1) + tid];
      // strips: columns p1 .. k of A, then 0 .. p0 of M, eight at a time
      const int na = k - p1, cols = na + p0;
      for (int g = blockIdx.x; g * 8 < cols; g += gridDim.x) {
        const int i = tid >> 3, c = g * 8 + (tid & 7);
        double* base = c < na ? w.A + (int64_t)p0 * k + p1 + c : w.M + (int64_t)p0 * k + (c - na);
        if (i < nb && c < cols) sx[i][tid & 7] = __ldcg(base + (int64_t)i * k);
        __syncthreads();
        double x = 0.0;
        if (i < nb && c < cols) {
          x = sx[i][tid & 7];
          for (int l = 0; l < i; ++l) x = fma(sN[i * (CB + 1) + l], sx[l][tid & 7], x);
        }
        if (i < nb && c < cols) __stcg(base + (int64_t)i * k, x);
        __syncthreads();
      }
      if (blockIdx.x == gridDim.x - 1) {             // the diagonal block itself
        for (int v = tid; v < nb * nb; v += CHOLB_THREADS) {
          const int i = v / nb, j = v % nb;
          if (j <= i) __stcg(w.M + (int64_t)(p0 + i) * k + p0 + j, i == j ? 1.0 : sN[i * (CB + 1) + j]);
          if (j >= i) __stcg(w.D + (int64_t)(p0 + i) * k + p0 + j, sN[i * (CB + 1) + j]);
        }
      }
      if (!sync()) return;
      if (p1 >= k) break;
      // rows below: A[q][c] (c >= q) and M[q][c] (c < p1) lose sum_l (X[l][q] / D_l) X[l][c]
      const int nq = (k - p1 + 15) / 16, nm = (p1 + 15) / 16;
      const int ta = nq * (nq + 1) / 2, total = ta + nq * nm;
      for (int t = blockIdx.x; t < total; t += gridDim.x) {
        int qb, cb;
        const bool in_a = t < ta;
        if (in_a) {
          qb = 0;
          int rest = t;
          while (rest >= nq - qb) { rest -= nq - qb; ++qb; }
          cb = qb + rest;
        } else {
          qb = (t - ta) / nm;
          cb = (t - ta) - qb * nm;
        }
        const int q0 = p1 + 16 * qb, c0 = in_a ? p1 + 16 * cb : 16 * cb;
        const int c_end = in_a ? k : p1;
        __syncthreads();
        for (int v = tid; v < nb * 16; v += CHOLB_THREADS) {
          const int l = v >> 4, e = v & 15;
          const int64_t row = (int64_t)(p0 + l) * k;
          sf[l][e] = q0 + e < k ? __ldcg(w.A + row + q0 + e) * inv_d[l] : 0.0;
          double x = 0.0;
          if (c0 + e < c_end)
            x = in_a ? __ldcg(w.A + row + c0 + e) : c0 + e < p0 ? __ldcg(w.M + row + c0 + e)
                : c0 + e - p0 < l ? sN[l * (CB + 1) + c0 + e - p0] : c0 + e - p0 == l ? 1.0 : 0.0;
          sx[l][e] = x;
        }
        __syncthreads();
        const int q = q0 + (tid >> 4), c = c0 + (tid & 15);
        if (q < k && c < c_end && (!in_a || c >= q)) {
          double* dst = (in_a ? w.A : w.M) + (int64_t)q * k + c;
          double x = __ldcg(dst);
          for (int l = 0; l < nb; ++l) x = fma(-sf[l][tid >> 4], sx[l][tid & 15], x);
          __stcg(dst, x);
        }
      }
      if (!sync()) return;
    }
  }
  if (!ok) {
    if (gtid == 0) record_error(w.status, ZOACT_ERR_NONFINITE);
    return;
  }
  if (gtid == 0) *w.shift = shift;
  // R[j][q] = X[j][q] / sqrt(D_j); R^-1 = L^-T D^-1/2 (the diagonal blocks' rows came to D's place)
  for (int64_t v = gtid; v < (int64_t)k * k; v += gthreads) {
    const int i = (int)(v / k), j = (int)(v % k);
    const double di = __ldcg(w.D + (int64_t)i * k + i), dj = __ldcg(w.D + (int64_t)j * k + j);
    if (j >= i) {
      const double x = j / CB == i / CB ? __ldcg(w.D + v) : __ldcg(w.A + v);
      w.Rinv[v] = __ldcg(w.M + (int64_t)j * k + i) / sqrt(dj);
      __stcg(w.A + v, x / sqrt(di));
    } else {
      w.Rinv[v] = 0.0;
      __stcg(w.A + v, 0.0);
    }
  }
}

// ---- products with X on the tensor cores ----
// With 16-bit X and no more than GRAM_TOKENS d tokens the Gram matrix is never formed: G Q = X^T (X Q), two products of
// the projection kernel (k_proj_tc.cu: X exact in 16 bits, the fp32 factor split into three 16-bit terms), the second
// on the transposed copy of X.  A step then reads X twice instead of the d x d matrix (14336 wide, 512 tokens: 29 MB
// against 822 MB) and does 4 n d k operations instead of 2 d^2 k.
// The factors' operand form: rows [g NB + term RT + j] of a [groups NB, ld] 16-bit matrix, rank g RT + j, rows of the
// factor as columns.  fp16 cannot hold the small parts of small entries, so its factors are scaled by powers of two:
// Q, whose entries are at most 1, by 2^13, and P = X Q, bounded by max|X| sqrt(d), to at most 2^14.
struct Operand {
  void* op;
  int64_t ld;
  int rt, nb;
};
constexpr int GRAM_TOKENS = 8;
constexpr float Q_SCALE_FP16 = 8192.f;

template <typename T16> __device__ __forceinline__ float q_scale() { return 1.f; }
template <> __device__ __forceinline__ float q_scale<__half>() { return Q_SCALE_FP16; }
// The power of two that brings max|X| sqrt(d) to [2^13, 2^14).
template <typename T16> __device__ __forceinline__ float p_scale(const int*, int) { return 1.f; }
template <> __device__ __forceinline__ float p_scale<__half>(const int* absmax, int d) {
  const float bound = __int_as_float(*absmax) * sqrtf((float)d);
  if (!(bound > 0.f) || !isfinite(bound)) return 1.f;
  return ldexpf(1.f, 13 - ilogbf(bound));
}

// Eight consecutive rows' values of one rank, scaled, as three 16-bit terms (each the rounding of what is left).
template <typename T16>
__device__ __forceinline__ void write_operand(const Operand& o, int rank, int64_t col, const float* v, float scale) {
  const int g = rank / o.rt, j = rank - g * o.rt;
  T16* row = static_cast<T16*>(o.op) + ((int64_t)g * o.nb + j) * o.ld + col;
  float rest[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) rest[i] = v[i] * scale;
#pragma unroll
  for (int t = 0; t < 3; ++t) {
    union { uint4 w; T16 e[8]; } u;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      u.e[i] = from_f32<T16>(rest[i]);
      rest[i] -= to_f32<T16>(u.e[i]);
    }
    *reinterpret_cast<uint4*>(row + (int64_t)t * o.rt * o.ld) = u.w;
  }
}

// The K-splits' partials [group][split][rows][rt] of a product, added in split order, to out [rows, k] (or null) and,
// TO_OP, to the operand form of the next product (zero in its padding columns).  The scales of the product's own
// operand (Q's: mode 0, P's: mode 1) are taken out.
constexpr int RED_ROWS = 8;
template <typename T16, bool TO_OP>
__global__ void __launch_bounds__(256) reduce_parts_kernel(const float* __restrict__ part, int64_t rows, int k, int splits,
                                                           int rt, float* __restrict__ out, Operand op, int mode,
                                                           const int* __restrict__ absmax, int d) {
  __shared__ float tile[64][RED_ROWS + 1];
  pdl_wait();
  pdl_trigger();
  const int g = blockIdx.y;
  const int64_t r0 = (int64_t)blockIdx.x * RED_ROWS;
  const float* src = part + (int64_t)g * splits * rows * rt;
  const float ps = p_scale<T16>(absmax, d);
  const float un = 1.f / (mode == 0 ? q_scale<T16>() : ps);
  for (int v = threadIdx.x; v < RED_ROWS * rt; v += 256) {
    const int rr = v / rt, j = v - rr * rt;
    const int64_t row = r0 + rr;
    float s = 0.f;
    if (row < rows && g * rt + j < k) {
      const float* p = src + row * rt + j;
#pragma unroll 8
      for (int sp = 0; sp < splits; ++sp) s += __ldg(p + (int64_t)sp * rows * rt);
      s *= un;
      if (out) out[row * k + g * rt + j] = s;
    }
    if (TO_OP) tile[j][rr] = s;
  }
  if (!TO_OP) return;
  __syncthreads();
  for (int v = threadIdx.x; v < rt * (RED_ROWS / 8); v += 256) {
    const int j = v / (RED_ROWS / 8), e = (v % (RED_ROWS / 8)) * 8;
    if (g * rt + j < k && r0 + e < op.ld) {
      float x[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) x[i] = tile[j][e + i];
      write_operand<T16>(op, g * rt + j, r0 + e, x, ps);
    }
  }
}

// ---- out [rows, c] = A [rows, k] (fp32) M [k, ldm] (fp64, first c columns) ----
// Every product is exact (an fp32 entry times a two-float split of M's, 48 bits) and added with its rounding error
// carried along (two-sum), so a sum holds ~46 bits: eleven fp32 instructions a term, against one fp64 FMA at a
// sixty-fourth of their rate.  tri: M is upper triangular.  With a 16-bit T16 the result's operand form is written too.
// 5120 x 48 x 48: 73 us in fp64, 28 here; 4096 x 272 x 272: 836 and 121.
// CT columns by 4096 / CT rows a block (32 columns where k <= 32 or the triangle leaves more out); the widest columns,
// whose sums are longest, come first.
template <typename T16, int CT>
__global__ void __launch_bounds__(256) apply_kernel(const float* __restrict__ A, const double* __restrict__ M,
                                                    float* __restrict__ out, int64_t rows, int k, int ldm, int c,
                                                    int tri, Operand op) {
  constexpr int RT = 4096 / CT, TX = CT / 4;         // rows of the tile; threads along its columns
  constexpr int AP = RT + 4, HB = 2048 / CT, TP = CT + 4;
  __shared__ __align__(16) float As[32 * AP];        // [p][row]; the epilogue's [row of half a tile][column]
  __shared__ __align__(16) float Mh[32][CT], Ml[32][CT];   // [p][column]
  static_assert(HB * TP <= 32 * AP, "the epilogue's tile exceeds the operand's room");
  pdl_wait();
  pdl_trigger();
  const int tx = threadIdx.x % TX, ty = threadIdx.x / TX;
  const int64_t r0 = (int64_t)blockIdx.x * RT;
  const int c0 = (int)(gridDim.y - 1 - blockIdx.y) * CT;
  const bool live = c0 + tx * 4 < c;
  float s[4][4] = {}, lo[4][4] = {};
  const int p_end = tri ? min(k, c0 + CT) : k;
  for (int p0 = 0; p0 < p_end; p0 += 32) {
    __syncthreads();
    for (int v = threadIdx.x; v < RT * 32; v += 256) {
      const int rr = v / 32, p = v % 32;
      As[p * AP + rr] = r0 + rr < rows && p0 + p < k ? A[(r0 + rr) * k + p0 + p] : 0.f;
    }
    for (int v = threadIdx.x; v < 32 * CT; v += 256) {
      const int p = v / CT, cc = v % CT;
      const double m = p0 + p < k && c0 + cc < c ? M[(int64_t)(p0 + p) * ldm + c0 + cc] : 0.0;
      const float h = (float)m;
      Mh[p][cc] = h;
      Ml[p][cc] = (float)(m - (double)h);
    }
    __syncthreads();
    if (live) {
#pragma unroll 4
      for (int p = 0; p < 32; ++p) {
        const float4 a4 = *reinterpret_cast<const float4*>(&As[p * AP + ty * 4]);
        const float4 h4 = *reinterpret_cast<const float4*>(&Mh[p][tx * 4]);
        const float4 l4 = *reinterpret_cast<const float4*>(&Ml[p][tx * 4]);
        const float av[4] = {a4.x, a4.y, a4.z, a4.w}, hv[4] = {h4.x, h4.y, h4.z, h4.w}, lv[4] = {l4.x, l4.y, l4.z, l4.w};
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const float pr = __fmul_rn(av[i], hv[j]);
            const float e = __fmaf_rn(av[i], lv[j], __fmaf_rn(av[i], hv[j], -pr));
            const float t = __fadd_rn(s[i][j], pr);
            const float b = __fsub_rn(t, s[i][j]);
            const float err = __fadd_rn(__fsub_rn(s[i][j], __fsub_rn(t, b)), __fsub_rn(pr, b));
            s[i][j] = t;
            lo[i][j] = __fadd_rn(lo[i][j], __fadd_rn(err, e));
          }
      }
    }
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int64_t row = r0 + ty * 4 + i;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      s[i][j] += lo[i][j];
      if (row < rows && c0 + tx * 4 + j < c) out[row * c + c0 + tx * 4 + j] = s[i][j];
    }
  }
  if constexpr (sizeof(T16) == 2) {
    // the tile by columns, half of its rows at a time
    for (int h = 0; h < 2; ++h) {
      __syncthreads();
      if (ty * 4 / HB == h)
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j) As[(ty * 4 % HB + i) * TP + tx * 4 + j] = s[i][j];
      __syncthreads();
      const int cc = threadIdx.x % CT, e = threadIdx.x / CT * 8;
      const int64_t row = r0 + HB * h + e;
      if (c0 + cc < c && row < rows) {               // rows is a multiple of 8 here
        float x[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) x[i] = As[(e + i) * TP + cc];
        write_operand<T16>(op, c0 + cc, row, x, q_scale<T16>());
      }
    }
  }
}

// ---- eigenpairs of S (k x k, fp64), k <= KMAX: two-sided Jacobi in one block ----
// Each round of the round-robin schedule (n = k rounded up to even, n - 1 rounds a sweep) rotates n / 2 disjoint
// pairs: one warp forms the angles, then every thread updates the 2 x 2 blocks J_i^T A J_j of the symmetric matrix in
// shared memory, half of them (i <= j).  Bound by the fp64 pipe (2 lanes a cycle and SM), so the eigenvectors are left
// out: the angles are logged and jacobi_vectors_kernel applies them to every row of V on its own SM.  The matrix is
// padded to n with a zero row, whose rotations are trivial.  Stops when off(A)^2 <= 1e-30 |A|_F^2.
// k = 48: 17.2 ms as rotations taken one by one with the vectors beside them; 0.60 ms here (its vectors 0.07).
constexpr int JAC_THREADS = 512;
constexpr int JAC_SWEEPS = 60;
constexpr int JACOBI_SMEM = KMAX * (KMAX + 1) * 8;
__device__ __forceinline__ int rr_member(int slot, int round, int n) {
  // slot 0 stays; slots 1 .. n-1 rotate by `round`
  int m = slot - 1 + round;
  if (m >= n - 1) m -= n - 1;
  return slot == 0 ? 0 : 1 + m;
}
// The float nearest below |x| 2^(1023 - e), signed: an fp64 value's leading 23 bits, by integer instructions alone.
__device__ __forceinline__ float scaled_float(double x, int e) {
  const int hi = __double2hiint(x), ex = ((hi >> 20) & 0x7ff) - e + 127;
  const uint32_t mant = (((uint32_t)hi & 0xfffffu) << 3) | ((uint32_t)__double2loint(x) >> 29);
  return ex <= 0 ? 0.f : __uint_as_float(((uint32_t)hi & 0x80000000u) | ((uint32_t)ex << 23) | mant);
}
// A rotation (c, s) that zeroes apq to about 2^-20 of itself: its tangent (the smaller root, so |angle| <= pi / 4) is
// formed in fp32, c and s are orthonormal to fp64 for that tangent (rsqrtf and a third-order step).  In fp64 throughout
// the divisions and roots were most of a round: a dependent fp64 instruction takes ~70 cycles.  d = aqq - app.
__device__ __forceinline__ void jacobi_angle(double d, double apq, double& c, double& s) {
  c = 1.0; s = 0.0;
  const int ed = (__double2hiint(d) >> 20) & 0x7ff, eg = ((__double2hiint(apq) >> 20) & 0x7ff) + 1;
  const int e = max(ed, eg);
  if (eg < 3 || e > 2044) return;                    // (a matrix at the ends of fp64's range is left as it is)
  const float fg = 2.f * scaled_float(apq, e);
  if (fg == 0.f) return;                             // below 2^-126 of d
  const float theta = __fdividef(scaled_float(d, e), fg);
  const float t = copysignf(__fdividef(1.f, fabsf(theta) + sqrtf(fmaf(theta, theta, 1.f))), theta);
  if (!(fabsf(t) > 0.f)) return;
  const double td = (double)t, x = fma(td, td, 1.0), y = (double)rsqrtf((float)x);
  const double rr = fma(-x, y * y, 1.0);             // |rr| < 2^-21: y (1 + rr / 2 + 3 rr^2 / 8) is off by 2^-64
  c = fma(y, rr * fma(0.375, rr, 0.5), y);
  s = td * c;
}
// Integers in the order of fp64 values: -0 equals 0, a NaN comes below all others.  With ties broken by index, ranks by
// these keys are a permutation whatever the values (comparisons of a NaN would give several columns one rank).
__device__ __forceinline__ long long order_key(double x) {
  const long long b = __double_as_longlong(x), mag = b & 0x7fffffffffffffffll;
  if (mag > 0x7ff0000000000000ll) return -0x7fffffffffffffffll - 1;
  return b < 0 ? -mag : mag;
}
__global__ void __launch_bounds__(JAC_THREADS) jacobi_kernel(const double* __restrict__ S, double2* __restrict__ log,
                                                             int* __restrict__ n_rounds, double* __restrict__ evals,
                                                             int* __restrict__ order, int k) {
  extern __shared__ double A[];                      // [n][n + 1]
  __shared__ double cs_c[KMAX / 2], cs_s[KMAX / 2];
  __shared__ int pp[KMAX / 2], qq[KMAX / 2];
  __shared__ double red[2][JAC_THREADS / 32];
  pdl_wait();
  pdl_trigger();
  const int n = (k + 1) / 2 * 2, np = n / 2, ld = n + 1;
  const int tid = threadIdx.x;
  for (int v = tid; v < n * n; v += JAC_THREADS) {
    const int i = v / n, j = v % n;
    A[i * ld + j] = i < k && j < k ? 0.5 * (S[i * k + j] + S[j * k + i]) : 0.0;
  }
  const int n_blk = np * (np + 1) / 2;
  int rounds = 0;
  for (int sweep = 0; sweep < JAC_SWEEPS; ++sweep) {
    __syncthreads();
    double off = 0.0, tot = 0.0;
    for (int v = tid; v < n * n; v += JAC_THREADS) {
      const int i = v / n, j = v % n;
      const double a = A[i * ld + j];
      tot += a * a;
      if (i != j) off += a * a;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      off += __shfl_xor_sync(0xffffffffu, off, o);
      tot += __shfl_xor_sync(0xffffffffu, tot, o);
    }
    if ((tid & 31) == 0) { red[0][tid >> 5] = off; red[1][tid >> 5] = tot; }
    __syncthreads();
    off = tot = 0.0;
    for (int w = 0; w < JAC_THREADS / 32; ++w) { off += red[0][w]; tot += red[1][w]; }
    if (!(off > 1e-30 * tot)) break;                 // (also for a matrix that is not finite)
    // elements that could all stay and still meet that bound are not rotated
    const double skip = 1e-30 * tot / ((double)n * (double)n);
    for (int round = 0; round < n - 1; ++round, ++rounds) {
      if (tid < 32 && tid < np) {
        int p = rr_member(tid, round, n), q = rr_member(n - 1 - tid, round, n);
        if (p > q) { const int x = p; p = q; q = x; }
        double c = 1.0, s = 0.0;
        const double apq = A[p * ld + q];
        if (apq * apq > skip) jacobi_angle(A[q * ld + q] - A[p * ld + p], apq, c, s);
        pp[tid] = p; qq[tid] = q; cs_c[tid] = c; cs_s[tid] = s;
        log[(int64_t)rounds * np + tid] = make_double2(c, s);
      }
      __syncthreads();
      for (int b = tid; b < n_blk; b += JAC_THREADS) {
        // block (i, j), i <= j, of the triangle's row-major order counted from its end
        const int r = n_blk - 1 - b;
        int h = (int)((sqrtf(8.0f * (float)r + 1.0f) - 1.0f) * 0.5f);
        if ((h + 1) * (h + 2) / 2 <= r) ++h;
        if (h * (h + 1) / 2 > r) --h;
        const int i = np - 1 - h, j = np - 1 - (r - h * (h + 1) / 2);
        const int pi = pp[i], qi = qq[i], pj = pp[j], qj = qq[j];
        const double ci = cs_c[i], si = cs_s[i], cj = cs_c[j], sj = cs_s[j];
        if (si == 0.0 && sj == 0.0) continue;
        const double a = A[pi * ld + pj], bq = A[pi * ld + qj], cq = A[qi * ld + pj], dq = A[qi * ld + qj];
        const double a1 = cj * a - sj * bq, b1 = sj * a + cj * bq, c1 = cj * cq - sj * dq, d1 = sj * cq + cj * dq;
        const double a2 = ci * a1 - si * c1, c2 = si * a1 + ci * c1, b2 = ci * b1 - si * d1, d2 = si * b1 + ci * d1;
        A[pi * ld + pj] = A[pj * ld + pi] = a2;
        A[qi * ld + qj] = A[qj * ld + qi] = d2;
        A[pi * ld + qj] = A[qj * ld + pi] = b2;
        if (i != j) A[qi * ld + pj] = A[pj * ld + qi] = c2;      // (i = j: the same element)
      }
      __syncthreads();
    }
  }
  if (tid == 0) *n_rounds = rounds;
  for (int i = tid; i < k; i += JAC_THREADS) {       // descending; first index first on ties
    const double e = A[i * ld + i];
    const long long key = order_key(e);
    int rank = 0;
    for (int j = 0; j < k; ++j) {
      const long long f = order_key(A[j * ld + j]);
      if (f > key || (f == key && j < i)) ++rank;
    }
    order[rank] = i;
    evals[rank] = e;
  }
}
// V = the product of the logged rotations, one row per warp (row i of the identity times every J in turn), columns in
// the order of the eigenvalues.
__global__ void __launch_bounds__(32) jacobi_vectors_kernel(const double2* __restrict__ log,
                                                            const int* __restrict__ n_rounds,
                                                            const int* __restrict__ order, double* __restrict__ Vout,
                                                            int k) {
  __shared__ double v[KMAX];
  constexpr int AHEAD = 8;                           // rounds whose angles are loaded together
  pdl_wait();
  pdl_trigger();
  const int n = (k + 1) / 2 * 2, np = n / 2, lane = threadIdx.x;
  const int rounds = *n_rounds;
  for (int j = lane; j < n; j += 32) v[j] = j == (int)blockIdx.x ? 1.0 : 0.0;
  __syncwarp();
  int round = 0;
  for (int r0 = 0; r0 < rounds; r0 += AHEAD) {
    double2 cs[AHEAD];
#pragma unroll
    for (int a = 0; a < AHEAD; ++a)
      cs[a] = lane < np && r0 + a < rounds ? log[(int64_t)(r0 + a) * np + lane] : make_double2(1.0, 0.0);
#pragma unroll
    for (int a = 0; a < AHEAD; ++a) {
      if (r0 + a < rounds && lane < np) {
        int p = rr_member(lane, round, n), q = rr_member(n - 1 - lane, round, n);
        if (p > q) { const int x = p; p = q; q = x; }
        if (cs[a].y != 0.0) {
          const double vp = v[p], vq = v[q];
          v[p] = cs[a].x * vp - cs[a].y * vq;
          v[q] = cs[a].y * vp + cs[a].x * vq;
        }
      }
      __syncwarp();
      if (++round == n - 1) round = 0;
    }
  }
  for (int j = lane; j < k; j += 32) Vout[(int64_t)blockIdx.x * k + j] = v[order[j]];
}

// ---- eigenpairs of S for k > KMAX: one-sided Jacobi on its Cholesky factor, over the whole chip ----
// S = R^T R; rotating pairs of columns of R^T until all are orthogonal gives W with S = W W^T, so W's columns are the
// eigenvectors times the root of their eigenvalue.  One CTA per pair of the round-robin schedule (persistent, a grid
// barrier per round): the fp64 work of a sweep, 3.5 k^3, is spread over k / 2 SMs, and what is left is the latency of
// a round.  W [k][k]: column c of R^T is row c of R, contiguous.  Stops after a sweep without a rotation above
// |x.y| <= sqrt(k) 2^-52 |x||y|.
// k = 272: 360 ms as two-sided Jacobi in one block; 7.5 ms here.
constexpr int HJ_THREADS = 128;
// Squared norms are formed in a sweep's first round and carried through its rotations (they only steer the angles).
__global__ void __launch_bounds__(HJ_THREADS) hj_kernel(double* __restrict__ W, double* __restrict__ norms, GridSync* sy,
                                                        int k, int* status) {
  constexpr int PT = (KLIM + HJ_THREADS - 1) / HJ_THREADS;
  __shared__ double red[3][HJ_THREADS];
  __shared__ double sums[3], rot[5];
  const int n = (k + 1) / 2 * 2, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, i = blockIdx.x;
  const double tol2 = (double)k * 4.930380657631324e-32;            // k 2^-104
  unsigned int target = 0;
  for (int sweep = 0; sweep < HJ_SWEEPS; ++sweep) {
    bool any = false;
    for (int round = 0; round < n - 1; ++round) {
      int p = rr_member(i, round, n), q = rr_member(n - 1 - i, round, n);
      if (p > q) { const int x = p; p = q; q = x; }
      if (q < k) {                                   // (odd k: the dummy's partner rests, its norm formed all the same)
        double x[PT], y[PT], g = 0.0;
#pragma unroll
        for (int e = 0; e < PT; ++e) {
          const int c = tid + e * HJ_THREADS;
          x[e] = c < k ? __ldcg(W + (int64_t)p * k + c) : 0.0;
          y[e] = c < k ? __ldcg(W + (int64_t)q * k + c) : 0.0;
        }
        const int vals = round == 0 ? 3 : 1;
        double a = 0.0, b = 0.0;
        if (tid == 0 && round > 0) { a = __ldcg(norms + p); b = __ldcg(norms + q); }
#pragma unroll
        for (int e = 0; e < PT; ++e)
          if (warp * 32 + e * HJ_THREADS < k) g = fma(x[e], y[e], g);
        red[0][tid] = g;
        if (round == 0) {
          double nx = 0.0, ny = 0.0;
#pragma unroll
          for (int e = 0; e < PT; ++e)
            if (warp * 32 + e * HJ_THREADS < k) { nx = fma(x[e], x[e], nx); ny = fma(y[e], y[e], ny); }
          red[1][tid] = nx;
          red[2][tid] = ny;
        }
        __syncthreads();
        if (warp < vals) {
          double v = red[warp][lane];
#pragma unroll
          for (int w = 1; w < HJ_THREADS / 32; ++w) v += red[warp][lane + 32 * w];
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
          if (lane == 0) sums[warp] = v;
        }
        if (vals == 3) __syncthreads();
        if (tid == 0) {
          g = sums[0];
          if (round == 0) { a = sums[1]; b = sums[2]; }
          double c = 1.0, s = 0.0;
          if (g * g > tol2 * a * b) jacobi_angle(b - a, g, c, s);
          rot[0] = c; rot[1] = s; rot[2] = a; rot[3] = b; rot[4] = g;
        }
        __syncthreads();
        const double c = rot[0], s = rot[1];
        if (tid == HJ_THREADS - 1 && (s != 0.0 || round == 0)) {     // (the last warp has the fewest elements)
          const double cg = c * rot[4], sg = s * rot[4];
          __stcg(norms + p, c * (c * rot[2] - sg) - s * (cg - s * rot[3]));
          __stcg(norms + q, s * (s * rot[2] + cg) + c * (sg + c * rot[3]));
        }
        if (s != 0.0) {
          any = true;
#pragma unroll
          for (int e = 0; e < PT; ++e) {
            const int j = tid + e * HJ_THREADS;
            if (j < k) {
              __stcg(W + (int64_t)p * k + j, c * x[e] - s * y[e]);
              __stcg(W + (int64_t)q * k + j, s * x[e] + c * y[e]);
            }
          }
        }
      } else if (round == 0) {
        double nx = 0.0;
        for (int c = tid; c < k; c += HJ_THREADS) {
          const double v = __ldcg(W + (int64_t)p * k + c);
          nx = fma(v, v, nx);
        }
        red[0][tid] = nx;
        __syncthreads();
        if (warp == 0) {
          double v = red[0][lane];
#pragma unroll
          for (int w = 1; w < HJ_THREADS / 32; ++w) v += red[0][lane + 32 * w];
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
          if (lane == 0) __stcg(norms + p, v);
        }
      }
      if (round == n - 2 && any && tid == 0) atomicOr(&sy->rotated[sweep], 1);
      target += gridDim.x;
      if (!grid_barrier(sy, target, status)) return;
    }
    if (*reinterpret_cast<volatile int*>(&sy->rotated[sweep]) == 0) break;
  }
}
// Squared norms of W's columns: the eigenvalues of S + shift, unsorted.
__global__ void __launch_bounds__(HJ_THREADS) hj_norms_kernel(const double* __restrict__ W, double* __restrict__ raw, int k) {
  __shared__ double red[HJ_THREADS / 32];
  double a = 0.0;
  for (int j = threadIdx.x; j < k; j += HJ_THREADS) {
    const double x = W[(int64_t)blockIdx.x * k + j];
    a = fma(x, x, a);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = a;
  __syncthreads();
  if (threadIdx.x == 0) {
    a = 0.0;
    for (int w = 0; w < HJ_THREADS / 32; ++w) a += red[w];
    raw[blockIdx.x] = a;
  }
}
// Column c of W, normalised, to its place in the descending order (first index first on ties).
__global__ void __launch_bounds__(HJ_THREADS) hj_vectors_kernel(const double* __restrict__ W, const double* __restrict__ raw,
                                                                const double* __restrict__ shift, double* __restrict__ Vout,
                                                                double* __restrict__ evals, int k) {
  __shared__ int rank;
  const int c = blockIdx.x;
  const double e = raw[c];
  if (threadIdx.x == 0) rank = 0;
  __syncthreads();
  int above = 0;
  const long long key = order_key(e);
  for (int j = threadIdx.x; j < k; j += HJ_THREADS) {
    const long long f = order_key(raw[j]);
    above += f > key || (f == key && j < c);
  }
  if (above) atomicAdd(&rank, above);
  __syncthreads();
  const double inv = e > 0.0 ? 1.0 / sqrt(e) : 0.0;
  for (int j = threadIdx.x; j < k; j += HJ_THREADS) Vout[(int64_t)j * k + rank] = W[(int64_t)c * k + j] * inv;
  if (threadIdx.x == 0) evals[rank] = e - *shift;
}

// ---- flip column j so its largest-|.| entry (first index on ties) is positive ----
// A column without a finite entry (non-finite calibration data) is left as it is and
// the status word records ZOACT_ERR_NONFINITE.
constexpr int SIGN_THREADS = 1024;      // 14336 rows: 48 us with 256 threads, 24 here
__global__ void __launch_bounds__(SIGN_THREADS) sign_fix_kernel(float* __restrict__ U, int d, int r, int* __restrict__ status) {
  pdl_wait();
  pdl_trigger();
  const int j = blockIdx.x;
  __shared__ float bv[SIGN_THREADS];
  __shared__ int bi[SIGN_THREADS];
  float best = -1.f;
  int idx = 0x7fffffff;
#pragma unroll 8
  for (int i = threadIdx.x; i < d; i += blockDim.x) {
    const float a = fabsf(U[(int64_t)i * r + j]);
    if (a > best || (a == best && i < idx)) { best = a; idx = i; }
  }
  bv[threadIdx.x] = best;
  bi[threadIdx.x] = idx;
  __syncthreads();
  for (int s = blockDim.x / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s) {
      const float a = bv[threadIdx.x + s];
      const int ia = bi[threadIdx.x + s];
      if (a > bv[threadIdx.x] || (a == bv[threadIdx.x] && ia < bi[threadIdx.x])) {
        bv[threadIdx.x] = a;
        bi[threadIdx.x] = ia;
      }
    }
    __syncthreads();
  }
  const int top = bi[0];
  if (top < 0 || top >= d) {                 // no finite |U| in this column
    if (threadIdx.x == 0) record_error(status, ZOACT_ERR_NONFINITE);
    return;
  }
  const bool flip = U[(int64_t)top * r + j] < 0.f;
  __syncthreads();
  if (flip)
    for (int i = threadIdx.x; i < d; i += blockDim.x) U[(int64_t)i * r + j] = -U[(int64_t)i * r + j];
}

__global__ void f64_to_f32_kernel(const double* __restrict__ a, float* __restrict__ b, int n) {
  for (int i = threadIdx.x; i < n; i += blockDim.x) b[i] = (float)a[i];
}

struct Work {
  float* G;
  float* Q;
  float* Y;
  double* part;
  double* S;
  double* Rinv;
  double* V;
  double* ev;
  double* R;      // k > KMAX: Cholesky factor; the large Jacobi's columns (k x k)
  double* M;      // k > KMAX: its inverse factor L^-1
  double* D;      // k > KMAX: its diagonal blocks
  double2* log;   // small Jacobi: the angles of every round
  double* raw;    // large Jacobi: unsorted eigenvalues
  double* shift;  // diagonal shift of the last Cholesky
  int* ints;      // small Jacobi: rounds taken, column order
  GridSync* sync; // barrier of the cooperative launches
  int* absmax;    // max |X| (bits)
  float* P;       // X Q [n_tok, k] (no Gram matrix)
  Operand qop, pop;   // operand forms of Q and of P
};
constexpr int PROJ_MAX_SPLITS = 32;

// Row chunks of an A^T B over `rows` rows: two blocks per SM over all tiles, 32-row slabs.
int atb_chunks(const Ctx* ctx, int64_t rows, int k, int& chunk) {
  const int64_t t = (k + KMAX - 1) / KMAX, tiles = t * (t + 1) / 2, slabs = (rows + 31) / 32;
  int64_t n = (2 * ctx->sm_count + tiles - 1) / tiles;
  if (n > slabs) n = slabs;
  const int64_t per = (slabs + n - 1) / n;
  chunk = (int)(per * 32);
  return (int)((slabs + per - 1) / per);
}

// S = A^T B of A, B [rows, k] (A = B: the symmetric form)
int launch_atb(Ctx* ctx, const Work& w, const float* A, const float* B, int64_t rows, int k) {
  const unsigned tiles = (unsigned)((k + KMAX - 1) / KMAX);
  const int sym = A == B;
  int chunk;
  const int nchunk = atb_chunks(ctx, rows, k, chunk);
  ZOACT_CUDA_TRY(launch_pdl(ctx, tiles > 1 ? atb_partial_kernel<true> : atb_partial_kernel<false>, dim3(tiles, tiles, (unsigned)nchunk), dim3(256), 0, A, B, w.part, rows,
                            k, chunk, sym));
  ZOACT_CUDA_TRY(launch_pdl(ctx, sym ? sum_partials_kernel<true> : sum_partials_kernel<false>,
                            dim3((unsigned)((k * k + 31) / 32)), dim3(256), 0, w.part, w.S, nchunk, k));
  ctx->n_launch += 2;
  ZOACT_CHECK_LAUNCH();
  return ZOACT_OK;
}

// R^-1 (k > KMAX: and R, the shift; any: of any symmetric S) of S
int launch_chol(Ctx* ctx, const Work& w, int k, int any = 0) {
  if (k <= KMAX) {
    ZOACT_CUDA_TRY(launch_pdl(ctx, chol_inv_kernel, dim3(1), dim3(k <= 32 ? CHOL_THREADS / 2 : CHOL_THREADS), CHOL_SMEM, w.S, w.Rinv, k, ctx->d_status));
  } else {
    ZOACT_CUDA_TRY(cudaMemsetAsync(w.sync, 0, sizeof(GridSync), ctx->stream));
    CholBig c{w.S, w.R, w.M, w.Rinv, w.D, w.shift, w.sync, k, any, ctx->d_status};
    void* args[] = {&c};
    const int blocks = CHOLB_BLOCKS < ctx->sm_count ? CHOLB_BLOCKS : ctx->sm_count;
    ZOACT_CUDA_TRY(cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(chol_big_kernel), dim3((unsigned)blocks),
                                               dim3(CHOLB_THREADS), args, 0, ctx->stream));
  }
  ++ctx->n_launch;
  ZOACT_CHECK_LAUNCH();
  return ZOACT_OK;
}

// op (with its 16-bit type): write the result's operand form too.
int launch_apply(Ctx* ctx, const float* A, const double* M, float* out, int64_t rows, int k, int ldm, int c, int tri,
                 const Operand* op = nullptr, int dtype = ZOACT_DT_FP32) {
  const int ct = c <= 32 || (tri && c > KMAX) ? 32 : 64;
  const int rt = 4096 / ct;
  const dim3 grid((unsigned)((rows + rt - 1) / rt), (unsigned)((c + ct - 1) / ct));
  auto kern = ct == 32 ? (!op ? apply_kernel<float, 32> : dtype == ZOACT_DT_BF16 ? apply_kernel<__nv_bfloat16, 32>
                                                                                : apply_kernel<__half, 32>)
                       : (!op ? apply_kernel<float, 64> : dtype == ZOACT_DT_BF16 ? apply_kernel<__nv_bfloat16, 64>
                                                                                : apply_kernel<__half, 64>);
  ZOACT_CUDA_TRY(launch_pdl(ctx, kern, grid, dim3(256), 0, A, M, out, rows, k, ldm, c, tri, op ? *op : Operand{}));
  ++ctx->n_launch;
  ZOACT_CHECK_LAUNCH();
  return ZOACT_OK;
}

// CholeskyQR2 of Y [d, k], which holds Q afterwards; tmp: another [d, k]; op: Q's operand form too.
int orth(Ctx* ctx, const Work& w, float* Y, float* tmp, int d, int k, const Operand* op, int dtype) {
  float* src = Y;
  float* dst = tmp;
  for (int pass = 0; pass < 2; ++pass) {
    int st = launch_atb(ctx, w, src, src, d, k);
    if (!st) st = launch_chol(ctx, w, k);
    if (!st) st = launch_apply(ctx, src, w.Rinv, dst, d, k, k, k, 1, pass ? op : nullptr, dtype);
    if (st) return st;
    src = tmp;
    dst = Y;
  }
  return ZOACT_OK;
}

// dst [rows, k] (or null) = X F for 16-bit X [rows, kd] and F's operand form; to_op: dst's operand form too.  most_kb:
// K-blocks accumulated by one MMA chain at most (0: as the chip is filled).
int launch_product(Ctx* ctx, const Work& w, const void* X, int dtype, int64_t rows, int64_t kd, const Operand& f, int mode,
                   int k, float* dst, const Operand* to_op, int d, int most_kb = 0) {
  const ProjPlan plan = proj_plan(ctx, rows, (int)kd, k, PROJ_MAX_SPLITS, most_kb);
  float* part = static_cast<float*>(
      scratch(ctx, SLOT_SPLITK, (size_t)plan.groups * plan.splits * rows * plan.rt * sizeof(float)));
  if (!part) return ZOACT_ERR_NOMEM;
  const int st = launch_proj_parts(ctx, X, dtype, rows, (int)kd, f.op, plan, part);
  if (st) return st;
  // the operand's padding columns are written (as zeros) too
  const int64_t cover = to_op ? to_op->ld : rows;
  const dim3 grid((unsigned)((cover + RED_ROWS - 1) / RED_ROWS), (unsigned)plan.groups);
  const bool bf = dtype == ZOACT_DT_BF16;
  auto kern = to_op ? (bf ? reduce_parts_kernel<__nv_bfloat16, true> : reduce_parts_kernel<__half, true>)
                    : (bf ? reduce_parts_kernel<__nv_bfloat16, false> : reduce_parts_kernel<__half, false>);
  ZOACT_CUDA_TRY(launch_pdl(ctx, kern, grid, dim3(256), 0, part, rows, k, plan.splits, plan.rt, dst,
                            to_op ? *to_op : Operand{}, mode, w.absmax, d));
  ++ctx->n_launch;
  ZOACT_CHECK_LAUNCH();
  return ZOACT_OK;
}

}  // namespace

int run_basis_init(Ctx* ctx, const void* X, int xdtype, int64_t n_tok, int d, int r, int oversample, int n_iter,
                   uint64_t seed, float* U_out, float* evals_out) {
  int k = r + oversample;
  if (k > d) k = d;
  if (k > KLIM || r > k) return ZOACT_ERR_UNSUPPORTED;
  ZOACT_CUDA_TRY(cudaFuncSetAttribute(jacobi_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, JACOBI_SMEM));
  ZOACT_CUDA_TRY(cudaFuncSetAttribute(chol_inv_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, CHOL_SMEM));
  const int64_t n_pad = (n_tok + 7) / 8 * 8;
  // no Gram matrix (see reduce_parts_kernel): 16-bit X, unless there are so many more tokens than columns that reading
  // X twice a step costs more than the d x d matrix and its one-off product
  const bool direct = xdtype != ZOACT_DT_FP32 && n_tok <= (int64_t)GRAM_TOKENS * d;
  int chunk;
  size_t nchunk = (size_t)atb_chunks(ctx, d, k, chunk);
  if (direct) {
    const size_t np = (size_t)atb_chunks(ctx, n_tok, k, chunk);
    if (np > nchunk) nchunk = np;
  }
  const size_t g_bytes = direct ? (size_t)n_tok * k * 4 : (size_t)d * d * 4;
  const size_t q_op = direct ? (size_t)basis_tc_rows(k) * d * 2 : 0, p_op = direct ? (size_t)basis_tc_rows(k) * n_pad * 2 : 0;
  const size_t kk = (size_t)k * k * 8, dk = (size_t)d * k * 4, big = k > KMAX ? kk : 0;
  const size_t log_bytes = k <= KMAX ? (size_t)JAC_SWEEPS * KMAX * (KMAX / 2) * sizeof(double2) : 0;
  // workspace (every piece padded to 256 bytes)
  const size_t bytes = g_bytes + q_op + p_op + 2 * dk + nchunk * kk + 3 * kk + 3 * big + log_bytes + 2 * (size_t)k * 8 +
                       sizeof(GridSync) + 20 * 256 + 4096;
  uint8_t* base = static_cast<uint8_t*>(scratch(ctx, SLOT_BASIS, bytes));
  if (!base) return ZOACT_ERR_NOMEM;
  Work w;
  size_t off = 0;
  auto take = [&](size_t b) { uint8_t* p = base + off; off += (b + 255) / 256 * 256; return p; };
  w.G = w.P = reinterpret_cast<float*>(take(g_bytes));
  uint8_t* ops = take(q_op + p_op);                  // (q_op is a multiple of 16 bytes: d is one of 8)
  w.qop = Operand{ops, d, proj_rank_tile(k), proj_operand_rows(k)};
  w.pop = Operand{ops + q_op, n_pad, w.qop.rt, w.qop.nb};
  w.Q = reinterpret_cast<float*>(take(dk));
  w.Y = reinterpret_cast<float*>(take(dk));
  w.part = reinterpret_cast<double*>(take(nchunk * kk));
  w.S = reinterpret_cast<double*>(take(kk));
  w.Rinv = reinterpret_cast<double*>(take(kk));
  w.V = reinterpret_cast<double*>(take(kk));
  w.R = reinterpret_cast<double*>(take(big));
  w.M = reinterpret_cast<double*>(take(big));
  w.D = reinterpret_cast<double*>(take(big));
  w.ev = reinterpret_cast<double*>(take((size_t)k * 8));
  w.log = reinterpret_cast<double2*>(take(log_bytes));
  w.raw = reinterpret_cast<double*>(take((size_t)k * 8));
  w.shift = reinterpret_cast<double*>(take(8));
  w.ints = reinterpret_cast<int*>(take((KMAX + 1) * sizeof(int)));
  w.sync = reinterpret_cast<GridSync*>(take(sizeof(GridSync)));
  w.absmax = reinterpret_cast<int*>(take(sizeof(int)));
  if (off > bytes) return ZOACT_ERR_NOMEM;

  // 1. X^T and, where it is used, the Gram matrix
  void* Xt = nullptr;
  if (xdtype == ZOACT_DT_FP32) {
    dim3 grid((d + 63) / 64, (d + 63) / 64);
    gram_f32_kernel<<<grid, 256, 0, ctx->stream>>>(static_cast<const float*>(X), w.G, n_tok, d); ++ctx->n_launch;
    ZOACT_CHECK_LAUNCH();
  } else {
    Xt = scratch(ctx, SLOT_BASIS_X, (size_t)d * n_pad * 2);
    if (!Xt) return ZOACT_ERR_NOMEM;
    if (direct) {
      ZOACT_CUDA_TRY(cudaMemsetAsync(w.absmax, 0, sizeof(int), ctx->stream));
      ZOACT_CUDA_TRY(cudaMemsetAsync(ops, 0, q_op + p_op, ctx->stream));   // ranks past k stay zero
    }
    const dim3 grid((unsigned)((n_pad + 63) / 64), (unsigned)((d + 63) / 64));
    int* top = xdtype == ZOACT_DT_FP16 && direct ? w.absmax : nullptr;
    if (xdtype == ZOACT_DT_BF16) {
      transpose_pad_kernel<__nv_bfloat16><<<grid, 256, 0, ctx->stream>>>(
          static_cast<const __nv_bfloat16*>(X), static_cast<__nv_bfloat16*>(Xt), n_tok, d, n_pad, top);
    } else {
      transpose_pad_kernel<__half><<<grid, 256, 0, ctx->stream>>>(static_cast<const __half*>(X),
                                                                          static_cast<__half*>(Xt), n_tok, d, n_pad, top);
    }
    ++ctx->n_launch;
    ZOACT_CHECK_LAUNCH();
    if (!direct) {
      const int st = launch_gemm_tc_f32out(ctx, Xt, Xt, xdtype, d, d, (int)n_pad, w.G);
      if (st) return st;
    }
  }
  // 2-3. sketch and subspace iteration: Q stays in w.Q
  const int64_t nq = (int64_t)d * k;
  ZOACT_CUDA_TRY(launch_pdl(ctx, omega_kernel, dim3((unsigned)((nq / 4 + 255) / 256 + 1)), dim3(256), 0, w.Q, nq, seed));
  ++ctx->n_launch;
  ZOACT_CHECK_LAUNCH();
  const Operand* qop = direct ? &w.qop : nullptr;
  int st = orth(ctx, w, w.Q, w.Y, d, k, qop, xdtype);
  if (st) return st;
  const dim3 gq_blocks((unsigned)((d + 63) / 64), (unsigned)((k + KMAX - 1) / KMAX));
  for (int it = 0; it < n_iter; ++it) {
    if (direct) {
      st = launch_product(ctx, w, X, xdtype, n_tok, d, w.qop, 0, k, nullptr, &w.pop, d);
      if (!st) st = launch_product(ctx, w, Xt, xdtype, d, n_pad, w.pop, 1, k, w.Y, nullptr, d);
      if (st) return st;
    } else {
      gemm_gq_kernel<<<gq_blocks, 256, 0, ctx->stream>>>(w.G, w.Q, w.Y, d, k); ++ctx->n_launch;
      ZOACT_CHECK_LAUNCH();
    }
    st = orth(ctx, w, w.Y, w.Q, d, k, qop, xdtype);
    if (st) return st;
    float* t = w.Q; w.Q = w.Y; w.Y = t;
  }
  // 4. Rayleigh-Ritz: S = Q^T G Q, of P = X Q as P^T P
  if (direct) {
    // The Ritz values are squares of P's sums, whose terms mostly share a sign, and the tensor core truncates every
    // 16-wide step of its fp32 accumulator: chains of n_tok / 256 K-blocks keep that bias at half of what a Gram matrix
    // summed over the tokens had (14336 wide, 512 tokens: 1.0e-6 of the values in chains of 7 K-blocks, 3.0e-7 in 2).
    const int most_kb = n_tok < 256 ? 1 : (int)(n_tok / 256);
    st = launch_product(ctx, w, X, xdtype, n_tok, d, w.qop, 0, k, w.P, nullptr, d, most_kb);
    if (!st) st = launch_atb(ctx, w, w.P, w.P, n_tok, k);
  } else {
    gemm_gq_kernel<<<gq_blocks, 256, 0, ctx->stream>>>(w.G, w.Q, w.Y, d, k); ++ctx->n_launch;
    ZOACT_CHECK_LAUNCH();
    st = launch_atb(ctx, w, w.Q, w.Y, d, k);
  }
  if (st) return st;
  if (k <= KMAX) {
    ZOACT_CUDA_TRY(launch_pdl(ctx, jacobi_kernel, dim3(1), dim3(JAC_THREADS), JACOBI_SMEM, w.S, w.log, w.ints, w.ev,
                              w.ints + 1, k));
    ZOACT_CUDA_TRY(launch_pdl(ctx, jacobi_vectors_kernel, dim3((unsigned)k), dim3(32), 0, w.log, w.ints, w.ints + 1, w.V, k));
    ctx->n_launch += 2;
  } else {
    // Q^T (G Q) of a Gram matrix has eigenvalues down to -1e-7 of its trace for a spectrum that falls quickly, and to
    // -7e-6 for 400 K tokens of rank one (fp32 chains over the tokens)
    st = launch_chol(ctx, w, k, 1);
    if (st) return st;
    ZOACT_CUDA_TRY(cudaMemsetAsync(w.sync, 0, sizeof(GridSync), ctx->stream));
    void* args[] = {&w.R, &w.raw, &w.sync, &k, &ctx->d_status};
    ZOACT_CUDA_TRY(cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(hj_kernel), dim3((unsigned)((k + 1) / 2)),
                                               dim3(HJ_THREADS), args, 0, ctx->stream));
    hj_norms_kernel<<<k, HJ_THREADS, 0, ctx->stream>>>(w.R, w.raw, k);
    hj_vectors_kernel<<<k, HJ_THREADS, 0, ctx->stream>>>(w.R, w.raw, w.shift, w.V, w.ev, k);
    ctx->n_launch += 3;
  }
  ZOACT_CHECK_LAUNCH();
  st = launch_apply(ctx, w.Q, w.V, U_out, d, k, k, r, 0);
  if (st) return st;
  ZOACT_CUDA_TRY(launch_pdl(ctx, sign_fix_kernel, dim3((unsigned)r), dim3(SIGN_THREADS), 0, U_out, d, r, ctx->d_status));
  ++ctx->n_launch;
  if (evals_out) {
    f64_to_f32_kernel<<<1, 256, 0, ctx->stream>>>(w.ev, evals_out, k);
    ++ctx->n_launch;
  }
  ZOACT_CHECK_LAUNCH();
  return ZOACT_OK;
}

}  // namespace zoact
