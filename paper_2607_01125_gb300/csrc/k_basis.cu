// One-shot activation basis (Algorithm 1: top-r right singular vectors of the
// calibration activations X, i.e. the top-r eigenvectors of G = X^T X).
//
// Device pipeline (no host round trip, every step a kernel):
//   1. G = X^T X in fp32: for 16-bit X, X is transposed into a zero-padded
//      [d, n_pad] copy and multiplied with itself on the tcgen05 GEMM;
//      for fp32 X a CUDA-core kernel forms X^T X directly.
//   2. Omega [d, k] from the Z generator (seed, layer 0, query 0), k = r + oversample.
//   3. Q = orth(Omega); n_iter times Q = orth(G Q).  orth() is CholeskyQR2:
//      S = Y^T Y (64 x 64 output tiles; fp32 over 32-row slabs, fp64 across
//      slabs and row chunks), Cholesky S = R^T R and R^-1 in one block (fp64,
//      in global memory), Q = Y R^-1; done twice for orthogonality.
//   4. Rayleigh-Ritz: S = Q^T G Q (fp64), Jacobi (fp64): two-sided in one block's
//      shared memory for k <= 64, one-sided on the Cholesky factor over the whole
//      chip above; eigenpairs sorted by value, U = Q V[:, :r], each column flipped so
//      its largest-magnitude entry is positive (first index on ties).
//   k = r + oversample <= 512.
#include "internal.h"
#include "philox.cuh"

namespace zoact {
namespace {

constexpr int KMAX = 64;        // k handled by the shared-memory Jacobi and R^-1 application
constexpr int KLIM = 512;       // largest k

// ---- X [n, d] (16-bit) -> Xt [d, n_pad], zero in columns n .. n_pad-1 ----
template <typename T>
__global__ void transpose_pad_kernel(const T* __restrict__ X, T* __restrict__ Xt, int64_t n, int d, int64_t n_pad) {
  __shared__ T tile[32][33];
  const int64_t t0 = (int64_t)blockIdx.x * 32;
  const int i0 = blockIdx.y * 32;
  for (int y = threadIdx.y; y < 32; y += 8) {
    const int64_t t = t0 + y;
    const int i = i0 + threadIdx.x;
    tile[y][threadIdx.x] = (t < n && i < d) ? X[t * d + i] : from_f32<T>(0.f);
  }
  __syncthreads();
  for (int y = threadIdx.y; y < 32; y += 8) {
    const int i = i0 + y;
    const int64_t t = t0 + threadIdx.x;
    if (i < d && t < n_pad) Xt[(int64_t)i * n_pad + t] = tile[threadIdx.x][y];
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

// ---- partial S = A^T B over a chunk of rows, A, B [d, k]: 64 x 64 output tiles per block (grid x, y),
// row chunks on grid z; fp32 products over 32-row slabs, added into fp64 per slab ----
constexpr int ATB_CHUNK = 2048;
__global__ void __launch_bounds__(256) atb_partial_kernel(const float* __restrict__ A, const float* __restrict__ B,
                                                          double* __restrict__ part, int d, int k) {
  __shared__ float As[32][KMAX + 4];
  __shared__ float Bs[32][KMAX + 4];
  const int p0 = blockIdx.y * KMAX, q0 = blockIdx.x * KMAX;
  const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
  const int64_t r_begin = (int64_t)blockIdx.z * ATB_CHUNK;
  const int64_t r_end = r_begin + ATB_CHUNK < d ? r_begin + ATB_CHUNK : d;
  double acc[4][4] = {};
  for (int64_t s0 = r_begin; s0 < r_end; s0 += 32) {
    __syncthreads();
    for (int v = threadIdx.x; v < 32 * KMAX; v += 256) {
      const int rr = v / KMAX, c = v % KMAX;
      const int64_t row = s0 + rr;
      As[rr][c] = (row < r_end && p0 + c < k) ? A[row * k + p0 + c] : 0.f;
      Bs[rr][c] = (row < r_end && q0 + c < k) ? B[row * k + q0 + c] : 0.f;
    }
    __syncthreads();
    float a32[4][4] = {};
#pragma unroll 8
    for (int rr = 0; rr < 32; ++rr) {
      float a[4], b[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) { a[i] = As[rr][ty * 4 + i]; b[i] = Bs[rr][tx * 4 + i]; }
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) a32[i][j] = fmaf(a[i], b[j], a32[i][j]);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[i][j] += (double)a32[i][j];
  }
  double* out = part + (int64_t)blockIdx.z * k * k;
  for (int i = 0; i < 4; ++i)
    for (int j = 0; j < 4; ++j) {
      const int p = p0 + ty * 4 + i, q = q0 + tx * 4 + j;
      if (p < k && q < k) out[(int64_t)p * k + q] = acc[i][j];
    }
}

__global__ void sum_partials_kernel(const double* __restrict__ part, double* __restrict__ S, int nblk, int kk) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < kk; i += gridDim.x * blockDim.x) {
    double s = 0.0;
    for (int b = 0; b < nblk; ++b) s += part[(int64_t)b * kk + i];
    S[i] = s;
  }
}

// ---- Cholesky S = R^T R (R upper) and Rinv, one block, R in global memory (k x k fp64); shift on breakdown ----
__global__ void __launch_bounds__(256) chol_inv_kernel(const double* __restrict__ S, double* __restrict__ R,
                                                       double* __restrict__ Rinv, double* __restrict__ shift_out,
                                                       int k, int* status) {
  __shared__ int bad;
  __shared__ double shift, rjj_s;
  __shared__ double red[256];
  const int t = threadIdx.x;
  if (t == 0) { shift = 0.0; bad = 0; }
  __syncthreads();
  for (int attempt = 0; attempt < 4; ++attempt) {
    for (int v = t; v < k * k; v += blockDim.x) {
      const int i = v / k, j = v % k;
      R[v] = (j >= i) ? S[v] + (i == j ? shift : 0.0) : 0.0;
    }
    if (t == 0) bad = 0;
    __syncthreads();
    for (int j = 0; j < k; ++j) {
      // r_jj = sqrt(R[j][j] - sum_{p<j} R[p][j]^2)
      double part = 0.0;
      for (int p = t; p < j; p += blockDim.x) part += R[(int64_t)p * k + j] * R[(int64_t)p * k + j];
      red[t] = part;
      __syncthreads();
      for (int h = blockDim.x / 2; h > 0; h >>= 1) {
        if (t < h) red[t] += red[t + h];
        __syncthreads();
      }
      if (t == 0) {
        const double djj = R[(int64_t)j * k + j] - red[0];
        if (!(djj > 0.0)) {
          bad = 1;
        } else {
          rjj_s = sqrt(djj);
          R[(int64_t)j * k + j] = rjj_s;
        }
      }
      __syncthreads();
      if (bad) break;
      // R[j][q] = (R[j][q] - sum_{p<j} R[p][j] R[p][q]) / r_jj for q > j
      for (int q = j + 1 + t; q < k; q += blockDim.x) {
        double s2 = R[(int64_t)j * k + q];
        for (int p = 0; p < j; ++p) s2 -= R[(int64_t)p * k + j] * R[(int64_t)p * k + q];
        R[(int64_t)j * k + q] = s2 / rjj_s;
      }
      __syncthreads();
    }
    if (!bad) break;
    if (t == 0) {
      double tr = 0.0;
      for (int i = 0; i < k; ++i) tr += S[(int64_t)i * k + i];
      shift = (shift == 0.0) ? 1e-12 * tr : shift * 1e3;
    }
    __syncthreads();
  }
  if (bad) {
    if (t == 0) record_error(status, ZOACT_ERR_NONFINITE);
    return;
  }
  if (t == 0) *shift_out = shift;
  // Rinv: solve R * Ri = I column by column (column c per thread)
  for (int c = t; c < k; c += blockDim.x) {
    for (int i = k - 1; i >= 0; --i) {
      double s2 = (i == c) ? 1.0 : 0.0;
      for (int p = i + 1; p <= c; ++p) s2 -= R[(int64_t)i * k + p] * Rinv[(int64_t)p * k + c];
      Rinv[(int64_t)i * k + c] = i > c ? 0.0 : s2 / R[(int64_t)i * k + i];
    }
  }
}

// ---- Q [d, k] = Y [d, k] * Rinv [k, k] (fp64 accumulate, fp32 out); Q may alias Y ----
// One warp per row: every lane reads the row before any lane writes it.
// R^-1 is read from shared memory for k <= KMAX, else from global memory (L2).
__global__ void apply_rinv_kernel(const float* Y, const double* __restrict__ Rinv, float* Q, int d, int k) {
  __shared__ double Rs[KMAX * KMAX];
  const bool in_smem = k <= KMAX;
  if (in_smem)
    for (int v = threadIdx.y * blockDim.x + threadIdx.x; v < k * k; v += blockDim.x * blockDim.y) Rs[v] = Rinv[v];
  __syncthreads();
  const double* Rm = in_smem ? Rs : Rinv;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.y + threadIdx.y; i < d; i += (int64_t)gridDim.x * blockDim.y) {
    float out[KLIM / 32];
#pragma unroll
    for (int h = 0; h < KLIM / 32; ++h) {
      const int c = threadIdx.x + 32 * h;
      double s = 0.0;
      if (c < k)
        for (int p = 0; p <= c; ++p) s += (double)Y[i * k + p] * Rm[(int64_t)p * k + c];
      out[h] = (float)s;
    }
    __syncwarp();
#pragma unroll
    for (int h = 0; h < KLIM / 32; ++h) {
      const int c = threadIdx.x + 32 * h;
      if (c < k) Q[i * k + c] = out[h];
    }
    __syncwarp();
  }
}

// ---- eigenpairs of S (k x k, fp64), k <= KMAX: two-sided Jacobi in one block ----
// Each round of the round-robin schedule (n = k rounded up to even, n - 1 rounds a sweep) rotates n / 2 disjoint
// pairs: one warp forms the angles, then every thread updates the 2 x 2 blocks J_i^T A J_j of the symmetric matrix in
// shared memory, half of them (i <= j).  Bound by the fp64 pipe (2 lanes a cycle and SM), so the eigenvectors are left
// out: the angles are logged and jacobi_vectors_kernel applies them to every row of V on its own SM.  The matrix is
// padded to n with a zero row, whose rotations are trivial.  Stops when off(A)^2 <= 1e-30 |A|_F^2.
// k = 48: 17.2 ms as rotations taken one by one with the vectors beside them; 0.92 ms here (its vectors 0.07).
constexpr int JAC_THREADS = 512;
constexpr int JAC_SWEEPS = 60;
constexpr int JACOBI_SMEM = KMAX * (KMAX + 1) * 8;
__device__ __forceinline__ int rr_member(int slot, int round, int n) {
  // slot 0 stays; slots 1 .. n-1 rotate by `round`
  int m = slot - 1 + round;
  if (m >= n - 1) m -= n - 1;
  return slot == 0 ? 0 : 1 + m;
}
// The rotation that zeroes apq: t = s / c is the smaller root, so |angle| <= pi / 4.
__device__ __forceinline__ void jacobi_angle(double app, double aqq, double apq, double& c, double& s, double& t) {
  c = 1.0; s = 0.0; t = 0.0;
  if (fabs(apq) > 1e-300) {
    const double theta = (aqq - app) / (2.0 * apq);
    if (fabs(theta) > 1e150) t = 0.5 / theta;
    else t = (theta >= 0 ? 1.0 : -1.0) / (fabs(theta) + sqrt(theta * theta + 1.0));
    c = 1.0 / sqrt(1.0 + t * t);
    s = t * c;
  }
}
__global__ void __launch_bounds__(JAC_THREADS) jacobi_kernel(const double* __restrict__ S, double2* __restrict__ log,
                                                             int* __restrict__ n_rounds, double* __restrict__ evals,
                                                             int* __restrict__ order, int k) {
  extern __shared__ double A[];                      // [n][n + 1]
  __shared__ double cs_c[KMAX / 2], cs_s[KMAX / 2], cs_t[KMAX / 2];
  __shared__ int pp[KMAX / 2], qq[KMAX / 2];
  __shared__ double red[2][JAC_THREADS / 32];
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
    for (int round = 0; round < n - 1; ++round, ++rounds) {
      if (tid < 32 && tid < np) {
        int p = rr_member(tid, round, n), q = rr_member(n - 1 - tid, round, n);
        if (p > q) { const int x = p; p = q; q = x; }
        double c, s, t;
        jacobi_angle(A[p * ld + p], A[q * ld + q], A[p * ld + q], c, s, t);
        pp[tid] = p; qq[tid] = q; cs_c[tid] = c; cs_s[tid] = s; cs_t[tid] = t;
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
        if (i == j) {
          const double d = cs_t[i] * A[pi * ld + qi];
          if (d != 0.0) {
            A[pi * ld + pi] -= d;
            A[qi * ld + qi] += d;
            A[pi * ld + qi] = A[qi * ld + pi] = 0.0;
          }
          continue;
        }
        const double ci = cs_c[i], si = cs_s[i], cj = cs_c[j], sj = cs_s[j];
        const double a = A[pi * ld + pj], bq = A[pi * ld + qj], cq = A[qi * ld + pj], dq = A[qi * ld + qj];
        const double a1 = cj * a - sj * bq, b1 = sj * a + cj * bq, c1 = cj * cq - sj * dq, d1 = sj * cq + cj * dq;
        const double a2 = ci * a1 - si * c1, c2 = si * a1 + ci * c1, b2 = ci * b1 - si * d1, d2 = si * b1 + ci * d1;
        A[pi * ld + pj] = A[pj * ld + pi] = a2;
        A[pi * ld + qj] = A[qj * ld + pi] = b2;
        A[qi * ld + pj] = A[pj * ld + qi] = c2;
        A[qi * ld + qj] = A[qj * ld + qi] = d2;
      }
      __syncthreads();
    }
  }
  if (tid == 0) *n_rounds = rounds;
  for (int i = tid; i < k; i += JAC_THREADS) {       // descending; first index first on ties
    const double e = A[i * ld + i];
    int rank = 0;
    for (int j = 0; j < k; ++j) {
      const double f = A[j * ld + j];
      if (f > e || (f == e && j < i)) ++rank;
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
        const double vp = v[p], vq = v[q];
        v[p] = cs[a].x * vp - cs[a].y * vq;
        v[q] = cs[a].y * vp + cs[a].x * vq;
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
// |x.y| <= sqrt(k) 2^-52 |x||y|.  Every spin is bounded (2 s): a barrier that gives up records ZOACT_ERR_TIMEOUT and
// releases the others through the abort word.
// k = 272: 360 ms as two-sided Jacobi in one block; ~10 ms here.
constexpr int HJ_THREADS = 128;
constexpr int HJ_SWEEPS = 40;
struct HjSync {
  unsigned int count;             // arrivals since the launch
  int abort;
  int rotated[HJ_SWEEPS];
};
__device__ __forceinline__ bool hj_barrier(HjSync* sy, unsigned int target, int* status) {
  __shared__ int give_up;
  __syncthreads();
  if (threadIdx.x == 0) {
    give_up = 0;
    __threadfence();
    atomicAdd(&sy->count, 1u);
    uint64_t t0 = 0;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
    while (*reinterpret_cast<volatile unsigned int*>(&sy->count) < target) {
      if (*reinterpret_cast<volatile int*>(&sy->abort)) { give_up = 1; break; }
      uint64_t now;
      asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(now));
      if (now - t0 > 2000000000ull) {
        atomicExch(&sy->abort, 1);
        record_error(status, ZOACT_ERR_TIMEOUT);
        give_up = 1;
        break;
      }
    }
    __threadfence();
  }
  __syncthreads();
  return give_up == 0;
}
__global__ void __launch_bounds__(HJ_THREADS) hj_kernel(double* __restrict__ W, HjSync* sy, int k, int* status) {
  constexpr int PT = (KLIM + HJ_THREADS - 1) / HJ_THREADS;
  __shared__ double red[3][HJ_THREADS / 32];
  __shared__ double rot[2];
  const int n = (k + 1) / 2 * 2, tid = threadIdx.x, i = blockIdx.x;
  const double tol = sqrt((double)k) * 2.220446049250313e-16;
  unsigned int target = 0;
  for (int sweep = 0; sweep < HJ_SWEEPS; ++sweep) {
    bool any = false;
    for (int round = 0; round < n - 1; ++round) {
      int p = rr_member(i, round, n), q = rr_member(n - 1 - i, round, n);
      if (p > q) { const int x = p; p = q; q = x; }
      if (q < k) {                                   // (odd k: the dummy's partner rests)
        double x[PT], y[PT], a = 0.0, b = 0.0, g = 0.0;
#pragma unroll
        for (int e = 0; e < PT; ++e) {
          const int c = tid + e * HJ_THREADS;
          x[e] = c < k ? __ldcg(W + (int64_t)p * k + c) : 0.0;
          y[e] = c < k ? __ldcg(W + (int64_t)q * k + c) : 0.0;
        }
#pragma unroll
        for (int e = 0; e < PT; ++e) {
          if (e * HJ_THREADS < k) {
            a = fma(x[e], x[e], a);
            b = fma(y[e], y[e], b);
            g = fma(x[e], y[e], g);
          }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          a += __shfl_xor_sync(0xffffffffu, a, o);
          b += __shfl_xor_sync(0xffffffffu, b, o);
          g += __shfl_xor_sync(0xffffffffu, g, o);
        }
        if ((tid & 31) == 0) { red[0][tid >> 5] = a; red[1][tid >> 5] = b; red[2][tid >> 5] = g; }
        __syncthreads();
        if (tid == 0) {
          a = b = g = 0.0;
          for (int w = 0; w < HJ_THREADS / 32; ++w) { a += red[0][w]; b += red[1][w]; g += red[2][w]; }
          double c = 1.0, s = 0.0, t = 0.0;
          if (g * g > tol * tol * a * b) jacobi_angle(a, b, g, c, s, t);
          rot[0] = c; rot[1] = s;
        }
        __syncthreads();
        const double c = rot[0], s = rot[1];
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
      }
      if (round == n - 2 && any && tid == 0) atomicOr(&sy->rotated[sweep], 1);
      target += gridDim.x;
      if (!hj_barrier(sy, target, status)) return;
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
  for (int j = threadIdx.x; j < k; j += HJ_THREADS) above += raw[j] > e || (raw[j] == e && j < c);
  if (above) atomicAdd(&rank, above);
  __syncthreads();
  const double inv = e > 0.0 ? 1.0 / sqrt(e) : 0.0;
  for (int j = threadIdx.x; j < k; j += HJ_THREADS) Vout[(int64_t)j * k + rank] = W[(int64_t)c * k + j] * inv;
  if (threadIdx.x == 0) evals[rank] = e - *shift;
}

// ---- U [d, r] = Q [d, k] * V[:, :r] ----
__global__ void ritz_kernel(const float* __restrict__ Q, const double* __restrict__ V, float* __restrict__ U, int d,
                            int k, int r) {
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < (int64_t)d * r;
       v += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = v / r;
    const int j = (int)(v % r);
    double s = 0.0;
    for (int p = 0; p < k; ++p) s += (double)Q[i * k + p] * V[p * k + j];
    U[v] = (float)s;
  }
}

// ---- flip column j so its largest-|.| entry (first index on ties) is positive ----
// A column without a finite entry (non-finite calibration data) is left as it is and
// the status word records ZOACT_ERR_NONFINITE.
__global__ void sign_fix_kernel(float* __restrict__ U, int d, int r, int* __restrict__ status) {
  const int j = blockIdx.x;
  __shared__ float bv[256];
  __shared__ int bi[256];
  float best = -1.f;
  int idx = 0x7fffffff;
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
  double* R;      // Cholesky factor; the large Jacobi's columns (k x k)
  double2* log;   // small Jacobi: the angles of every round
  double* raw;    // large Jacobi: unsorted eigenvalues
  double* shift;  // diagonal shift of the last Cholesky
  int* ints;      // small Jacobi: rounds taken, column order
  HjSync* sync;   // large Jacobi's barrier
  int nchunk;     // row chunks of the A^T B partials
};

void launch_atb(Ctx* ctx, const Work& w, const float* A, const float* B, int d, int k) {
  const unsigned tiles = (unsigned)((k + KMAX - 1) / KMAX);
  atb_partial_kernel<<<dim3(tiles, tiles, (unsigned)w.nchunk), 256, 0, ctx->stream>>>(A, B, w.part, d, k);
  ++ctx->n_launch;
  sum_partials_kernel<<<(k * k + 255) / 256, 256, 0, ctx->stream>>>(w.part, w.S, w.nchunk, k * k);
  ++ctx->n_launch;
}

int orth(Ctx* ctx, Work& w, float* Y, float* Q, int d, int k) {
  // CholeskyQR2: Q = Y R^-1 twice
  const float* src = Y;
  for (int pass = 0; pass < 2; ++pass) {
    launch_atb(ctx, w, src, src, d, k);
    chol_inv_kernel<<<1, 256, 0, ctx->stream>>>(w.S, w.R, w.Rinv, w.shift, k, ctx->d_status); ++ctx->n_launch;
    apply_rinv_kernel<<<(d + 7) / 8 < 4096 ? (d + 7) / 8 : 4096, dim3(32, 8), 0, ctx->stream>>>(src, w.Rinv, Q, d, k); ++ctx->n_launch;
    ZOACT_CHECK_LAUNCH();
    src = Q;
  }
  return ZOACT_OK;
}

}  // namespace

int run_basis_init(Ctx* ctx, const void* X, int xdtype, int64_t n_tok, int d, int r, int oversample, int n_iter,
                   uint64_t seed, float* U_out, float* evals_out) {
  int k = r + oversample;
  if (k > d) k = d;
  if (k > KLIM || r > k) return ZOACT_ERR_UNSUPPORTED;
  ZOACT_CUDA_TRY(cudaFuncSetAttribute(jacobi_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, JACOBI_SMEM));
  const int nchunk = (d + ATB_CHUNK - 1) / ATB_CHUNK;
  // workspace: G d*d f32 | Q, Y d*k f32 | part nchunk*k*k f64 | S, Rinv, V, R k*k f64 | ev, raw, shift f64 | Jacobi
  const size_t log_bytes = k <= KMAX ? (size_t)JAC_SWEEPS * KMAX * (KMAX / 2) * sizeof(double2) : 0;
  const size_t bytes = (size_t)d * d * 4 + 2 * (size_t)d * k * 4 + (size_t)nchunk * k * k * 8 +
                       4 * (size_t)k * k * 8 + 2 * (size_t)k * 8 + log_bytes + sizeof(HjSync) + 8192;
  uint8_t* base = static_cast<uint8_t*>(scratch(ctx, SLOT_BASIS, bytes));
  if (!base) return ZOACT_ERR_NOMEM;
  Work w;
  size_t off = 0;
  auto take = [&](size_t b) { uint8_t* p = base + off; off += (b + 255) / 256 * 256; return p; };
  w.G = reinterpret_cast<float*>(take((size_t)d * d * 4));
  w.Q = reinterpret_cast<float*>(take((size_t)d * k * 4));
  w.Y = reinterpret_cast<float*>(take((size_t)d * k * 4));
  w.part = reinterpret_cast<double*>(take((size_t)nchunk * k * k * 8));
  w.S = reinterpret_cast<double*>(take((size_t)k * k * 8));
  w.Rinv = reinterpret_cast<double*>(take((size_t)k * k * 8));
  w.V = reinterpret_cast<double*>(take((size_t)k * k * 8));
  w.ev = reinterpret_cast<double*>(take((size_t)k * 8));
  w.R = reinterpret_cast<double*>(take((size_t)k * k * 8));
  w.log = reinterpret_cast<double2*>(take(log_bytes));
  w.raw = reinterpret_cast<double*>(take((size_t)k * 8));
  w.shift = reinterpret_cast<double*>(take(8));
  w.ints = reinterpret_cast<int*>(take((KMAX + 1) * sizeof(int)));
  w.sync = reinterpret_cast<HjSync*>(take(sizeof(HjSync)));
  w.nchunk = nchunk;
  (void)off;

  // 1. Gram
  if (xdtype == ZOACT_DT_FP32) {
    dim3 grid((d + 63) / 64, (d + 63) / 64);
    gram_f32_kernel<<<grid, 256, 0, ctx->stream>>>(static_cast<const float*>(X), w.G, n_tok, d); ++ctx->n_launch;
    ZOACT_CHECK_LAUNCH();
  } else {
    const int64_t n_pad = (n_tok + 7) / 8 * 8;
    void* Xt = scratch(ctx, SLOT_BASIS_X, (size_t)d * n_pad * 2);
    if (!Xt) return ZOACT_ERR_NOMEM;
    dim3 grid((unsigned)((n_pad + 31) / 32), (unsigned)((d + 31) / 32));
    if (xdtype == ZOACT_DT_BF16) {
      transpose_pad_kernel<__nv_bfloat16><<<grid, dim3(32, 8), 0, ctx->stream>>>(
          static_cast<const __nv_bfloat16*>(X), static_cast<__nv_bfloat16*>(Xt), n_tok, d, n_pad);
    } else {
      transpose_pad_kernel<__half><<<grid, dim3(32, 8), 0, ctx->stream>>>(static_cast<const __half*>(X),
                                                                          static_cast<__half*>(Xt), n_tok, d, n_pad);
    }
    ++ctx->n_launch;
    ZOACT_CHECK_LAUNCH();
    const int st = launch_gemm_tc_f32out(ctx, Xt, Xt, xdtype, d, d, (int)n_pad, w.G);
    if (st) return st;
  }
  // 2-3. sketch and subspace iteration
  const int64_t nq = (int64_t)d * k;
  omega_kernel<<<(unsigned)((nq / 4 + 255) / 256 + 1), 256, 0, ctx->stream>>>(w.Y, nq, seed); ++ctx->n_launch;
  ZOACT_CHECK_LAUNCH();
  int st = orth(ctx, w, w.Y, w.Q, d, k);
  if (st) return st;
  const dim3 gq_blocks((unsigned)((d + 63) / 64), (unsigned)((k + KMAX - 1) / KMAX));
  for (int it = 0; it < n_iter; ++it) {
    gemm_gq_kernel<<<gq_blocks, 256, 0, ctx->stream>>>(w.G, w.Q, w.Y, d, k); ++ctx->n_launch;
    ZOACT_CHECK_LAUNCH();
    st = orth(ctx, w, w.Y, w.Q, d, k);
    if (st) return st;
  }
  // 4. Rayleigh-Ritz
  gemm_gq_kernel<<<gq_blocks, 256, 0, ctx->stream>>>(w.G, w.Q, w.Y, d, k); ++ctx->n_launch;
  launch_atb(ctx, w, w.Q, w.Y, d, k);
  if (k <= KMAX) {
    jacobi_kernel<<<1, JAC_THREADS, JACOBI_SMEM, ctx->stream>>>(w.S, w.log, w.ints, w.ev, w.ints + 1, k);
    jacobi_vectors_kernel<<<k, 32, 0, ctx->stream>>>(w.log, w.ints, w.ints + 1, w.V, k);
    ctx->n_launch += 2;
  } else {
    chol_inv_kernel<<<1, 256, 0, ctx->stream>>>(w.S, w.R, w.Rinv, w.shift, k, ctx->d_status);
    ZOACT_CUDA_TRY(cudaMemsetAsync(w.sync, 0, sizeof(HjSync), ctx->stream));
    void* args[] = {&w.R, &w.sync, &k, &ctx->d_status};
    ZOACT_CUDA_TRY(cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(hj_kernel), dim3((unsigned)((k + 1) / 2)),
                                               dim3(HJ_THREADS), args, 0, ctx->stream));
    hj_norms_kernel<<<k, HJ_THREADS, 0, ctx->stream>>>(w.R, w.raw, k);
    hj_vectors_kernel<<<k, HJ_THREADS, 0, ctx->stream>>>(w.R, w.raw, w.shift, w.V, w.ev, k);
    ctx->n_launch += 4;
  }
  ZOACT_CHECK_LAUNCH();
  ritz_kernel<<<(unsigned)(((int64_t)d * r + 255) / 256), 256, 0, ctx->stream>>>(w.Q, w.V, U_out, d, k, r); ++ctx->n_launch;
  sign_fix_kernel<<<r, 256, 0, ctx->stream>>>(U_out, d, r, ctx->d_status); ++ctx->n_launch;
  if (evals_out) {
    f64_to_f32_kernel<<<1, 256, 0, ctx->stream>>>(w.ev, evals_out, k);
    ++ctx->n_launch;
  }
  ZOACT_CHECK_LAUNCH();
  return ZOACT_OK;
}

}  // namespace zoact
