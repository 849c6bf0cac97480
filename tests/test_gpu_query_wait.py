"""A wait for the Z tables of the q-query epilogue that gives up: every thread has to get the same answer.

Each epilogue thread waits for the tables by itself, so one may see them land while another sees the abort flag.  A thread
that left the tile on its own answer would leave the others in a named barrier that it never reaches.  The epilogue runs
here in a kernel of its own on a tile without rows (nothing is read from tensor memory or stored): a warp raises the
accumulator barrier once the tables have landed, the threads from ``split`` on then wait for a phase that nothing
completes, and the warp raises the abort flag.  Every wait is bounded.
"""
import ctypes
import subprocess

import pytest
import torch

from paper_2607_01125_gb300 import build as zbuild

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "pair_tc2_kernel.cuh"
using namespace zoact;
using namespace zoact::pairtc;

__device__ void pause(uint64_t ns) {
  const uint64_t t0 = tc::global_timer_ns();
  while (tc::global_timer_ns() - t0 < ns) {
  }
}

__global__ void __launch_bounds__(EPI_THREADS + 32)
epilogue_alone(const __grid_constant__ TmaSet tm, const __grid_constant__ Params prm, int split, int aborted, int* out) {
  extern __shared__ __align__(1024) uint8_t smem[];
  __shared__ SharedState2 ss;
  if (threadIdx.x == 0) {
    tc::mbar_init(tc::smem_u32(&ss.tload[0]), 1);
    tc::mbar_init(tc::smem_u32(&ss.tload[1]), 1);
    tc::mbar_init(tc::smem_u32(&ss.tmem_full[0]), 1);
    ss.abort_flag = 0;
    tc::fence_mbar_init();
  }
  __syncthreads();
  if (threadIdx.x < EPI_THREADS) {
    const int etid = threadIdx.x;
    uint32_t tphase = etid >= split ? 1u : 0u;
    bool pending = false;
    const bool ok = epi_multi4_staged<__nv_bfloat16, 8, MODE_PAIR>(
        prm, tm, &ss, reinterpret_cast<float*>(smem), etid, etid >> 7, (etid >> 5) & 3, etid & 31, 0, 0, BN, 0, 0, 0,
        &ss.abort_flag, pending, tphase);
    out[etid] = ok ? 1 : 0;
  } else if (threadIdx.x == EPI_THREADS) {
    pause(1000000ull);
    tc::mbar_arrive(tc::smem_u32(&ss.tmem_full[0]));
    pause(1000000ull);                 // thread 0 has taken it
    if (aborted) *const_cast<volatile int*>(&ss.abort_flag) = 1;
  }
}

extern "C" int run(const void* z, int d_out, int split, int aborted, int* status, int* out) {
  TmaSet tm{};
  Params p{};
  p.d_out = d_out;                     // rows = 0: no row of the tile is live
  p.r = 8;
  p.nb = 1;
  p.coef[0] = 1.f;
  p.Zt = static_cast<const float*>(z);
  p.zt_qstride = (int64_t)z_table_words(8, d_out);
  p.status = status;
  cudaFuncSetAttribute(epilogue_alone, cudaFuncAttributeMaxDynamicSharedMemorySize, TBL_FLOATS * 4);
  epilogue_alone<<<1, EPI_THREADS + 32, TBL_FLOATS * 4>>>(tm, p, split, aborted, out);
  if (cudaGetLastError() != cudaSuccess) return 1;
  return cudaDeviceSynchronize() == cudaSuccess ? 0 : 2;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("query_wait")
    (d / "k.cu").write_text(SOURCE)
    subprocess.run([zbuild._nvcc()] + zbuild.NVCC_FLAGS + ["-I", zbuild.CSRC, "-shared", "-o", str(d / "k.so"),
                                                           str(d / "k.cu")], check=True)
    return ctypes.CDLL(str(d / "k.so"))


@pytest.mark.parametrize("split,aborted,answer", [(256, 0, 1),    # every table lands
                                                  (256, 1, 1),    # ... and nobody looks at the flag
                                                  (255, 1, 0), (128, 1, 0), (33, 1, 0)])
def test_one_answer(lib, split, aborted, answer):
    words = 3 * 32 * 2 * 4               # 64 columns, rank tile 8
    z = torch.zeros(words, dtype=torch.int32, device="cuda:0")
    status = torch.zeros(1, dtype=torch.int32, device="cuda:0")
    out = torch.full((256,), 7, dtype=torch.int32, device="cuda:0")
    torch.cuda.synchronize()
    p = ctypes.c_void_p
    assert lib.run(p(z.data_ptr()), 64, split, aborted, p(status.data_ptr()), p(out.data_ptr())) == 0
    assert out.tolist() == [answer] * 256
    assert int(status) == 0
