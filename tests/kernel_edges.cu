// Single kernels of the library behind plain functions, for tests/test_gpu_kernel_edges.py.
#include <cstdint>
#include <cstring>
#include <cuda_fp16.h>
#include "small_solvers.cuh"
#include "tc_common.cuh"
#include "tc_gemm.cuh"
#include "tc_orth.cuh"

using namespace jolt;

__global__ void rcp_kernel(const double *d, double *out, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) { out[i] = tc::rcp_pos(d[i]); out[n + i] = 1.0 / d[i]; }
}

extern "C" int edge_rcp(const double *d, double *out, int n) {
  rcp_kernel<<<(n + 255) / 256, 256>>>(d, out, n);
  return (int)cudaDeviceSynchronize();
}

// A64: n x n fp64, or part: n_chunks x kp x kp fp32; L64: n * n + 1; hi, lo: kp x kp; info: {exponent of L^-1, status}
extern "C" int edge_cholesky(const double *A64, const float *part, int n_chunks, int n, int kp, double dead_rel, double *L64, void *hi, void *lo, int *info) {
  tc::CholInvTask t;
  memset(&t, 0, sizeof t);
  t.part = part; t.n_chunks = n_chunks; t.kp = kp; t.A64 = A64; t.k = n;
  t.Lhi = (__half *)hi; t.Llo = (__half *)lo; t.l_exp = info; t.L64 = L64; t.status = info + 1; t.dead_rel = dead_rel;
  tc::CholInvTask *d = nullptr;
  int e = (int)cudaMalloc(&d, sizeof t);
  if (e) return e;
  e = (int)cudaMemcpy(d, &t, sizeof t, cudaMemcpyHostToDevice);
  if (!e) e = (int)cudaFuncSetAttribute(tc::cholinv_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)tc::cholinv_smem_bytes(tc::kCholInvMaxN));
  if (!e) {
    tc::cholinv_kernel<<<1, tc::kCholInvThreads, tc::cholinv_smem_bytes(n)>>>(d);
    e = (int)cudaDeviceSynchronize();
  }
  cudaFree(d);
  return e;
}
