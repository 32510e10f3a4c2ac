// Portable batched GEMM on CUDA cores: C = alpha * A B (+ C), arbitrary strides, a K axis that may be
// split into strided segments (the merged layer/head index of a cell), f16 / f32 inputs, fp32 or fp64
// accumulation.  It is the reference kernel family of the library: every tensor-core kernel is checked
// against it, and it serves fp32 caches and shapes the tensor-core kernels do not take.
#pragma once
#include <cooperative_groups.h>
#include <cstring>

#include "common.cuh"

namespace jolt {

struct GemmTask {
  const void *A, *B;
  void *C;
  int M, N, K;            // K: length of one segment
  int nseg, seg_inner;    // segment s -> (so, si) = (s / seg_inner, s % seg_inner)
  long long a_rs, a_cs, a_so, a_si;   // A(i, k, s) at i*a_rs + k*a_cs + so*a_so + si*a_si
  long long b_rs, b_cs, b_so, b_si;   // B(k, j, s) at k*b_rs + j*b_cs + so*b_so + si*b_si
  long long c_rs, c_cs;
  int ta, tb, tc;         // DType tags
  float alpha;
  const int *alpha_exp;   // optional: alpha *= 2^(*alpha_exp)
  int accumulate;         // 1: C += result
  int symmetric;          // 1: B = A^T, C symmetric: only the tiles on and below the diagonal are computed, the rest mirrored
};

__device__ __forceinline__ float load_elem(const void *p, int t, long long i) {
  if (t == DT_F16) return __half2float(((const __half *)p)[i]);
  if (t == DT_F32) return ((const float *)p)[i];
  return (float)((const double *)p)[i];
}

// 64 x 64 tiles, 4 x 4 per thread, operands converted once on the way into shared memory (an fp64 product of operands
// converted in the inner loop is bound by the conversions: a 1024 x 1024 x 4096 Gram took 1.5 ms where the fp64 pipe
// needs 0.13), the next 16 steps of K in registers.  A cluster of S CTAs shares a tile: each takes every S-th part of the
// K steps (all segments together), and the S partial tiles are added in a fixed order through distributed shared memory.  S
// is chosen so that a launch with few tiles still fills the machine (add_gemm): one 512-token cell has 16 output tiles
// and 64 dependent K steps each, 84 us with S = 1 and 13 us with S = 8.
template <typename Acc>
__global__ void __launch_bounds__(256) simt_gemm_kernel(const GemmTask *__restrict__ tasks) {
  namespace cg = cooperative_groups;
  cg::cluster_group cluster = cg::this_cluster();
  constexpr int BM = 64, BN = 64, BK = 16, P = 64 + 16 / (int)sizeof(Acc);      // pitch: rows start 16 bytes apart in the banks
  const GemmTask t = tasks[blockIdx.z];
  const int S = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  const int m0 = blockIdx.y * BM, n0 = (int)(blockIdx.x / S) * BN;
  if (m0 >= t.M || n0 >= t.N || (t.symmetric && n0 > m0)) return;               // the whole cluster
  __shared__ __align__(16) Acc sm[BM * BN > 2 * BK * P ? BM * BN : 2 * BK * P];
  Acc(*As)[P] = (Acc(*)[P])sm;
  Acc(*Bs)[P] = (Acc(*)[P])(sm + BK * P);
  const int tid = threadIdx.x;
  const int tx = tid & 15, ty = tid >> 4;
  Acc acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = Acc(0);
  const bool a_kfast = (t.a_cs == 1);
  const bool b_kfast = (t.b_rs == 1);
  const int spk = (t.K + BK - 1) / BK, steps = t.nseg * spk;
  const int s_lo = (int)((long long)steps * rank / S), s_hi = (int)((long long)steps * (rank + 1) / S);
  float pa[4], pb[4];
  auto fetch = [&](int step) {
    const int s = step / spk, k0 = (step - s * spk) * BK;
    const int so = s / t.seg_inner, si = s - so * t.seg_inner;
    const long long abase = so * t.a_so + si * t.a_si;
    const long long bbase = so * t.b_so + si * t.b_si;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int idx = tid + e * 256;
      int i, kk, j, kb;
      if (a_kfast) { i = idx >> 4; kk = idx & 15; } else { kk = idx >> 6; i = idx & 63; }
      if (b_kfast) { j = idx >> 4; kb = idx & 15; } else { kb = idx >> 6; j = idx & 63; }
      pa[e] = (m0 + i < t.M && k0 + kk < t.K) ? load_elem(t.A, t.ta, abase + (long long)(m0 + i) * t.a_rs + (long long)(k0 + kk) * t.a_cs) : 0.f;
      pb[e] = (n0 + j < t.N && k0 + kb < t.K) ? load_elem(t.B, t.tb, bbase + (long long)(k0 + kb) * t.b_rs + (long long)(n0 + j) * t.b_cs) : 0.f;
    }
  };
  if (s_lo < s_hi) fetch(s_lo);
  for (int step = s_lo; step < s_hi; ++step) {
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int idx = tid + e * 256;
      if (a_kfast) As[idx & 15][idx >> 4] = (Acc)pa[e]; else As[idx >> 6][idx & 63] = (Acc)pa[e];
      if (b_kfast) Bs[idx & 15][idx >> 4] = (Acc)pb[e]; else Bs[idx >> 6][idx & 63] = (Acc)pb[e];
    }
    __syncthreads();
    if (step + 1 < s_hi) fetch(step + 1);
#pragma unroll
    for (int kk = 0; kk < BK; ++kk) {
      Acc a[4], b[4];
      if constexpr (sizeof(Acc) == 8) {
        const double2 a0 = *(const double2 *)&As[kk][ty * 4], a1 = *(const double2 *)&As[kk][ty * 4 + 2];
        const double2 b0 = *(const double2 *)&Bs[kk][tx * 4], b1 = *(const double2 *)&Bs[kk][tx * 4 + 2];
        a[0] = a0.x; a[1] = a0.y; a[2] = a1.x; a[3] = a1.y; b[0] = b0.x; b[1] = b0.y; b[2] = b1.x; b[3] = b1.y;
      } else {
        const float4 a0 = *(const float4 *)&As[kk][ty * 4], b0 = *(const float4 *)&Bs[kk][tx * 4];
        a[0] = a0.x; a[1] = a0.y; a[2] = a0.z; a[3] = a0.w; b[0] = b0.x; b[1] = b0.y; b[2] = b0.z; b[3] = b0.w;
      }
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] += a[i] * b[j];
    }
    __syncthreads();
  }
  float alpha = t.alpha;
  if (t.alpha_exp) alpha = ldexpf(alpha, *t.alpha_exp);
  auto put = [&](int r, int c, Acc v) {
    const long long o = (long long)r * t.c_rs + (long long)c * t.c_cs;
    v *= (Acc)alpha;
    if (t.tc == DT_F32) {
      float *C = (float *)t.C;
      C[o] = t.accumulate ? C[o] + (float)v : (float)v;
    } else if (t.tc == DT_F64) {
      double *C = (double *)t.C;
      C[o] = t.accumulate ? C[o] + (double)v : (double)v;
    } else {
      ((__half *)t.C)[o] = __float2half_rn((float)v);
    }
  };
  auto emit = [&](int r, int c, Acc v) {
    if (r >= t.M || c >= t.N) return;
    put(r, c, v);
    if (t.symmetric && n0 < m0) put(c, r, v);
  };
  if (S == 1) {
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) emit(m0 + ty * 4 + i, n0 + tx * 4 + j, acc[i][j]);
    return;
  }
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) sm[(ty * 4 + i) * BN + tx * 4 + j] = acc[i][j];
  cluster.sync();
  const int per = BM * BN / S;
  for (int e = rank * per + tid; e < (rank + 1) * per; e += 256) {
    Acc v = Acc(0);
    for (int q = 0; q < S; ++q) v += cluster.map_shared_rank(sm, q)[e];
    emit(m0 + (e >> 6), n0 + (e & 63), v);
  }
  cluster.sync();                       // nobody leaves while its partial tile is being read
}

template <typename Acc>
inline void simt_gemm_launch(const GemmTask *d, int tn, int tm, int nz, int S, cudaStream_t s) {
  cudaLaunchConfig_t cfg;
  memset(&cfg, 0, sizeof cfg);
  cfg.gridDim = dim3(tn * S, tm, nz); cfg.blockDim = dim3(256); cfg.stream = s;
  cudaLaunchAttribute at;
  memset(&at, 0, sizeof at);
  at.id = cudaLaunchAttributeClusterDimension; at.val.clusterDim.x = S; at.val.clusterDim.y = 1; at.val.clusterDim.z = 1;
  cfg.attrs = &at; cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, simt_gemm_kernel<Acc>, d);
}

// fp32 in, fp32 out, one K segment, no accumulate: 128 x 64 tiles, 8 x 4 results per thread read from shared memory
// as 16-byte vectors, the next K slab fetched into registers while the current one is multiplied.
inline bool sgemm_fast_ok(const GemmTask &t) {
  return t.ta == DT_F32 && t.tb == DT_F32 && t.tc == DT_F32 && t.nseg == 1 && !t.accumulate && !t.alpha_exp;
}

__global__ void __launch_bounds__(256, 2) simt_sgemm_kernel(const GemmTask *__restrict__ tasks) {
  constexpr int BM = 128, BN = 64, BK = 16;
  const GemmTask t = tasks[blockIdx.z];
  const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
  if (m0 >= t.M || n0 >= t.N) return;
  __shared__ __align__(16) float As[BK][BM + 4];
  __shared__ __align__(16) float Bs[BK][BN + 4];
  const int tid = threadIdx.x;
  const int tx = tid & 15, ty = tid >> 4;
  const float *A = (const float *)t.A, *B = (const float *)t.B;
  const bool a_kfast = (t.a_cs == 1), b_kfast = (t.b_rs == 1);
  float acc[8][4];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
  float pa[8], pb[4];
  auto fetch = [&](int k0) {
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const int idx = tid + e * 256;
      int i, kk;
      if (a_kfast) { i = idx >> 4; kk = idx & 15; } else { kk = idx >> 7; i = idx & 127; }
      pa[e] = (m0 + i < t.M && k0 + kk < t.K) ? A[(long long)(m0 + i) * t.a_rs + (long long)(k0 + kk) * t.a_cs] : 0.f;
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int idx = tid + e * 256;
      int j, kb;
      if (b_kfast) { j = idx >> 4; kb = idx & 15; } else { kb = idx >> 6; j = idx & 63; }
      pb[e] = (n0 + j < t.N && k0 + kb < t.K) ? B[(long long)(k0 + kb) * t.b_rs + (long long)(n0 + j) * t.b_cs] : 0.f;
    }
  };
  fetch(0);
  for (int k0 = 0; k0 < t.K; k0 += BK) {
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const int idx = tid + e * 256;
      int i, kk;
      if (a_kfast) { i = idx >> 4; kk = idx & 15; } else { kk = idx >> 7; i = idx & 127; }
      As[kk][i] = pa[e];
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int idx = tid + e * 256;
      int j, kb;
      if (b_kfast) { j = idx >> 4; kb = idx & 15; } else { kb = idx >> 6; j = idx & 63; }
      Bs[kb][j] = pb[e];
    }
    __syncthreads();
    if (k0 + BK < t.K) fetch(k0 + BK);
#pragma unroll
    for (int kk = 0; kk < BK; ++kk) {
      const float4 a0 = *(const float4 *)&As[kk][ty * 8], a1 = *(const float4 *)&As[kk][ty * 8 + 4];
      const float4 b4 = *(const float4 *)&Bs[kk][tx * 4];
      const float a[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
      const float b[4] = {b4.x, b4.y, b4.z, b4.w};
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
    }
    __syncthreads();
  }
  float *C = (float *)t.C;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int r = m0 + ty * 8 + i;
    if (r >= t.M) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int c = n0 + tx * 4 + j;
      if (c < t.N) C[(long long)r * t.c_rs + (long long)c * t.c_cs] = acc[i][j] * t.alpha;
    }
  }
}

}  // namespace jolt
