// Cholesky factor and inverse of the Gram matrices of the range finder (Sec. 5; Q = R L^-T): G = L L^T in fp64, L^-1 written
// as an fp16 hi + lo pair, one cluster of eight CTAs per matrix, any n up to kCholClMaxN.
//
// Right-looking by panels of 32 columns on [G; I] = [L; X] L^T: the same panel operations that give the rows of L give the
// rows of X = L^-T.  X is upper triangular and the Schur complement only needs its lower triangle, so both live in one
// n x n column-major array W (in global memory, i.e. in L2: a panel step touches it once).  Per panel, two cluster barriers:
//   update   the solved panel P (n x 32) is staged in every CTA's shared memory and EVERY CTA forms the next diagonal
//            block; then warps 0 and 1 factor and invert it (redundantly: no CTA waits for another's factor) while the others
//            take their share of the trailing tiles W[I][J] -= P_I P_J^T, 32 x 16 at a time
//   solve    the rows of the next panel times the inverse of the diagonal block, 32 rows x 8 columns per warp
// What bounds it at n = 138 (five panels) is the chain: 32 pivots (a reciprocal square root each) per panel, shared-memory
// round trips, two cluster barriers; and instruction fetch, since nothing runs more than a few times, so the phases are loops
// over short bodies (a fully unrolled triangular solve of 32 columns alone took 6.7 us per panel).
// A pivot not above `dead_rel` of its original diagonal entry belongs to a direction that is dependent to working accuracy:
// its column of L and its row / column of L^-1 are zero, status bit 1.
#pragma once
#include <algorithm>
#include <mutex>
#include <cooperative_groups.h>
#include "device_once.h"
#include "small_solvers.cuh"

namespace jolt {

struct CholTask {
  const float *part; int n_chunks;          // Gram partials [n_chunks][kp][kp]: entry (row r, column c >= r) is summed in fp64
  int n, kp;
  double *W;                // n x n scratch (gram_sum_kernel -> chol_cluster_kernel)
  double *P;                // 2 * 32 * n scratch: solved panels, by parity
  __half *Lhi, *Llo;        // L^-1 [kp][kp], rows / columns >= n zero
  int *l_exp;               // L^-1 is stored times 2^l_exp
  int *status;
  double dead_rel;
  // Single-precision Grams lose pivots below about 1e-7 of their diagonal entry, and a lost pivot is a lost direction.
  // A first task with `redo` set reports whether a pivot came below `redo_rel`; a second one with `only` = that flag and
  // the fp64 Gram in `A64` (n x n) then does the work again (nothing otherwise).
  int *redo; double redo_rel;
  const int *only; const double *A64;
};
constexpr int kCholCluster = 8;
constexpr int kCholThreads = 512;
constexpr int kCholNB = 32;
constexpr int kCholClMaxN = 784;
__host__ __device__ inline int chol_pad(int n) { return (n + kCholNB - 1) / kCholNB * kCholNB; }
inline size_t chol_scratch_doubles(int n) { return (size_t)n * n + 2 * kCholNB * (size_t)n; }
__host__ __device__ inline size_t chol_smem_doubles(int n) { return (size_t)kCholNB * chol_pad(n) + 32 * 33 * 2 + 32 + n; }      // panel, D, X, reciprocal pivots, diagonal
inline size_t chol_smem_bytes_cl(int n) { return chol_smem_doubles(n) * sizeof(double); }

// Gram partials -> W (lower triangle, column-major: entry (i, j), i >= j, at W[j * n + i]): row j of the partials, summed in
// fp64; a warp per row, 64 entries and eight chunks in flight.  A launch of its own: eight CTAs alone would wait for the
// loads (10 us at n = 138, 55 us at n = 522).
constexpr int kGramRedRows = 8;
__global__ void __launch_bounds__(32 * kGramRedRows) gram_sum_kernel(const CholTask *__restrict__ tasks) {
  const CholTask &t = tasks[blockIdx.y];
  if (t.only && !*t.only) return;
  const int n = t.n, j = blockIdx.x * kGramRedRows + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (j >= n) return;
  const size_t cs = (size_t)t.kp * t.kp;
  const float *p = t.part + (size_t)j * t.kp;
  double *Wj = t.W + (size_t)j * n;
  const int chunks = t.n_chunks;
  if (t.A64) {
    for (int i = j + lane; i < n; i += 32) Wj[i] = t.A64[(size_t)j * n + i];
    return;
  }
  for (int i0 = j + lane; i0 < n + lane; i0 += 64) {
    const int q0 = min(i0, n - 1), q1 = min(i0 + 32, n - 1);
    double v0 = 0.0, v1 = 0.0;
    for (int ch = 0; ch < chunks; ch += 8) {
      float a[8], b[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const bool on = ch + q < chunks;
        const float *pc = p + (size_t)(ch + q) * cs;
        a[q] = on ? __ldg(pc + q0) : 0.f; b[q] = on ? __ldg(pc + q1) : 0.f;
      }
      v0 += (((double)a[0] + (double)a[1]) + ((double)a[2] + (double)a[3])) + (((double)a[4] + (double)a[5]) + ((double)a[6] + (double)a[7]));
      v1 += (((double)b[0] + (double)b[1]) + ((double)b[2] + (double)b[3])) + (((double)b[4] + (double)b[5]) + ((double)b[6] + (double)b[7]));
    }
    if (i0 < n) Wj[i0] = v0;
    if (i0 + 32 < n) Wj[i0 + 32] = v1;
  }
}

__device__ __forceinline__ void chol_pair_bar() { asm volatile("bar.sync 1, 64;" ::: "memory"); }

// Warps 0 and 1 factor the 32 x 32 block D (row r of lane r, shared memory, pitch 33) in place and form X = L^-T beside
// it.  Eight columns at a time: every lane of warp 0 factors the 8 x 8 block in registers, then the lanes of warp 0
// solve and update the rows of D, and one step behind them the lanes of warp 1 those of X (the unit rows).  Columns at or
// beyond w are dead.  Returns (warp 0) what happened to the pivots.
__device__ __forceinline__ int chol_factor_block(double (*D)[33], double (*X)[33], double *ip, const double *diag0, int w,
                                                 double dead_rel, double redo_rel, int warp, int lane) {
  int dead = 0;                            // bit 0: a pivot died, bit 1: one came below redo_rel
  double (*const M)[33] = warp == 0 ? D : X;
  if (warp == 1) {
#pragma unroll 4
    for (int c = 0; c < 32; ++c) X[lane][c] = c == lane ? 1.0 : 0.0;
  }
#pragma unroll 1
  for (int c0 = 0; c0 < 32; c0 += 8) {
    if (warp == 0) {
      double Lb[8][8], piv[8];
#pragma unroll
      for (int r = 0; r < 8; ++r)
#pragma unroll
        for (int c = 0; c <= r; ++c) Lb[r][c] = D[c0 + r][c0 + c];
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        const double d = Lb[c][c], dg = c0 + c < w ? diag0[c0 + c] : 0.0;
        const bool bad = !(d > dead_rel * dg) || !(dg > 0);
        const double rs = bad ? 0.0 : rsqrt_pos(d);
        Lb[c][c] = d * rs;
        if (c0 + c < w) dead |= (bad ? 1 : 0) | (d > redo_rel * dg ? 0 : 2);
        piv[c] = rs;
#pragma unroll
        for (int r = c + 1; r < 8; ++r) Lb[r][c] *= rs;
#pragma unroll
        for (int c2 = c + 1; c2 < 8; ++c2)
#pragma unroll
          for (int r = c2; r < 8; ++r) Lb[r][c2] = fma(-Lb[r][c], Lb[c2][c], Lb[r][c2]);
      }
      __syncwarp();
      if (lane == 0) {
#pragma unroll
        for (int r = 0; r < 8; ++r) {
          ip[c0 + r] = piv[r];
#pragma unroll
          for (int c = 0; c < r; ++c) D[c0 + r][c0 + c] = Lb[r][c];
        }
      }
      __syncwarp();
    } else chol_pair_bar();
    // rows below (warp 0), rows of X (warp 1): x_c = (p_c - sum_{l<c} x_l L[c][l]) / L[c][c]
    if (warp == 1 || lane >= c0 + 8) {
      double x[8];
#pragma unroll
      for (int c = 0; c < 8; ++c) x[c] = M[lane][c0 + c];
#pragma unroll
      for (int c = 0; c < 8; ++c) {
#pragma unroll
        for (int l = 0; l < c; ++l) x[c] = fma(-x[l], D[c0 + c][c0 + l], x[c]);
        x[c] *= ip[c0 + c];
      }
#pragma unroll
      for (int c = 0; c < 8; ++c) M[lane][c0 + c] = x[c];
    }
    __syncwarp();
    if (warp == 0) chol_pair_bar();          // the eight columns of L are final
#pragma unroll 1
    for (int j = c0 + 8; j < 32; j += 4) {
      if (warp == 1 || lane >= j) {
        double a[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) a[q] = M[lane][j + q];
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          const double v = M[lane][c0 + c];
#pragma unroll
          for (int q = 0; q < 4; ++q) a[q] = fma(-v, D[j + q][c0 + c], a[q]);
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) if (warp == 1 || j + q <= lane) M[lane][j + q] = a[q];
      }
    }
    __syncwarp();
  }
  return dead;
}

__global__ void __cluster_dims__(kCholCluster, 1, 1) __launch_bounds__(kCholThreads, 1) chol_cluster_kernel(const CholTask *__restrict__ tasks) {
  namespace cg = cooperative_groups;
  cg::cluster_group cluster = cg::this_cluster();
  const CholTask t = tasks[blockIdx.y];
  const int n = t.n, kp = t.kp, rank = (int)cluster.block_rank();
  if (n <= 0 || (t.only && !*t.only)) return;             // the whole cluster
  extern __shared__ __align__(16) double cc_sh[];
  const int np = chol_pad(n), NT = np / kCholNB;
  double *Ps = cc_sh;                                     // [32][np] the solved panel, column c at Ps + c * np
  double (*D)[33] = (double (*)[33])(Ps + (size_t)kCholNB * np);      // diagonal block
  double (*X)[33] = D + 32;                               // L^-T of it
  double *ip = (double *)(X + 32);                        // [32] reciprocal pivots
  double *diag0 = ip + 32;                                // [n] original diagonal
  __shared__ float s_red[kCholThreads / 32], s_mx[kCholCluster];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  constexpr int NW = kCholThreads / 32;
  const int gw = warp * kCholCluster + rank;              // warp number in the cluster: neighbouring units go to different SMs
  double *const W = t.W;
  for (int i = tid; i < n; i += kCholThreads) diag0[i] = __ldcg(W + (size_t)i * n + i);
  // the first diagonal block
  for (int e = tid; e < 1024; e += kCholThreads) {
    const int r = e & 31, c = e >> 5;
    D[r][c] = (r < n && c <= r) ? __ldcg(W + (size_t)c * n + r) : 0.0;
  }
  __syncthreads();
  int dead = 0;
  float mx = 0.f;
  if (warp < 2) dead = chol_factor_block(D, X, ip, diag0, min(32, n), t.dead_rel, t.redo_rel, warp, lane);
  __syncthreads();
  for (int p = 0; p < NT; ++p) {
    const int j0 = p * kCholNB, w = min(kCholNB, n - j0);
    double *P = t.P + (size_t)(p & 1) * kCholNB * n;
    // ---- solve: rows of X above, the unit rows inside (X itself), rows of L below; results go to P
    for (int u = gw; u < 4 * NT; u += NW * kCholCluster) {
      const int I = u >> 2, cg8 = (u & 3) * 8, i = I * kCholNB + lane;
      double acc[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) acc[q] = 0.0;
      if (I == p) {
#pragma unroll
        for (int q = 0; q < 8; ++q) acc[q] = X[lane][cg8 + q];
      } else {
#pragma unroll 1
        for (int l0 = 0; l0 < cg8 + 8; l0 += 8) {        // X is upper triangular
          double v[8];
#pragma unroll
          for (int l = 0; l < 8; ++l) v[l] = (i < n && l0 + l < w) ? __ldcg(W + (size_t)(j0 + l0 + l) * n + i) : 0.0;
#pragma unroll
          for (int l = 0; l < 8; ++l)
#pragma unroll
            for (int q = 0; q < 8; ++q) acc[q] = fma(v[l], X[l0 + l][cg8 + q], acc[q]);
        }
      }
      if (i < n) {
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          const int c = cg8 + q;
          if (c < w) {
            if (I <= p) mx = fmaxf(mx, fabsf((float)acc[q]));
            __stcg(P + (size_t)c * n + i, acc[q]);       // W itself is still read by the other units of these rows
          }
        }
      }
    }
    cluster.sync();
    if (p + 1 == NT) {                                    // the last panel's X rows go back to W
      for (int c = gw; c < w; c += NW * kCholCluster)
        for (int i = lane; i <= j0 + c; i += 32) __stcg(W + (size_t)(j0 + c) * n + i, __ldcg(P + (size_t)c * n + i));
      cluster.sync();
      break;
    }
    // ---- the solved panel into shared memory
    for (int e = tid; e < kCholNB * np; e += kCholThreads) {
      const int c = e / np, i = e - c * np;
      Ps[e] = (i < n && c < w) ? __ldcg(P + (size_t)c * n + i) : 0.0;
    }
    __syncthreads();
    const int m0 = j0 + kCholNB, wn = min(kCholNB, n - m0);
    {                                                     // next diagonal block: lane = row, two columns per warp
      const int i = m0 + lane, c = 2 * warp;
      double a0 = (i < n && c <= lane) ? __ldcg(W + (size_t)(m0 + c) * n + i) : 0.0;
      double a1 = (i < n && c + 1 <= lane) ? __ldcg(W + (size_t)(m0 + c + 1) * n + i) : 0.0;
#pragma unroll 8
      for (int l = 0; l < 32; ++l) {
        const double v = Ps[(size_t)l * np + i];
        const double2 q = *(const double2 *)(Ps + (size_t)l * np + m0 + c);
        a0 = fma(-v, q.x, a0); a1 = fma(-v, q.y, a1);
      }
      D[lane][c] = c <= lane ? a0 : 0.0;
      D[lane][c + 1] = c + 1 <= lane ? a1 : 0.0;
    }
    __syncthreads();
    if (warp < 2) dead |= chol_factor_block(D, X, ip, diag0 + m0, wn, t.dead_rel, t.redo_rel, warp, lane);
    else {
      // X rows of the panel go back to W
      for (int c = warp - 2 + (NW - 2) * rank; c < w; c += (NW - 2) * kCholCluster)
        for (int i = lane; i <= j0 + c; i += 32) __stcg(W + (size_t)(j0 + c) * n + i, Ps[(size_t)c * np + i]);
      // trailing tiles: columns J > p in halves of 16, rows I <= p (X; first touched by panel I) and I >= J
      const int uw = (warp - 2) * kCholCluster + rank, nu = (NW - 2) * kCholCluster;
      int u = uw;
      for (int J = p + 1; J < NT; ++J) {
        const int cnt = 2 * (p + 1 + NT - J);
        for (; u < cnt; u += nu) {
          const int Iq = u >> 1, I = Iq <= p ? Iq : J + (Iq - p - 1), jc = J * kCholNB + (u & 1) * 16;
          if (jc >= n || (I == p + 1 && J == p + 1)) continue;         // the next diagonal block is formed above
          const int i = I * kCholNB + lane;
          double acc[16];
          const bool fresh = I == p;
#pragma unroll
          for (int q = 0; q < 16; ++q) acc[q] = (!fresh && i < n && jc + q < n) ? __ldcg(W + (size_t)(jc + q) * n + i) : 0.0;
          const double *pi = Ps + i, *pj = Ps + jc;
#pragma unroll 4
          for (int l = 0; l < 32; ++l) {
            const double v = pi[(size_t)l * np];
#pragma unroll
            for (int q = 0; q < 16; q += 2) {
              const double2 b = *(const double2 *)(pj + (size_t)l * np + q);
              acc[q] = fma(-v, b.x, acc[q]); acc[q + 1] = fma(-v, b.y, acc[q + 1]);
            }
          }
#pragma unroll
          for (int q = 0; q < 16; ++q)
            if (i < n && jc + q < n) __stcg(W + (size_t)(jc + q) * n + i, acc[q]);
        }
        u -= cnt;
      }
    }
    cluster.sync();
  }
  if (warp == 0 && lane == 0 && rank == 0) {
    if (t.redo) *t.redo = (dead & 2) != 0;
    if ((dead & 1) && t.status && !t.redo) atomicOr(t.status, 2);
  }
  // ---- L^-1 (row i, column c <= i) = X[c][i] = W[i * n + c], scaled so that the largest entry lies in [2^9, 2^10)
  for (int o = 16; o; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if (lane == 0) s_red[warp] = mx;
  __syncthreads();
  if (warp == 0) {
    mx = lane < NW ? s_red[lane] : 0.f;
    for (int o = 16; o; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if (lane < kCholCluster) cluster.map_shared_rank(s_mx, lane)[rank] = mx;
  }
  cluster.sync();
  mx = 0.f;
  for (int q = 0; q < kCholCluster; ++q) mx = fmaxf(mx, s_mx[q]);
  int e = 0;
  if (mx > 0.f && isfinite(mx)) e = 9 - ilogbf(mx);
  if (tid == 0 && rank == 0) *t.l_exp = e;
  const double sc = ldexp(1.0, e);
  for (int i = gw; i < kp; i += NW * kCholCluster)
    for (int cb = 2 * lane; cb < kp + 2 * lane; cb += 256) {        // four pairs of columns in flight per lane
      double v[4][2];
#pragma unroll
      for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int u = 0; u < 2; ++u) { const int c = cb + 64 * q + u; v[q][u] = (i < n && c <= i) ? __ldcg(W + (size_t)i * n + c) : 0.0; }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int c = cb + 64 * q;
        if (c >= kp) continue;
        const __half2 h = __floats2half2_rn((float)(v[q][0] * sc), (float)(v[q][1] * sc));
        const float2 hf = __half22float2(h);
        *(__half2 *)(t.Lhi + (size_t)i * kp + c) = h;
        *(__half2 *)(t.Llo + (size_t)i * kp + c) = __floats2half2_rn((float)(v[q][0] * sc) - hf.x, (float)(v[q][1] * sc) - hf.y);
      }
    }
}

inline void chol_cluster_launch(const CholTask *d_tasks, int count, int max_n, cudaStream_t s) {
  static DeviceOnce once;
  once([] { cudaFuncSetAttribute(chol_cluster_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(kSmemOptIn - 1024)); });
  gram_sum_kernel<<<dim3((max_n + kGramRedRows - 1) / kGramRedRows, count), 32 * kGramRedRows, 0, s>>>(d_tasks);
  chol_cluster_kernel<<<dim3(kCholCluster, count), kCholThreads, chol_smem_bytes_cl(max_n), s>>>(d_tasks);
}

}  // namespace jolt
