// Symmetric eigen-solver in fp64 for the small dense problems of the path: the mode-3 Gram (Sec. 4), B B^T of the
// randomized token factor (Sec. 5) and the T x T Gram of the exact token path.
//
//   A = H T H^T         Householder tridiagonalisation: td_small_kernel (one CTA, n <= 160) or td_big_kernel (a cluster of
//                       16 CTAs per matrix, n <= 1024)
//   eigenvalues of T    Sturm counts, 32-way (9-way for large n) section: td_values_kernel
//   eigenvectors of T   two inverse iterations with partial pivoting, one thread per vector: td_vectors_kernel; members
//                       of a cluster of eigenvalues are re-orthogonalised by td_orth_kernel
//   U = H Z             td_back_kernel
//
// Every phase is a chain of dependent steps, so the time of a solve is latency times chain length: a tridiagonalisation
// has n steps where a Jacobi solver has (sweeps) x n rounds.  The result is fp64 throughout (residuals and
// orthogonality of the returned fp32 vectors are their rounding).
#pragma once
#include <algorithm>
#include <cstring>
#include <mutex>
#include <type_traits>

#include <cooperative_groups.h>
#include "device_once.h"
#include "small_solvers.cuh"

namespace jolt {

struct TdTask {
  const double *A;      // n x n symmetric, row-major (not modified)
  int n;
  double *d, *e, *h;    // n each: diagonal, off-diagonal, reflector factors (all of the scaled matrix)
  double *V;            // n x n: reflector k in V[k * n + i], i > k
  double *lam;          // n eigenvalues, descending, of the scaled matrix
  double *X;            // 5 * n * ldx: LU of the shifted matrix and the iterate (last), element (i, vector) at i * ldx + vector
  double *xn;           // ldx: 1 / norm of each iterate
  double *G;            // 6 per group of four reflectors: their products (see td_back_kernel)
  double *R;            // n x n: rows of the work matrix that do not fit in shared memory (n > kTdSmallMaxN)
  int ldx;              // r_out rounded up to a multiple of 32 (0: no vectors)
  int *exp2;            // the scaled matrix is A * 2^-exp2
  float *U_out; int ld_out, r_out; float *w_out; int w_sqrt;
  int *status;
};

constexpr int kTdSmallMaxN = 160;
constexpr int kTdMaxN = 1024;
constexpr double kTdClusterGap = 1e-9;    // eigenvalues closer than this (relative to the spread of T) are one cluster

inline size_t td_scratch_doubles(int n, int r) {
  const size_t ldx = (size_t)((r + 31) / 32 * 32);
  return 4 * (size_t)n + 6 * (size_t)((n + 3) / 4) + (size_t)n * n * (n > kTdSmallMaxN ? 2 : 1) + 5 * (size_t)n * ldx + ldx + 8;
}
// carves a task's scratch out of a block of td_scratch_doubles(n, r_out) doubles
inline void td_set_scratch(TdTask &t, double *p) {
  const size_t n = t.n;
  t.ldx = t.U_out ? (t.r_out + 31) / 32 * 32 : 0;
  t.d = p; t.e = p + n; t.h = p + 2 * n; t.lam = p + 3 * n; t.V = p + 4 * n;
  p = t.V + n * n;
  t.R = n > (size_t)kTdSmallMaxN ? p : nullptr;
  if (t.R) p += n * n;
  t.X = p; p += 5 * n * t.ldx;
  t.xn = p; p += t.ldx;
  t.G = p; p += 6 * ((n + 3) / 4);
  t.exp2 = (int *)p;
}

__device__ __forceinline__ double td_warp_sum(double v) {
#pragma unroll
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
// exponent of the largest diagonal entry (one warp): the matrix is positive semidefinite, so no entry exceeds it
__device__ __forceinline__ int td_diag_exp(const double *A, int n, int lane) {
  double mx = 0.0;
  for (int i = lane; i < n; i += 32) mx = fmax(mx, fabs(A[(size_t)i * n + i]));
  for (int o = 16; o; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  int e2 = 0;
  if (mx > 0.0 && mx < 1e300) frexp(mx, &e2);
  return e2;
}

template <int CNT>      // sums q[0 .. CNT) over the warp; lane l gets the sum of index l * CNT / 32
__device__ __forceinline__ double td_red(double (&q)[CNT], int lane) {
  int o = 16;
#pragma unroll
  for (int m = CNT / 2; m >= 1; m >>= 1, o >>= 1) {
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int u = 0; u < m; ++u) {
      const double give = up ? q[u] : q[u + m], keep = up ? q[u + m] : q[u];
      q[u] = keep + __shfl_xor_sync(0xffffffffu, give, o);
    }
  }
  double v = q[0];
#pragma unroll
  for (; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
// ---------------------------------------------------------------------------------------------- n <= 160: one CTA
// Sixteen worker warps keep the trailing 128 x 128 block in registers, rows and columns cyclic over a 4 x 4 grid of
// warps and an 8 x 4 grid of lanes (4 x 8 entries per thread; the matrix sits at the END of the block, so finished rows
// and columns are skipped a quarter at a time); the leading n - 128 rows of a larger matrix live in shared memory.  A
// seventeenth warp owns the chain.  Step k, three barriers:
//   A  -> A2  the head warp adds up p = A v of the previous reflector and forms w = h p - K v
//   A2 -> B   the workers apply it (A -= v w^T + w v^T) while the head warp applies it to row k alone and forms
//             reflector k from it
//   B  -> A   the workers multiply by the new reflector and publish row k + 1
// What bounds it: the chain.  3 (n - k)^2 fp64 operations per step on a pipe of 64 lanes per clock are 260 cycles at
// n = 128, against about 900 of barriers, two warp sums, a square root and shared-memory round trips.  The lane grid keeps
// the reduction of a row at three exchanges (with a row spread over a whole warp the exchanges alone were 290 cycles
// per step, and with every warp forming w for itself another 170).
// Vectors are stored in the order (index mod 4, index / 4): a warp then reads its rows and columns from neighbouring words.
constexpr int kTdWorkers = 16;
constexpr int kTdSmallThreads = 32 * (kTdWorkers + 1);
constexpr int kTdVec = 128 + 32;          // a vector: 128 entries of the register block, 32 of the head part
__host__ __device__ inline size_t td_small_smem_bytes(int n) {
  const int h0 = n > 128 ? n - 128 : 0;
  return ((size_t)2 * kTdVec + kTdVec + 5 * kTdVec + kTdVec + 3 * (size_t)n + 4 + (size_t)h0 * n) * sizeof(double);
}

template <int L>      // worker, A2 -> B
__device__ __forceinline__ void td_apply(double (&A)[4][8], const double2 *vwr, const double2 *vwc) {
#pragma unroll
  for (int hf = L / 2; hf < 2; ++hf) {      // two rows at a time: all four would not leave room for the entries
    const double2 r0 = vwr[16 * hf], r1 = vwr[16 * hf + 8];
#pragma unroll
    for (int b = 2 * L; b < 8; ++b) {
      const double2 q = vwc[4 * b];
      if (2 * hf >= L) A[2 * hf][b] = fma(-r0.x, q.y, fma(-r0.y, q.x, A[2 * hf][b]));
      A[2 * hf + 1][b] = fma(-r1.x, q.y, fma(-r1.y, q.x, A[2 * hf + 1][b]));
    }
  }
}
template <int L>      // worker, B -> A: this lane's share of its four rows' products, reduced over the four column lanes
__device__ __forceinline__ double td_product(const double (&A)[4][8], const double *vc, int lane) {
  double p[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
  for (int b = 2 * L; b < 8; ++b) {
    const double v = vc[4 * b];
#pragma unroll
    for (int a = L; a < 4; ++a) p[a] = fma(A[a][b], v, p[a]);
  }
  const bool u1 = lane & 1, u2 = lane & 2;
  const double k0 = u1 ? p[2] : p[0], k1 = u1 ? p[3] : p[1], g0 = u1 ? p[0] : p[2], g1 = u1 ? p[1] : p[3];
  const double q0 = k0 + __shfl_xor_sync(0xffffffffu, g0, 1), q1 = k1 + __shfl_xor_sync(0xffffffffu, g1, 1);
  return (u2 ? q1 : q0) + __shfl_xor_sync(0xffffffffu, u2 ? q0 : q1, 2);       // row a = 2 (lane & 1) + (lane >> 1 & 1)
}

__global__ void __launch_bounds__(kTdSmallThreads, 1) td_small_kernel(const TdTask *__restrict__ tasks) {
  const TdTask &t = tasks[blockIdx.x];
  const int n = t.n, base = n - 128, h0 = base > 0 ? base : 0;
  if (n <= 0) return;
  extern __shared__ __align__(16) double td_sh[];
  double2 *vw = (double2 *)td_sh;           // [kTdVec] (v, w) of the previous reflector
  double *vn = td_sh + 2 * kTdVec;          // [kTdVec] new reflector
  double *ps = vn + kTdVec;                 // [5][kTdVec] partial products (one per warp column; the head part's)
  double *rowb = ps + 5 * kTdVec;           // [kTdVec] row k with every reflector but the previous one applied
  double *sde = rowb + kTdVec;              // d, e, h: [3][n]
  double *S1 = sde + 3 * n + 4;             // [h0][n] leading rows
  __shared__ double s_scale;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const double *const Ag = t.A;
  double *const Vg = t.V;
  if (warp == 0) {
    const int e2 = td_diag_exp(Ag, n, lane);
    if (lane == 0) { s_scale = ldexp(1.0, -e2); *t.exp2 = e2; }
  }
  for (int i = tid; i < 9 * kTdVec; i += kTdSmallThreads) td_sh[i] = 0.0;
  __syncthreads();
  const double sc = 0.5 * s_scale;
  // position of matrix index i in a vector: the register block in (index mod 4, index / 4) order, the head part behind it
  auto pos = [&](int i) { return i < h0 ? 128 + i : (((i - base) & 3) << 5) + ((i - base) >> 2); };
  for (int i = tid; i < n; i += kTdSmallThreads) rowb[pos(i)] = (Ag[i] + Ag[(size_t)i * n]) * sc;
  if (warp == kTdWorkers) {
    // ---------------- head warp: entries base + 4 lane + c, and `lane` of the head part
    double v[4] = {0.0, 0.0, 0.0, 0.0}, w[4], vh = 0.0, wh = 0.0, h = 0.0;
    for (int k = 0; k < n; ++k) {
      __syncthreads();                                             // A: products of the previous reflector are in
      const bool head = k < h0;
      const int k1 = k + 1 < n ? k + 1 : k, pk = pos(k), p1 = pos(k1);
      double rb[4], dot = 0.0;
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const double *q = ps + 32 * c + lane;
        w[c] = (q[0] + q[kTdVec]) + (q[2 * kTdVec] + q[3 * kTdVec]);
        if (k <= h0 && h0) w[c] += q[4 * kTdVec];
        dot = fma(w[c], v[c], dot);
        rb[c] = rowb[32 * c + lane];
      }
      if (head) { wh = ps[4 * kTdVec + 128 + lane]; dot = fma(wh, vh, dot); }
      const double r1 = rowb[p1];
      dot = td_warp_sum(dot);
      const double K = 0.5 * h * h * dot;
#pragma unroll
      for (int c = 0; c < 4; ++c) { w[c] = fma(h, w[c], -K * v[c]); vw[32 * c + lane] = make_double2(v[c], w[c]); }
      if (head) { wh = fma(h, wh, -K * vh); vw[128 + lane] = make_double2(vh, wh); }
      __syncthreads();                                             // A2: (v, w) is out
      const double2 qk = vw[pk], q1 = vw[p1];
      const double alpha = fma(-qk.x, q1.y, fma(-qk.y, q1.x, r1));
      double s = 0.0, ch = 0.0;
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const int j = base + 4 * lane + c;
        const double x = fma(-qk.x, w[c], fma(-qk.y, v[c], rb[c]));
        if (j == k) sde[k] = x;
        v[c] = j > k ? x : 0.0;
        s = fma(v[c], v[c], s);
      }
      if (head) {
        const double x = fma(-qk.x, wh, fma(-qk.y, vh, rowb[128 + lane]));
        if (lane == k) sde[k] = x;
        ch = lane > k && lane < h0 ? x : 0.0;
        s = fma(ch, ch, s);
      }
      if (k == n - 1) break;
      s = td_warp_sum(s);
      double beta = alpha, v1 = 0.0, den = 0.0;
      const bool live = s > 1e-60;
      if (live) {
        const double nrm = s * rsqrt_pos(s);
        beta = alpha >= 0.0 ? -nrm : nrm;
        v1 = alpha - beta;
        den = fma(nrm, fabs(alpha), s);
      }
      double *const Vk = Vg + (size_t)k * n;
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const int j = base + 4 * lane + c;
        v[c] = !live ? 0.0 : (j == k1 ? v1 : v[c]);
        vn[32 * c + lane] = v[c];
      }
      vh = !live ? 0.0 : (lane == k1 && k1 < h0 ? v1 : ch);
      if (head) vn[128 + lane] = vh;
      __syncthreads();                                             // B: the new reflector is out
#pragma unroll
      for (int c = 0; c < 4; ++c) { const int j = base + 4 * lane + c; if (j >= h0) Vk[j] = v[c]; }
      if (lane < h0) Vk[lane] = vh;
      h = live ? 1.0 / den : 0.0;
      if (lane == 0) { sde[n + k] = beta; sde[2 * n + k] = h; }
    }
    if (lane == 0) { sde[2 * n - 1] = 0.0; sde[3 * n - 1] = 0.0; }
  } else {
    // ---------------- worker warps: rows base + wr + 4 (lr + 8 a), columns base + wc + 4 (lc + 4 b)
    const int wr = warp >> 2, wc = warp & 3, lr = lane >> 2, lc = lane & 3;
    const int ra = 2 * (lc & 1) + (lc >> 1);
    double A[4][8];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int b = 0; b < 8; ++b) {
        const int i = base + wr + 4 * (lr + 8 * a), j = base + wc + 4 * (lc + 4 * b);
        A[a][b] = (i >= 0 && j >= 0) ? (Ag[(size_t)i * n + j] + Ag[(size_t)j * n + i]) * sc : 0.0;
      }
    for (int i = warp; i < h0; i += kTdWorkers)
      for (int j = lane; j < n; j += 32) S1[(size_t)i * n + j] = (Ag[(size_t)i * n + j] + Ag[(size_t)j * n + i]) * sc;
    for (int k = 0; k < n; ++k) {
      __syncthreads();                                             // A
      __syncthreads();                                             // A2
      if (k == n - 1) break;
      const bool head = k < h0;
      const int l = (k - base) >> 5;        // quarters with index below l are finished (negative while in the head part)
      const double2 *vwr = vw + 32 * wr + lr, *vwc = vw + 32 * wc + lc;
      if (head)
        for (int i = warp; i < h0; i += kTdWorkers) {
          const double2 q = vw[128 + i];
          double *Si = S1 + (size_t)i * n;
          for (int j = lane; j < n; j += 32) { const double2 u = vw[pos(j)]; Si[j] = fma(-q.x, u.y, fma(-q.y, u.x, Si[j])); }
        }
      if (l <= 0) td_apply<0>(A, vwr, vwc);
      else if (l == 1) td_apply<1>(A, vwr, vwc);
      else if (l == 2) td_apply<2>(A, vwr, vwc);
      else td_apply<3>(A, vwr, vwc);
      __syncthreads();                                             // B
      const double *vc = vn + 32 * wc + lc;
      double p;
      if (l <= 0) p = td_product<0>(A, vc, lane);
      else if (l == 1) p = td_product<1>(A, vc, lane);
      else if (l == 2) p = td_product<2>(A, vc, lane);
      else p = td_product<3>(A, vc, lane);
      ps[wc * kTdVec + 32 * wr + lr + 8 * ra] = p;
      const int rel = k + 1 - base - wr;    // row k + 1 with every reflector but the new one applied
      if (k + 1 >= h0 && (rel & 3) == 0 && ((rel >> 2) & 7) == lr) {
        const bool hi = rel & 64, lo = rel & 32;
#pragma unroll
        for (int b = 0; b < 8; ++b) {
          const double x = lo ? A[1][b] : A[0][b], y = lo ? A[3][b] : A[2][b];
          rowb[32 * wc + lc + 4 * b] = hi ? y : x;
        }
      }
      if (head) {
        for (int i = warp; i < h0; i += kTdWorkers) {
          const double *Si = S1 + (size_t)i * n;
          double ph = 0.0;
          for (int j = lane; j < n; j += 32) { ph = fma(Si[j], vn[pos(j)], ph); if (i == k + 1) rowb[pos(j)] = Si[j]; }
          ph = td_warp_sum(ph);
          if (lane == 0) ps[4 * kTdVec + 128 + i] = ph;
        }
        if (tid < 128) {                    // the head part's columns in the products of the register block's rows
          const int i = base + 4 * (tid & 31) + (tid >> 5);
          double ph = 0.0;
          for (int j = k + 1; j < h0; ++j) ph = fma(S1[(size_t)j * n + i], vn[128 + j], ph);
          ps[4 * kTdVec + tid] = ph;
        }
      }
    }
  }
  __syncthreads();
  for (int e = tid; e < n; e += kTdSmallThreads) { t.d[e] = sde[e]; t.e[e] = sde[n + e]; t.h[e] = sde[2 * n + e]; }
}

// ---------------------------------------------------------------------------------------------- n <= 1024: a cluster
// Sixteen CTAs per matrix, row i on CTA i mod 16.  One cluster barrier per step: a CTA sends (p_i, a_i,k+1) of its rows
// to all sixteen (column k + 1 is row k + 1, so no CTA has to send a whole row), and after the barrier every CTA forms
// w, the updated column and the next reflector redundantly; ONE pass over its rows then applies the previous reflector
// and multiplies by the new one.  Rows stay in shared memory as far as they fit (all of them up to n = 600); the rest,
// always the rows that finish first, are streamed through the caches.
constexpr int kTdCluster = 16;
constexpr int kTdBigThreads = 512;
__host__ __device__ inline int td_big_slots(int n) { return (n + kTdCluster - 1) / kTdCluster; }
__host__ __device__ inline size_t td_big_vec_doubles(int n) { return 4 * (size_t)n + 4 * (size_t)n + 64; }   // pa[2] (p, a), vold, wold, vnew, e
inline int td_big_smem_slots(int n) {
  const size_t room = kSmemOptIn - 2048 - td_big_vec_doubles(n) * sizeof(double);
  return (int)std::min<size_t>(td_big_slots(n), room / (n * sizeof(double)));
}
inline size_t td_big_smem_bytes(int n) { return (td_big_vec_doubles(n) + (size_t)td_big_smem_slots(n) * n) * sizeof(double); }

__device__ __forceinline__ double td_block_sum(double v, double *red, int warp, int lane) {    // every thread gets the sum
  v = td_warp_sum(v);
  if (lane == 0) red[warp] = v;
  __syncthreads();
  const double2 *r2 = (const double2 *)red;
  double2 s0 = r2[0], s1 = r2[1], s2 = r2[2], s3 = r2[3];
  const double2 a = r2[4], b = r2[5], c = r2[6], d = r2[7];
  s0.x += a.x; s0.y += a.y; s1.x += b.x; s1.y += b.y; s2.x += c.x; s2.y += c.y; s3.x += d.x; s3.y += d.y;
  return ((s0.x + s0.y) + (s1.x + s1.y)) + ((s2.x + s2.y) + (s3.x + s3.y));
}

// NR rows of one warp share every load of the vectors; the entries of four column groups are requested before the first
// of them is written back (rows beyond the shared memory come from the caches)
template <int NR>
__device__ __forceinline__ void td_big_rows(double *const (&rp)[NR], const int (&row)[NR], int n, int k, const double *vo, const double *wo,
                                            const double *vn, int lane, double (&p)[NR], double (&a1)[NR]) {
  constexpr int U = NR == 1 ? 8 : 4;
  double vi[NR], wi[NR];
#pragma unroll
  for (int q = 0; q < NR; ++q) { vi[q] = vo[row[q]]; wi[q] = wo[row[q]]; p[q] = 0.0; a1[q] = 0.0; }
  const int j0 = (k + 1) & ~31;
  for (int jb = j0 + lane; jb < n + lane; jb += 32 * U) {
    double x[U][NR];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int j = jb + 32 * u;
#pragma unroll
      for (int q = 0; q < NR; ++q) x[u][q] = j < n ? rp[q][j] : 0.0;
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int j = jb + 32 * u;
      if (j < n) {
        const double vj = vo[j], wj = wo[j], nj = vn[j];
#pragma unroll
        for (int q = 0; q < NR; ++q) {
          const double y = fma(-vi[q], wj, fma(-wi[q], vj, x[u][q]));
          rp[q][j] = y;
          p[q] = fma(y, nj, p[q]);
          if (j == k + 1) a1[q] = y;
        }
      }
    }
  }
#pragma unroll
  for (int q = 0; q < NR; ++q) {
    p[q] = td_warp_sum(p[q]);
    a1[q] = __shfl_sync(0xffffffffu, a1[q], (k + 1) & 31);
  }
}

__global__ void __launch_bounds__(kTdBigThreads, 1) td_big_kernel(const TdTask *__restrict__ tasks, int smem_slots_max_n, int smem_slots_arg) {
  namespace cg = cooperative_groups;
  cg::cluster_group cluster = cg::this_cluster();
  const TdTask &t = tasks[blockIdx.y];
  const int n = t.n, rank = (int)cluster.block_rank();
  if (n <= 0) return;                       // the whole cluster
  extern __shared__ __align__(16) double tb_sh[];
  double2 *pa = (double2 *)tb_sh;           // [2][n]
  double *vo = tb_sh + 4 * (size_t)n, *wo = vo + n, *vn = wo + n;
  double *rows = tb_sh + td_big_vec_doubles(n);
  __shared__ __align__(16) double red[2][16];
  __shared__ double s_scale, s_b[4];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int slots = (n - rank + kTdCluster - 1) / kTdCluster;     // rows of this CTA
  // shared memory is sized for the largest matrix of the launch: a smaller one gets at least as many of its rows in
  const int all = td_big_slots(n);
  const size_t room = td_big_vec_doubles(smem_slots_max_n) + (size_t)smem_slots_arg * smem_slots_max_n - td_big_vec_doubles(n);
  const int in_smem = (int)min((size_t)all, room / (size_t)n), first = all - in_smem;     // slots >= first are in shared memory
  double *const Rg = t.R;
  auto row_ptr = [&](int s) { return s >= first ? rows + (size_t)(s - first) * n : Rg + (size_t)(s * kTdCluster + rank) * n; };
  if (warp == 0) {
    const int e2 = td_diag_exp(t.A, n, lane);
    if (lane == 0) { s_scale = ldexp(1.0, -e2); if (rank == 0) *t.exp2 = e2; }
  }
  for (int i = tid; i < n; i += kTdBigThreads) { vo[i] = 0.0; wo[i] = 0.0; vn[i] = 0.0; }
  __syncthreads();
  const double sc = 0.5 * s_scale;
  for (int s = warp; s < slots; s += kTdBigThreads / 32) {
    const int i = s * kTdCluster + rank;
    double *r = row_ptr(s);
    for (int j = lane; j < n; j += 32) r[j] = (t.A[(size_t)i * n + j] + t.A[(size_t)j * n + i]) * sc;
  }
  for (int j = tid; j < n; j += kTdBigThreads) pa[j] = make_double2(0.0, (t.A[j] + t.A[(size_t)j * n]) * sc);
  double h = 0.0;
  double *const Vg = t.V, *const dg = t.d, *const eg = t.e, *const hg = t.h;
  cluster.sync();
  for (int k = 0; k < n; ++k) {
    const double2 *cur = pa + (k & 1) * n;
    double2 *nxt = pa + ((k & 1) ^ 1) * n;
    // ---- w of the previous reflector (vn -> vo), column k, the new reflector: redundantly in every CTA
    double dot = 0.0;
    double pj[2], vj[2], aj[2];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int j = tid + u * kTdBigThreads;
      pj[u] = vj[u] = aj[u] = 0.0;
      if (j < n) { const double2 q = cur[j]; pj[u] = j >= k ? q.x : 0.0; aj[u] = q.y; vj[u] = vn[j]; dot = fma(pj[u], vj[u], dot); }
    }
    const double vk = vn[k], pk = cur[k].x;
    dot = td_block_sum(dot, red[0], warp, lane);
    const double K = 0.5 * h * h * dot, wk = fma(h, pk, -K * vk);
    double s = 0.0, c[2];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int j = tid + u * kTdBigThreads;
      const double w = fma(h, pj[u], -K * vj[u]);
      c[u] = fma(-vj[u], wk, fma(-w, vk, aj[u]));
      if (j < n) { vo[j] = vj[u]; wo[j] = w; }
      if (j == k && rank == 0) dg[k] = c[u];
      if (j == k + 1) s_b[k & 1] = c[u];
      if (j > k && j < n) s = fma(c[u], c[u], s);
    }
    if (k == n - 1) break;
    s = td_block_sum(s, red[1], warp, lane);
    const double alpha = s_b[k & 1];
    double beta = alpha, v1 = 0.0;
    h = 0.0;
    const bool live = s > 1e-60;
    if (live) {
      const double nrm = s * rsqrt_pos(s);
      beta = alpha >= 0.0 ? -nrm : nrm;
      v1 = alpha - beta;
      h = 1.0 / fma(nrm, fabs(alpha), s);
    }
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int j = tid + u * kTdBigThreads;
      if (j < n) {
        const double v = !live || j <= k ? 0.0 : (j == k + 1 ? v1 : c[u]);
        vn[j] = v;
        if (rank == (k & 15)) Vg[(size_t)k * n + j] = v;
      }
    }
    if (tid == 0 && rank == 0) { eg[k] = beta; hg[k] = h; }
    __syncthreads();
    // ---- one pass over the rows below k: previous reflector applied, product with the new one
    const int s0 = k + 1 > rank ? (k + 1 - rank + kTdCluster - 1) / kTdCluster : 0;
    const int alive = slots - s0;
    auto pass = [&](auto nr) {
      constexpr int NR = decltype(nr)::value;
      for (int sb = s0 + warp * NR; sb < slots; sb += NR * (kTdBigThreads / 32)) {
        double *rp[NR]; int row[NR]; double p[NR], a1[NR];
#pragma unroll
        for (int q = 0; q < NR; ++q) { const int sl = min(sb + q, slots - 1); row[q] = sl * kTdCluster + rank; rp[q] = row_ptr(sl); }
        if (NR > 1 && sb + NR > slots) {              // the last rows one by one: no row may be updated twice
          for (int q = 0; sb + q < slots; ++q) {
            double *r1[1] = {row_ptr(sb + q)}; const int i1[1] = {(sb + q) * kTdCluster + rank}; double p1[1], b1[1];
            td_big_rows<1>(r1, i1, n, k, vo, wo, vn, lane, p1, b1);
            if (lane < kTdCluster) cluster.map_shared_rank(nxt, lane)[i1[0]] = make_double2(p1[0], b1[0]);
          }
          break;
        }
        td_big_rows<NR>(rp, row, n, k, vo, wo, vn, lane, p, a1);
#pragma unroll
        for (int q = 0; q < NR; ++q)
          if (lane < kTdCluster) cluster.map_shared_rank(nxt, lane)[row[q]] = make_double2(p[q], a1[q]);
      }
    };
    if (alive > 32) pass(std::integral_constant<int, 4>());
    else if (alive > 16) pass(std::integral_constant<int, 2>());
    else pass(std::integral_constant<int, 1>());
    cluster.sync();
  }
  if (tid == 0 && rank == 0) { eg[n - 1] = 0.0; hg[n - 1] = 0.0; }
}

// ---------------------------------------------------------------------------------------------- eigenvalues of T
// LN lanes per eigenvalue count at LN interior points of the current interval per round.  The count is the number of
// sign changes of p_i = (d_i - x) p_{i-1} - e_{i-1}^2 p_{i-2} (one FMA per step on the dependent chain, no division),
// rescaled by a power of two every eight steps.  An exact zero needs no special case as long as no e is zero (the next
// value then has the sign opposite to the one before, one change in either reading), so e^2 is kept above 1e-60 of the
// scaled spectrum; eight steps then stay inside the exponent range.  LN = 32: eleven rounds of 33-fold section, one warp per
// eigenvalue; LN = 8 (n > 256, where the counts fill the machine): seventeen rounds of nine-fold section.
constexpr int kTdValThreads = 128;
template <int LN>
__global__ void __launch_bounds__(kTdValThreads) td_values_kernel(const TdTask *__restrict__ tasks) {
  constexpr int ROUNDS = LN == 32 ? 11 : 17, PER = kTdValThreads / LN;
  const TdTask &t = tasks[blockIdx.y];
  const int n = t.n, j0 = blockIdx.x * PER;
  if (j0 >= n) return;
  extern __shared__ double2 td_de[];        // [n rounded up to 8] (d, -e^2 of the entry before), scaled and centred
  __shared__ double s_lo[4], s_hi[4];
  const int tid = threadIdx.x, lane = tid & 31, n8 = (n + 7) & ~7;
  double lo = 1e300, hi = -1e300;
  bool finite = true;
  for (int i = tid; i < n; i += kTdValThreads) {
    const double r = (i > 0 ? fabs(t.e[i - 1]) : 0.0) + (i + 1 < n ? fabs(t.e[i]) : 0.0), d = t.d[i];
    finite = finite && fabs(d) + r < 1e300;                         // (false for a NaN, which fmin and fmax pass over)
    lo = fmin(lo, d - r); hi = fmax(hi, d + r);
  }
  if (!finite && blockIdx.x == 0 && t.status) atomicOr(t.status, 1);
  for (int o = 16; o; o >>= 1) { lo = fmin(lo, __shfl_xor_sync(0xffffffffu, lo, o)); hi = fmax(hi, __shfl_xor_sync(0xffffffffu, hi, o)); }
  if (lane == 0) { s_lo[tid >> 5] = lo; s_hi[tid >> 5] = hi; }
  __syncthreads();
  lo = fmin(fmin(s_lo[0], s_lo[1]), fmin(s_lo[2], s_lo[3]));
  hi = fmax(fmax(s_hi[0], s_hi[1]), fmax(s_hi[2], s_hi[3]));
  const double mid = 0.5 * (lo + hi), span = fmax(hi - lo, 1e-200);
  int ex; frexp(span, &ex);
  const double sc = ldexp(1.0, -ex), usc = ldexp(1.0, ex);      // the scaled spectrum lies in [-1/2, 1/2]
  for (int i = tid; i < n8; i += kTdValThreads) {
    // padding: decoupled entries at 4, above every point, so they never add to a count (p stays of one sign)
    const double e = i > 0 && i < n ? t.e[i - 1] * sc : 0.0;
    td_de[i] = i < n ? make_double2((t.d[i] - mid) * sc, -fmax(e * e, 1e-60)) : make_double2(4.0, -1e-60);
  }
  __syncthreads();
  // products of the reflectors within a group of four, for td_back_kernel (reflector n - 2 - 4 w - u is number u of group w)
  if (t.U_out)
    for (int w = blockIdx.x * (kTdValThreads / 32) + (tid >> 5); 4 * w < n - 1; w += gridDim.x * (kTdValThreads / 32)) {
      const double *v[4];
      bool ok[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) { const int k = n - 2 - 4 * w - u; ok[u] = k >= 0; v[u] = t.V + (size_t)max(k, 0) * n; }
      double g[6] = {0, 0, 0, 0, 0, 0};
      for (int i = lane; i < n; i += 32) {
        const double a = v[0][i], b = ok[1] ? v[1][i] : 0.0, c = ok[2] ? v[2][i] : 0.0, d = ok[3] ? v[3][i] : 0.0;
        g[0] = fma(a, b, g[0]); g[1] = fma(a, c, g[1]); g[2] = fma(b, c, g[2]);
        g[3] = fma(a, d, g[3]); g[4] = fma(b, d, g[4]); g[5] = fma(c, d, g[5]);
      }
#pragma unroll
      for (int u = 0; u < 6; ++u) { g[u] = td_warp_sum(g[u]); if (lane == u) t.G[6 * w + u] = g[u]; }
    }
  const int sub = tid % LN, j = j0 + tid / LN, m = n - 1 - j;   // j-th largest = m-th smallest
  const unsigned grp = LN == 32 ? 0xffffffffu : ((1u << (LN & 31)) - 1) << (lane & ~(LN - 1) & 31);
  double base = -0.5 - 1e-14, w = 1.0 + 2e-14;
  for (int round = 0; round < ROUNDS; ++round) {
    w *= 1.0 / (LN + 1);
    const double x = fma(w, (double)(sub + 1), base);
    double p = 1.0, pm = 0.0;
    int hp = 0, cnt = 0;
    double2 q[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) q[u] = td_de[u];
    for (int i = 0; i < n8; i += 8) {
      double2 qn[8];
      const int in = i + 8 < n8 ? i + 8 : i;
#pragma unroll
      for (int u = 0; u < 8; ++u) qn[u] = td_de[in + u];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const double pn = fma(q[u].x - x, p, q[u].y * pm);
        const int hn = __double2hiint(pn);
        cnt += (unsigned)(hn ^ hp) >> 31;
        hp = hn; pm = p; p = pn;
      }
      const int e1 = hp & 0x7ff00000, e2 = __double2hiint(pm) & 0x7ff00000;
      const double s = __hiloint2double(0x7fe00000 - max(e1, e2), 0);
      p *= s; pm *= s;
#pragma unroll
      for (int u = 0; u < 8; ++u) q[u] = qn[u];
    }
    const unsigned b = __ballot_sync(0xffffffffu, cnt <= m);
    base = fma(w, (double)__popc(b & grp), base);
  }
  if (sub == 0 && j < n) {
    const double lam = (base + 0.5 * w) * usc + mid;
    t.lam[j] = lam;
    if (t.w_out) {
      const double v = fmax(lam, 0.0) * ldexp(1.0, *t.exp2);
      t.w_out[j] = (float)(t.w_sqrt ? sqrt(v) : v);
      if (!(v < 1e300) && t.status) atomicOr(t.status, 1);
    }
  }
}

// ---------------------------------------------------------------------------------------------- eigenvectors of T
// Two inverse iterations per vector from a pseudo-random start with one LU factorisation (partial pivoting), one thread
// per vector.  The factors sit in shared memory when 32 vectors fit (n <= kTdVecSmemN), else in global scratch;
// consecutive vectors at consecutive addresses either way.
constexpr int kTdVecThreads = 32;
constexpr int kTdVecSmemN = kTdSmallMaxN;
inline size_t td_vec_smem_bytes(int n) {
  return ((size_t)2 * n + (n <= kTdVecSmemN ? (size_t)5 * n * 32 : 0)) * sizeof(double) + (size_t)((n + 31) / 32) * 32 * sizeof(unsigned);
}
template <bool SMEM>
__global__ void __launch_bounds__(kTdVecThreads) td_vectors_kernel(const TdTask *__restrict__ tasks) {
  const TdTask &t = tasks[blockIdx.y];
  const int n = t.n, vec = blockIdx.x * kTdVecThreads + threadIdx.x;
  if (!t.U_out || (int)(blockIdx.x * kTdVecThreads) >= t.r_out) return;
  extern __shared__ double td_sv[];
  double *sd = td_sv, *se = td_sv + n;
  unsigned *swp = (unsigned *)(td_sv + 2 * (size_t)n + (SMEM ? (size_t)5 * n * 32 : 0)) + threadIdx.x;     // [n / 32][32] row swaps
  double anorm = 0.0;
  for (int i = threadIdx.x; i < n; i += kTdVecThreads) {
    sd[i] = t.d[i]; se[i] = i + 1 < n ? t.e[i] : 0.0;
    anorm = fmax(anorm, fabs(sd[i]) + fabs(se[i]));
  }
  for (int o = 16; o; o >>= 1) anorm = fmax(anorm, __shfl_xor_sync(0xffffffffu, anorm, o));
  int ex; frexp(fmax(anorm, 1e-200), &ex);
  const double sc = ldexp(1.0, -ex), tiny = ldexp(1.0, -56);
  __syncwarp();
  for (int i = threadIdx.x; i < n; i += kTdVecThreads) { sd[i] *= sc; se[i] *= sc; }
  __syncwarp();
  if (vec >= t.r_out || vec >= n) return;
  const double lam = t.lam[vec] * sc;
  const size_t ld = SMEM ? 32 : t.ldx, pl = (size_t)n * ld;
  double *ip = SMEM ? td_sv + 2 * (size_t)n + threadIdx.x : t.X + vec;
  double *u1 = ip + pl, *u2 = u1 + pl, *ml = u2 + pl, *y = ml + pl;
  // start vector: a multiplicative hash of (entry, vector), uniform in [-1, 1)
  const uint32_t rb = (uint32_t)mix64(0x7d1ull + (uint64_t)vec);
  auto rnd = [&](int i) { uint32_t z = ((uint32_t)i + rb) * 0x9E3779B1u; z = (z ^ (z >> 15)) * 0x85EBCA77u; return (double)(int32_t)(z ^ (z >> 13)) * 4.656612873077393e-10; };
  // factorisation, the start vector riding along: U (inverse pivot, first and second superdiagonal) and the multipliers
  double b = sd[0] - lam, c = se[0], r = rnd(0);
  unsigned bits = 0;
  for (int i = 0; i < n - 1; ++i) {
    const double sub = se[i], dn = sd[i + 1] - lam, en = se[i + 1], rn = rnd(i + 1);
    const bool swap = fabs(sub) > fabs(b);
    double piv = swap ? sub : b;
    if (fabs(piv) < tiny) piv = piv < 0.0 ? -tiny : tiny;
    const double inv = 1.0 / piv, mlt = (swap ? b : sub) * inv;
    const double U1 = swap ? dn : c, U2 = swap ? en : 0.0;
    b = fma(-mlt, U1, swap ? c : dn); c = fma(-mlt, U2, swap ? 0.0 : en);
    const size_t o = (size_t)i * ld;
    ip[o] = inv; u1[o] = U1; u2[o] = U2; ml[o] = mlt;
    y[o] = r;                               // the start vector is taken as the already transformed right-hand side
    r = rn;
    bits |= (swap ? 1u : 0u) << (i & 31);
    if ((i & 31) == 31) { swp[i & ~31] = bits; bits = 0; }
  }
  swp[(n - 1) & ~31] = bits;
  if (fabs(b) < tiny) b = b < 0.0 ? -tiny : tiny;
  const double ib = 1.0 / b;
  double s_in = 1.0;
  constexpr int P = 8;                      // entries requested ahead of their use
  for (int it = 0; it < 2; ++it) {
    if (it) {                               // forward substitution of the first iterate with the stored multipliers
      r = y[0] * s_in;
      double ym[P], mm[P];
#pragma unroll
      for (int u = 0; u < P; ++u) { const size_t o = (size_t)min(u, n - 1) * ld; mm[u] = ml[o]; ym[u] = y[(size_t)min(u + 1, n - 1) * ld]; }
      unsigned bw = 0;
      for (int i0 = 0; i0 < n - 1; i0 += P) {
        double yc[P], mc[P];
#pragma unroll
        for (int u = 0; u < P; ++u) { yc[u] = ym[u] * s_in; mc[u] = mm[u]; }
#pragma unroll
        for (int u = 0; u < P; ++u) {
          const int i = i0 + P + u;
          mm[u] = ml[(size_t)min(i, n - 1) * ld]; ym[u] = y[(size_t)min(i + 1, n - 1) * ld];
        }
        if ((i0 & 31) == 0) bw = swp[i0];
#pragma unroll
        for (int u = 0; u < P; ++u) {
          const int i = i0 + u;
          if (i < n - 1) {
            const bool swap = (bw >> (i & 31)) & 1u;
            const double yi = swap ? yc[u] : r, x3 = swap ? r : yc[u];
            y[(size_t)i * ld] = yi;
            r = fma(-mc[u], yi, x3);
          }
        }
      }
    }
    double x1 = r * ib, x2 = 0.0, norm2 = x1 * x1;
    y[(size_t)(n - 1) * ld] = x1;
    double pi[P], p1[P], p2[P], py[P];
    auto fetch = [&](int itop) {
#pragma unroll
      for (int u = 0; u < P; ++u) {
        const size_t o = (size_t)max(itop - u, 0) * ld;
        pi[u] = ip[o]; p1[u] = u1[o]; p2[u] = u2[o]; py[u] = y[o];
      }
    };
    fetch(n - 2);
    for (int i0 = n - 2; i0 >= 0; i0 -= P) {
      double qi[P], q1[P], q2[P], qy[P];
#pragma unroll
      for (int u = 0; u < P; ++u) { qi[u] = pi[u]; q1[u] = -p1[u] * pi[u]; q2[u] = -p2[u] * pi[u]; qy[u] = py[u] * pi[u]; }
      if (i0 >= P) fetch(i0 - P);
#pragma unroll
      for (int u = 0; u < P; ++u) {
        if (i0 - u >= 0) {
          const double x = fma(q1[u], x1, fma(q2[u], x2, qy[u]));
          y[(size_t)(i0 - u) * ld] = x;
          norm2 = fma(x, x, norm2);
          x2 = x1; x1 = x;
        }
      }
    }
    s_in = norm2 > 0.0 && norm2 < 1e300 ? rsqrt(norm2) : 0.0;
  }
  if (SMEM) {
    double *Y = t.X + 4 * (size_t)n * t.ldx + vec;
    for (int i = 0; i < n; ++i) Y[(size_t)i * t.ldx] = y[(size_t)i * ld];
  }
  t.xn[vec] = s_in;
  if (!(s_in > 0.0) && t.status) atomicOr(t.status, 1);
}

// Members of a cluster are orthogonalised against each other (classical Gram-Schmidt, twice); one CTA per matrix,
// nothing to do for most matrices.
constexpr int kTdOrthThreads = 512;
__global__ void __launch_bounds__(kTdOrthThreads) td_orth_kernel(const TdTask *__restrict__ tasks) {
  constexpr int NW = kTdOrthThreads / 32;
  const TdTask &t = tasks[blockIdx.x];
  const int n = t.n, r = min(t.r_out, n), ldx = t.ldx;
  if (!t.U_out) return;
  extern __shared__ double td_so[];          // [n] vector, [r] coefficients
  double *x = td_so, *cf = td_so + n;
  __shared__ double s_red[NW], part[NW][32];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  double anorm = 0.0;
  for (int i = tid; i < n; i += kTdOrthThreads) anorm = fmax(anorm, fabs(t.d[i]) + fabs(t.e[i]));
  for (int o = 16; o; o >>= 1) anorm = fmax(anorm, __shfl_xor_sync(0xffffffffu, anorm, o));
  if (lane == 0) s_red[warp] = anorm;
  __syncthreads();
  for (int w = 0; w < NW; ++w) anorm = fmax(anorm, s_red[w]);
  const double gap = fmax(kTdClusterGap * anorm, 1e-150);
  double *Y = t.X + 4 * (size_t)n * ldx;
  int any = 0;
  for (int j = tid + 1; j < r; j += kTdOrthThreads) any |= t.lam[j - 1] - t.lam[j] <= gap;
  if (!__syncthreads_or(any)) return;
  int c0 = 0;
  for (int j = 1; j < r; ++j) {
    if (t.lam[j - 1] - t.lam[j] > gap) { c0 = j; continue; }
    const double s0 = t.xn[j];
    for (int i = tid; i < n; i += kTdOrthThreads) x[i] = Y[(size_t)i * ldx + j] * s0;
    __syncthreads();
    double nrm = 1.0;
    for (int pass = 0; pass < 2; ++pass) {
      // coefficients of 32 neighbouring vectors at a time: the rows are split over the warps (the loads run along the
      // vectors), the partial sums are added in a fixed order
      for (int q0 = c0; q0 < j; q0 += 32) {
        const int q = q0 + lane;
        double a0 = 0.0, a1 = 0.0;
        if (q < j) {
          int i = warp;
          for (; i + NW < n; i += 2 * NW) { a0 = fma(Y[(size_t)i * ldx + q], x[i], a0); a1 = fma(Y[(size_t)(i + NW) * ldx + q], x[i + NW], a1); }
          if (i < n) a0 = fma(Y[(size_t)i * ldx + q], x[i], a0);
        }
        part[warp][lane] = a0 + a1;
        __syncthreads();
        if (warp == 0 && q < j) {
          double a = 0.0;
          for (int w = 0; w < NW; ++w) a += part[w][lane];
          const double xq = t.xn[q];
          cf[q] = a * xq * xq;
        }
        __syncthreads();
      }
      double s = 0.0;
      for (int i = warp; i < n; i += NW) {
        double v = 0.0;
        for (int q = c0 + lane; q < j; q += 32) v = fma(cf[q], Y[(size_t)i * ldx + q], v);
        v = td_warp_sum(v);
        if (lane == 0) { const double u = x[i] - v; x[i] = u; s = fma(u, u, s); }
      }
      if (lane == 0) s_red[warp] = s;
      __syncthreads();
      s = 0.0;
      for (int w = 0; w < NW; ++w) s += s_red[w];
      nrm = s > 0.0 ? rsqrt(s) : 0.0;
      for (int i = tid; i < n; i += kTdOrthThreads) x[i] *= nrm;
      __syncthreads();
    }
    for (int i = tid; i < n; i += kTdOrthThreads) Y[(size_t)i * ldx + j] = x[i];
    if (tid == 0) t.xn[j] = 1.0;
    if (!(nrm > 0.0) && tid == 0 && t.status) atomicOr(t.status, 1);
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------------------------- U = H_0 H_1 ... Z
// A warp owns NV vectors (rows cyclic over the lanes, RA rows per lane).  Reflectors are staged in shared memory, the
// next stage in flight, and applied four at a time: the four dot products with the same vector are independent once the
// six products between the reflectors are known (td_values_kernel forms them), so a step of the chain serves four of them.
constexpr int kTdBackThreads = 128;
__device__ __forceinline__ void td_cp8(void *dst, const void *src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
template <int ST> inline size_t td_back_smem_bytes(int n) { return (2 * (size_t)ST * (n + 1) + 6 * (size_t)((n + 3) / 4)) * sizeof(double); }

template <int RA, int NV, int ST>
__global__ void __launch_bounds__(kTdBackThreads) td_back_kernel(const TdTask *__restrict__ tasks) {
  const TdTask &t = tasks[blockIdx.y];
  const int n = t.n, r = min(t.r_out, n), ldx = t.ldx;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (!t.U_out || (int)blockIdx.x * (kTdBackThreads / 32) * NV >= r) return;
  const int v0 = (blockIdx.x * (kTdBackThreads / 32) + warp) * NV;
  extern __shared__ double td_sb[];         // [2][ST][n], [2][ST]
  double *s_h = td_sb + 2 * (size_t)ST * n, *s_g = s_h + 2 * ST;     // [2][ST], products of every group
  for (int e = tid; e < 6 * ((n + 2) / 4); e += kTdBackThreads) s_g[e] = t.G[e];
  const double *Vg = t.V, *hg = t.h;
  // stage: slot u holds reflector k1 - 1 - u (the order they are applied in); missing ones have h = 0 and are zero
  auto stage = [&](int k1, int buf) {
    if (k1 > 0) {
      double *dst = td_sb + (size_t)buf * ST * n;
      for (int u = 0; u < ST; ++u) {
        const int k = k1 - 1 - u;
        if (k >= 0) { for (int e = tid; e < n; e += kTdBackThreads) td_cp8(dst + (size_t)u * n + e, Vg + (size_t)k * n + e); }
        else for (int e = tid; e < n; e += kTdBackThreads) dst[(size_t)u * n + e] = 0.0;
      }
      if (tid < ST) { const int k = k1 - 1 - tid; if (k >= 0) td_cp8(s_h + buf * ST + tid, hg + k); else s_h[buf * ST + tid] = 0.0; }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  stage(n - 1, 0);
  const double *Y = t.X + 4 * (size_t)n * ldx;
  double z[RA][NV];
#pragma unroll
  for (int q = 0; q < NV; ++q) {
    const double s = v0 + q < r ? t.xn[v0 + q] : 0.0;
#pragma unroll
    for (int a = 0; a < RA; ++a) {
      const int i = lane + 32 * a;
      z[a][q] = (i < n && v0 + q < r) ? Y[(size_t)i * ldx + v0 + q] * s : 0.0;
    }
  }
  int buf = 0;
  for (int k1 = n - 1; k1 > 0; k1 -= ST, buf ^= 1) {
    stage(k1 - ST, buf ^ 1);
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    __syncthreads();
    const double *sv = td_sb + (size_t)buf * ST * n;
    for (int w = 0; w < ST / 4; ++w) {
      const int kmin = max(0, k1 - 4 * w - 4);         // entries at or below kmin of all four reflectors are zero
      if (k1 - 4 * w <= 0) break;
      const double *v = sv + (size_t)w * 4 * n;
      double dot[4 * NV];
#pragma unroll
      for (int u = 0; u < 4 * NV; ++u) dot[u] = 0.0;
#pragma unroll
      for (int a = 0; a < RA; ++a) {
        if (32 * a + 31 > kmin && lane + 32 * a < n) {
          const double *va = v + lane + 32 * a;
          const double x0 = va[0], x1 = va[n], x2 = va[2 * n], x3 = va[3 * n];
#pragma unroll
          for (int q = 0; q < NV; ++q) {
            dot[4 * q] = fma(x0, z[a][q], dot[4 * q]); dot[4 * q + 1] = fma(x1, z[a][q], dot[4 * q + 1]);
            dot[4 * q + 2] = fma(x2, z[a][q], dot[4 * q + 2]); dot[4 * q + 3] = fma(x3, z[a][q], dot[4 * q + 3]);
          }
        }
      }
      const double mine = td_red<4 * NV>(dot, lane);        // this lane's of the 4 NV sums; index bits sit in the top lane bits
      const double *hs = s_h + buf * ST + 4 * w, *g = s_g + 6 * ((n - 1 - k1) / 4 + w);
      double m[4][NV];
#pragma unroll
      for (int q = 0; q < NV; ++q) {
        double d[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          constexpr int SH = 32 / (4 * NV);
          d[u] = __shfl_sync(0xffffffffu, mine, (4 * q + u) * SH);
        }
        m[0][q] = -hs[0] * d[0];
        m[1][q] = -hs[1] * fma(m[0][q], g[0], d[1]);
        m[2][q] = -hs[2] * fma(m[1][q], g[2], fma(m[0][q], g[1], d[2]));
        m[3][q] = -hs[3] * fma(m[2][q], g[5], fma(m[1][q], g[4], fma(m[0][q], g[3], d[3])));
      }
#pragma unroll
      for (int a = 0; a < RA; ++a) {
        if (32 * a + 31 > kmin && lane + 32 * a < n) {
          const double *va = v + lane + 32 * a;
          const double x0 = va[0], x1 = va[n], x2 = va[2 * n], x3 = va[3 * n];
#pragma unroll
          for (int q = 0; q < NV; ++q)
            z[a][q] = fma(m[3][q], x3, fma(m[2][q], x2, fma(m[1][q], x1, fma(m[0][q], x0, z[a][q]))));
        }
      }
    }
    __syncthreads();
  }
#pragma unroll
  for (int a = 0; a < RA; ++a) {
    const int i = lane + 32 * a;
    if (i < n)
#pragma unroll
      for (int q = 0; q < NV; ++q)
        if (v0 + q < r) t.U_out[(size_t)i * t.ld_out + v0 + q] = (float)z[a][q];
  }
}

// ---------------------------------------------------------------------------------------------- host
inline void td_opt_in() {
  static DeviceOnce once;
  once([] {
    const int lim = (int)(kSmemOptIn - 1024);
    cudaFuncSetAttribute(td_small_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
    cudaFuncSetAttribute(td_big_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
    cudaFuncSetAttribute(td_big_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    cudaFuncSetAttribute(td_vectors_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
    cudaFuncSetAttribute(td_vectors_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
    cudaFuncSetAttribute(td_orth_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 64 * 1024);
    cudaFuncSetAttribute(td_back_kernel<5, 2, 16>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
    cudaFuncSetAttribute(td_back_kernel<9, 2, 16>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
    cudaFuncSetAttribute(td_back_kernel<17, 1, 8>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
    cudaFuncSetAttribute(td_back_kernel<32, 1, 8>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
  });
}

// All tasks of one launch chain: n <= kTdSmallMaxN for every one, or kTdSmallMaxN < n <= kTdMaxN for every one.
// max_r = 0: no vectors.  Returns the number of launches.
inline int td_launch(const TdTask *d_tasks, int count, int max_n, int max_r, cudaStream_t s) {
  td_opt_in();
  int launches = 2;
  if (max_n <= kTdSmallMaxN) td_small_kernel<<<count, kTdSmallThreads, td_small_smem_bytes(max_n), s>>>(d_tasks);
  else {
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof cfg);
    cfg.gridDim = dim3(kTdCluster, count); cfg.blockDim = dim3(kTdBigThreads); cfg.dynamicSmemBytes = td_big_smem_bytes(max_n); cfg.stream = s;
    cudaLaunchAttribute at;
    memset(&at, 0, sizeof at);
    at.id = cudaLaunchAttributeClusterDimension; at.val.clusterDim.x = kTdCluster; at.val.clusterDim.y = 1; at.val.clusterDim.z = 1;
    cfg.attrs = &at; cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, td_big_kernel, d_tasks, max_n, td_big_smem_slots(max_n));
  }
  const size_t vsm = (size_t)((max_n + 7) & ~7) * sizeof(double2);
  if (max_n <= 256) td_values_kernel<32><<<dim3((max_n + 3) / 4, count), kTdValThreads, vsm, s>>>(d_tasks);
  else td_values_kernel<8><<<dim3((max_n + 15) / 16, count), kTdValThreads, vsm, s>>>(d_tasks);
  if (max_r > 0) {
    const dim3 vg((max_r + 31) / 32, count);
    if (max_n <= kTdVecSmemN) td_vectors_kernel<true><<<vg, kTdVecThreads, td_vec_smem_bytes(max_n), s>>>(d_tasks);
    else td_vectors_kernel<false><<<vg, kTdVecThreads, td_vec_smem_bytes(max_n), s>>>(d_tasks);
    td_orth_kernel<<<count, kTdOrthThreads, (size_t)(max_n + max_r) * sizeof(double), s>>>(d_tasks);
    if (max_n <= 160) td_back_kernel<5, 2, 16><<<dim3((max_r + 7) / 8, count), kTdBackThreads, td_back_smem_bytes<16>(max_n), s>>>(d_tasks);
    else if (max_n <= 288) td_back_kernel<9, 2, 16><<<dim3((max_r + 7) / 8, count), kTdBackThreads, td_back_smem_bytes<16>(max_n), s>>>(d_tasks);
    else if (max_n <= 544) td_back_kernel<17, 1, 8><<<dim3((max_r + 3) / 4, count), kTdBackThreads, td_back_smem_bytes<8>(max_n), s>>>(d_tasks);
    else td_back_kernel<32, 1, 8><<<dim3((max_r + 3) / 4, count), kTdBackThreads, td_back_smem_bytes<8>(max_n), s>>>(d_tasks);
    launches += 3;
  }
  return launches;
}

}  // namespace jolt
