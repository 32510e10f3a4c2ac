// CholeskyQR of the randomized range finder (Sec. 5; Q = orth(S)) on tensor cores.  The basis (T x k on the token
// side, m*128 x k on the feature side) lives as an fp16 hi + lo pair, transposed in panels: [panels][kp][rows per
// panel] (1 x T on the token side, m x 128 on the feature side) -- the layout the sweeps read their dense operand in.
//
//   orth_gram_kernel    G = R^T R             tcgen05, both MMA operands are the same K-major tile; hi hi + hi lo + lo hi
//   cholinv_kernel      G = L L^T, L^-1       fp64, one CTA per cell (shared memory), L^-1 written as fp16 hi + lo
//   orth_apply_kernel   Q = R L^-T            tcgen05 (A = R^T tile, MN-major; B = L^-1, K-major); writes Q as fp32 rows
//                                             and, in place, as the hi + lo operand of the next sweep
//
// Precision: fp16 products are exact in the fp32 accumulator and hi + lo carries 22 bits, so G is fp32-grade.  The
// accumulator of tcgen05.mma truncates (about 2^-24 of the running sum per MMA), so the Gram kernel flushes it after
// every 64 rows into fp32 registers of the epilogue threads (round-to-nearest adds) and the row chunks of a cell are
// added in fp64 by the Cholesky kernel.
#pragma once
#include "small_solvers.cuh"
#include "tc_common.cuh"

namespace jolt {
namespace tc {

constexpr int OR_MAX_KP = 160;            // D0 (128 x kp) and D1 (rows 128.. x kp - 128), double buffered, fit 512 columns
constexpr int OR_MAX_K = 152;             // the fp64 Cholesky work matrix stays in shared memory
constexpr int OR_THREADS = 192;           // warps 0-3 epilogue, warp 4 TMA, warp 5 MMA
constexpr int OR_STEPS_PER_CTA = 8;       // 64-row steps per Gram CTA
constexpr int OR_SMEM_LIMIT = 222 * 1024;

struct alignas(64) OrthCell {
  CUtensorMap tmHi, tmLo;     // basis [panels][kp][rpp] fp16: dims {rpp, kp, panels}, box {64, kp, 1}
  CUtensorMap tmLhi, tmLlo;   // L^-1 [kp][kp] fp16 (row c, column j): dims {kp, kp}, box {64, kp}
  float *part;                // Gram partials [n_chunks][kp][kp] (rows >= 128 hold columns >= 128 only)
  __half *Lhi, *Llo;          // L^-1 as written by cholinv_kernel, scaled by 2^l_exp
  int *l_exp;
  float *out32;               // apply: rows x ld fp32 (row = panel * rpp + row in panel), may be null
  int ld, k, kp;
  int rpp, panels;
  int n_chunks;
  int out_exp;                // the fp16 copy of Q is scaled by 2^out_exp
  int *status;
};

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float *v) {
  uint32_t *u = (uint32_t *)v;
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(u[0]), "=r"(u[1]), "=r"(u[2]), "=r"(u[3]), "=r"(u[4]), "=r"(u[5]), "=r"(u[6]), "=r"(u[7]), "=r"(u[8]),
        "=r"(u[9]), "=r"(u[10]), "=r"(u[11]), "=r"(u[12]), "=r"(u[13]), "=r"(u[14]), "=r"(u[15])
      : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tma_store_3d(const void *tmap, uint32_t src, int c0, int c1, int c2) {
  asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.bulk_group [%0, {%2, %3, %4}], [%1];"
               ::"l"(tmap), "r"(src), "r"(c0), "r"(c1), "r"(c2) : "memory");
}
__device__ __forceinline__ void tma_store_commit_wait() {
  asm volatile("cp.async.bulk.commit_group;" ::: "memory");
  asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
}

// ---------------------------------------------------------------------------------------------- Gram
__global__ void __launch_bounds__(OR_THREADS, 1) orth_gram_kernel(const OrthCell *__restrict__ cells, int n_stages) {
  extern __shared__ unsigned char smem_raw[];
  const OrthCell &c = cells[blockIdx.y];
  if ((int)blockIdx.x >= c.n_chunks) return;
  const int spp = c.rpp / 64;                         // 64-row steps per panel
  const int total = c.panels * spp;
  const int s0 = blockIdx.x * OR_STEPS_PER_CTA, n_steps = min(OR_STEPS_PER_CTA, total - s0);
  const int kp = c.kp, n1 = kp > 128 ? kp - 128 : 0, n0 = kp > 128 ? 128 : kp;     // D0: rows 0..n0-1 (M = 128), D1: rows 128..

  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  unsigned char *sm = smem_raw + (base - raw);
  const uint32_t tile = (uint32_t)kp * 128u;           // kp is a multiple of 16: a multiple of 2 KB
  const uint32_t stage_bytes = 2 * tile;
  // a 128-row A operand starting at row 128 of the last tile reads up to 16 KB past it: the slack below
  const uint32_t sBar = base + (uint32_t)n_stages * stage_bytes + 16384u;
  volatile int *abort_flag = (volatile int *)(sm + (size_t)n_stages * stage_bytes + 16384 + 256);
  uint32_t *tmem_slot = (uint32_t *)(sm + (size_t)n_stages * stage_bytes + 16384 + 264);
  auto bFull = [=](int s) { return sBar + 8 * s; };
  auto bEmpty = [=](int s) { return sBar + 64 + 8 * s; };
  auto bAfull = [=](int b) { return sBar + 128 + 8 * b; };
  auto bAempty = [=](int b) { return sBar + 144 + 8 * b; };

  const int warp = warp_uniform(), lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    *abort_flag = 0;
    for (int s = 0; s < 8; ++s) { mbar_init(bFull(s), 1); mbar_init(bEmpty(s), 1); }
    for (int b = 0; b < 2; ++b) { mbar_init(bAfull(b), 1); mbar_init(bAempty(b), 128); }
    fence_barrier_init();
  }
  if (warp == 4) { tmem_alloc(smem_u32(tmem_slot), 512); tmem_relinquish(); }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  if (warp == 4 && lane == 0) {
    tma_prefetch_desc(&c.tmHi); tma_prefetch_desc(&c.tmLo);
    bool ok = true;
    for (int j = 0; ok && j < n_steps; ++j) {
      const int s = j % n_stages, n = j / n_stages;
      ok = mbar_wait(bEmpty(s), (n & 1) ^ 1, abort_flag);
      if (!ok) break;
      const int step = s0 + j, panel = step / spp, r0 = (step - panel * spp) * 64;
      const uint32_t st = base + s * stage_bytes;
      mbar_expect_tx(bFull(s), 2 * tile);
      tma_load_3d(st, &c.tmHi, bFull(s), r0, 0, panel);
      tma_load_3d(st + tile, &c.tmLo, bFull(s), r0, 0, panel);
    }
  } else if (warp == 5) {
    const uint32_t id0 = umma_idesc_f16(128, kp, 0, 0);
    const uint32_t id1 = umma_idesc_f16(128, n1 > 0 ? n1 : 16, 0, 0);
    bool ok = true;
    for (int j = 0; ok && j < n_steps; ++j) {
      const int s = j % n_stages, n = j / n_stages, b = j & 1, nb = j >> 1;
      ok = mbar_wait_warp(bFull(s), n & 1, abort_flag);
      if (ok) ok = mbar_wait_warp(bAempty(b), (nb & 1) ^ 1, abort_flag);
      if (!ok) break;
      tc_fence_after();
      const uint32_t hi = base + s * stage_bytes, lo = hi + tile;
      const uint32_t d0 = tmem_base + b * 256, d1 = d0 + 160;
#pragma unroll
      for (int k4 = 0; k4 < 4; ++k4) {
        const uint64_t aH = umma_desc_sw128(hi + k4 * 32, 16, 1024), aL = umma_desc_sw128(lo + k4 * 32, 16, 1024);
        umma_f16(d0, aH, aH, id0, k4 != 0);
        umma_f16(d0, aH, aL, id0, 1);
        umma_f16(d0, aL, aH, id0, 1);
        if (n1 > 0) {
          const uint64_t a1H = umma_desc_sw128(hi + 16384 + k4 * 32, 16, 1024), a1L = umma_desc_sw128(lo + 16384 + k4 * 32, 16, 1024);
          umma_f16(d1, a1H, a1H, id1, k4 != 0);
          umma_f16(d1, a1H, a1L, id1, 1);
          umma_f16(d1, a1L, a1H, id1, 1);
        }
      }
      umma_commit(bEmpty(s));
      umma_commit(bAfull(b));
    }
  } else if (warp < 4) {
    float acc0[OR_MAX_KP], acc1[32];
#pragma unroll
    for (int i = 0; i < OR_MAX_KP; ++i) acc0[i] = 0.f;
#pragma unroll
    for (int i = 0; i < 32; ++i) acc1[i] = 0.f;
    const uint32_t t_lane = tmem_base + ((uint32_t)(warp * 32) << 16);
    bool ok = true;
    for (int j = 0; j < n_steps; ++j) {
      const int b = j & 1, nb = j >> 1;
      if (ok) ok = __all_sync(0xffffffffu, mbar_wait(bAfull(b), nb & 1, abort_flag));
      if (!ok) break;
      tc_fence_after();
#pragma unroll
      for (int ch = 0; ch < OR_MAX_KP / 16; ++ch) {
        if (ch * 16 < kp) {
          float v[16];
          tmem_ld16(t_lane + b * 256 + ch * 16, v);
          tmem_wait_ld();
#pragma unroll
          for (int i = 0; i < 16; ++i) acc0[ch * 16 + i] += v[i];
        }
      }
      if (warp == 0) {
#pragma unroll
        for (int ch = 0; ch < 2; ++ch) {
          if (ch * 16 < n1) {
            float v[16];
            tmem_ld16(t_lane + b * 256 + 160 + ch * 16, v);
            tmem_wait_ld();
#pragma unroll
            for (int i = 0; i < 16; ++i) acc1[ch * 16 + i] += v[i];
          }
        }
      }
      tc_fence_before();
      mbar_arrive(bAempty(b));
    }
    if (ok) {
      const int row = warp * 32 + lane;
      float *out = c.part + (size_t)blockIdx.x * kp * kp;
      if (row < n0) {
#pragma unroll
        for (int i = 0; i < OR_MAX_KP; ++i)
          if (i < kp) out[(size_t)row * kp + i] = acc0[i];
      }
      if (warp == 0 && lane < n1) {
#pragma unroll
        for (int i = 0; i < 32; ++i)
          if (i < n1) out[(size_t)(128 + lane) * kp + 128 + i] = acc1[i];
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (*abort_flag) {
    if (threadIdx.x == 0) atomicOr(c.status, 8);
    const long long t0 = clock64();
    while (clock64() - t0 < 2000000) {}
    __syncthreads();
  }
  if (warp == 4) { tc_fence_after(); tmem_dealloc(tmem_base, 512); }
}

// ---------------------------------------------------------------------------------------------- Cholesky + inverse
// G = L L^T in fp64, one CTA per matrix, right-looking by panels of 8 columns, with X = L^-T formed by the same
// panel operations on the rows of an identity appended below G ([G; I] = [L; X] L^T).
//
// 8 x 8 tiles in shared memory, row by row of the lower triangle, the updates on fp64 matrix instructions.  Tile
// (I, J), I >= J, of the Schur complement is finished when panel J is, and exactly then the tile (J, I) of X comes to life, so
// one place serves both, and the living tiles of panel p are all those of the rows I > p.  Tiles hold the negative of the matrix.
// An accumulator's two registers of a lane are entries 2 c and 2 c + 1 of row r (lane = 4 r + c), 16 bytes of the row-major tile; the pairs
// of rows 2 i and 2 i + 1 are stored exchanged by i (pair c in place c ^ i), so that a lane per row reads its eight entries without
// bank conflicts too.  The solved panel is kept as pairs (c, c + 4): the operand of two k = 4 instructions, columns 0 .. 3 and 4 .. 7.
// Warp 0 owns the chain: it brings the next 8 x 8 diagonal block up to date and factors it (L D L^T in registers, every lane the whole
// block) while twelve others update.  The rest of its quarter of the SM stays idle: a product there takes the fp64
// pipe for 16 cycles, and the chain's dependent operations queue behind them.  Panel p, two barriers:
//   solve    a thread per row, substitution against the block: rows of L below it, final rows of X above it; published
//   update   every living tile but the next diagonal block; its eight products are summed first and then subtracted
// The order of the operations is that of a matrix in shared memory updated by FMAs, one rounding each (the matrix instruction is four
// FMAs in the order of k, the reciprocal is correctly rounded), and so are the results, bit for bit.  Multiplying the panel by the explicit inverse
// of the block instead is 6 us shorter at n = 138 but not as good: the residual of L L^T in units of 2^-53 of the diagonal, 1081 against 3.2
// where neighbouring columns are close (n = 74), 7.6 against 4.1 on a graded matrix.
// What bounds it: fp64 operations and their latency: the chain, 8 x (estimate, five FMAs, product, FMA) and the substitution, and
// at n > 100 the products of the early panels.  The loops are short on purpose: nothing runs more than a few times, and with tiles in
// registers (unrolled bodies, 40 KB of code) the fetch of the instructions took as long as all the rest.  One matrix of n = 138 / 74 / 26 alone:
// 53 / 22 / 10 us, the same from 32 partial Grams 78 / 29 / 11 us; updates by FMAs (two passes over the matrix every eight
// columns) 78 / 34 / 15 and 103 / 43 / 19 us.
// A pivot not above `dead_rel` of its original diagonal entry belongs to a direction that is dependent to working
// accuracy: its column of L and its row / column of L^-1 are zero, status bit 1.
// Input: fp32 row-chunk partials of the Gram kernel (summed here in fp64) or an fp64 matrix.  Output: L^-1 as fp16
// hi + lo (times 2^l_exp) and / or L itself in fp64 for the Jacobi kernel.
struct CholInvTask {
  const float *part; int n_chunks, kp;      // Gram partials [n_chunks][kp][kp] (rows >= 128 hold columns >= 128 only), or
  const double *A64;                        // n x n symmetric fp64
  int k;
  __half *Lhi, *Llo;        // optional: L^-1 [kp][kp], rows / columns >= k zero
  int *l_exp;               // L^-1 is stored times 2^l_exp
  double *L64;              // optional: L column-major n x n, zeros above the diagonal, followed by one double holding
                            // the exponent e with max |L| < 2^e
  int *status;
  double dead_rel;
};
constexpr int kCholInvThreads = 512;
constexpr int kCholInvMaxN = 152;
constexpr int kCholInvRows = kCholInvMaxN / 8;      // block rows
constexpr int kCholInvWorkers = 12;
inline size_t cholinv_smem_bytes(int k) {
  const size_t nt = (k + 7) / 8;
  return ((nt * (nt + 1) / 2 + kCholInvRows + 2) * 64 + 8 + kCholInvMaxN) * sizeof(double);
}

// 1 / d, correctly rounded, for 2^-1000 < d < 2^1000: the hardware's estimate (relative error e of 2^-20 or less), one third-order step,
// 1 / d = y / (1 - e) = y (1 + e + e^2 + ..), which is good to a unit in the last place, and one of Newton's, which rounds such a number
// correctly (Markstein 1990; all ones in d's fraction excepted).
__device__ __forceinline__ double rcp_pos(double d) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(d));
  double e = fma(-d, y, 1.0);
  y = fma(y, fma(e, e, e), y);
  e = fma(-d, y, 1.0);
  return fma(y, e, y);
}

__global__ void __launch_bounds__(kCholInvThreads, 1) cholinv_kernel(const CholInvTask *__restrict__ tasks) {
  const CholInvTask t = tasks[blockIdx.x];
  const int n = t.k, kp = t.kp, NT = (n + 7) >> 3, n_tiles = NT * (NT + 1) / 2;
  if (n <= 0) return;
  extern __shared__ __align__(16) double ci_sh[];
  double2 *tile = (double2 *)ci_sh;                      // [tile][row][pair of columns]; finished tiles (J, I) of X stay here
  double2 *pan = tile + n_tiles * 32;                    // [row][pair c, c + 4] the solved panel
  double *blk = (double *)(pan + kCholInvRows * 32);     // [8][8] the next diagonal block, and its factor
  double *lb = blk + 64, *ipiv = lb + 64;                // ... 1 / L_qq (0 for a dead pivot)
  double *diag0 = ipiv + 8;                              // original diagonal
  __shared__ int s_red[kCholInvThreads / 32], s_dead;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, r = lane >> 2, c = lane & 3;
  const int at_lane = lane ^ (lane >> 3);                // pair c of row r of a tile
  constexpr int NW = kCholInvThreads / 32;
  auto row_start = [](int I) { return I * (I + 1) / 2; };
  if (tid == 0) s_dead = 0;
  {
    int I = 0, J = warp;
    for (int q = warp; q < n_tiles; q += NW, J += NW) {
      while (J > I) { J -= I + 1; ++I; }
      double v[2] = {0.0, 0.0};
      int at[2];
#pragma unroll
      for (int e = 0; e < 2; ++e) {                      // entry (row, column) with row <= column: stored for every such pair
        const int i = 8 * I + r, j = 8 * J + 2 * c + e, lo = min(i, j), hi = max(i, j);
        at[e] = hi < n ? lo * (t.A64 ? n : kp) + hi : -1;
      }
      if (t.A64) {
#pragma unroll
        for (int e = 0; e < 2; ++e) if (at[e] >= 0) v[e] = t.A64[at[e]];
      } else {
        const float *p = t.part;
        const int cs = kp * kp;
#pragma unroll 1
        for (int ch = 0; ch < t.n_chunks; ch += 8, p += 8 * cs) {
          float x[2][8];
#pragma unroll
          for (int e = 0; e < 2; ++e)
#pragma unroll
            for (int u = 0; u < 8; ++u) x[e][u] = at[e] >= 0 && ch + u < t.n_chunks ? __ldg(p + u * cs + at[e]) : 0.f;
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            const double x0 = x[e][0], x1 = x[e][1], x2 = x[e][2], x3 = x[e][3], x4 = x[e][4], x5 = x[e][5], x6 = x[e][6], x7 = x[e][7];
            if (ch + 8 <= t.n_chunks) v[e] += ((x0 + x1) + (x2 + x3)) + ((x4 + x5) + (x6 + x7));
            else v[e] = ((((((v[e] + x0) + x1) + x2) + x3) + x4) + x5) + x6;
          }
        }
      }
      tile[q * 32 + at_lane] = make_double2(-v[0], -v[1]);
      if (I == J) {
        if (2 * c == r) diag0[8 * I + r] = v[0];
        if (2 * c + 1 == r) diag0[8 * I + r] = v[1];
      }
    }
  }
  __syncthreads();
  int mxh = 0;                                           // largest |X| so far: the high word of its fp64
  if (warp & 3) {
    const int wi = 3 * (warp >> 2) + (warp & 3) - 1;
#pragma unroll 1
    for (int p = 0; p < NT; ++p) {
      __syncthreads();                                   // A: the block is factored
      const int i = wi * 32 + lane, b = i >> 3, rr = i & 7, s2 = rr >> 1;
      if (b < NT) {                                      // x_j = (p_j - sum_{l<j} x_l L_jl) / L_jj
        const bool below = b > p;
        double2 *w = tile + (below ? row_start(b) + p : row_start(p) + b) * 32 + rr * 4;
        double x[8];
#pragma unroll
        for (int j = 0; j < 4; ++j) { const double2 q = w[j ^ s2]; x[2 * j] = -q.x; x[2 * j + 1] = -q.y; }
        if (b == p) {
#pragma unroll
          for (int j = 0; j < 8; ++j) x[j] = j == rr ? 1.0 : 0.0;
        }
        double2 f[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) f[j] = ((const double2 *)ipiv)[j];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
#pragma unroll
          for (int l = 0; l < j; l += 2) {
            const double2 q = ((const double2 *)lb)[4 * j + (l >> 1)];
            x[j] = fma(-x[l], q.x, x[j]);
            if (l + 1 < j) x[j] = fma(-x[l + 1], q.y, x[j]);
          }
          x[j] *= j & 1 ? f[j >> 1].y : f[j >> 1].x;
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          pan[i * 4 + (j ^ s2)] = make_double2(x[j], x[j + 4]);
          w[j ^ s2] = below ? make_double2(0.0, 0.0) : make_double2(x[2 * j], x[2 * j + 1]);      // X's from here on / final
        }
        if (!below) {
#pragma unroll
          for (int j = 0; j < 8; ++j) mxh = max(mxh, __double2hiint(x[j]) & 0x7FFFFFFF);
        }
        if (t.L64 && b >= p && i < n) {
#pragma unroll
          for (int j = 0; j < 8; ++j)
            if (below || j <= rr) t.L64[(size_t)(8 * p + j) * n + i] = below ? x[j] : lb[8 * rr + j];
        }
      }
      __syncthreads();                                   // B: the panel is published
      if (p + 1 == NT) break;
      const int q0 = row_start(p + 1), next = q0 + p + 1;      // (the next diagonal block is warp 0's)
      int I = p + 1, J = wi;
#pragma unroll 2
      for (int q = q0 + wi; q < n_tiles; q += kCholInvWorkers, J += kCholInvWorkers) {
        while (J > I) { J -= I + 1; ++I; }
        if (q == next) continue;
        // Schur complement (J > p): P_I P_J^T; X (J, I): X_J P_I^T
        const double2 f = pan[(J > p ? I : J) * 32 + at_lane], g = pan[(J > p ? J : I) * 32 + at_lane], w = tile[q * 32 + at_lane];
        double d[2] = {0.0, 0.0};
        dmma(d, f.x, g.x);
        dmma(d, f.y, g.y);
        tile[q * 32 + at_lane] = make_double2(w.x + d[0], w.y + d[1]);
      }
    }
  } else if (warp) {
    for (int p = 0; p < NT; ++p) { __syncthreads(); __syncthreads(); }
  } else {
    // ---------------- the chain
#pragma unroll 1
    for (int p = 0; p < NT; ++p) {
      const double2 w0 = tile[(row_start(p) + p) * 32 + at_lane];
      double a0[2] = {w0.x, w0.y};
      if (p > 0) {                                       // columns 0, 2, 4, 6 of the panel, and 1, 3, 5, 7
        const double *q = (const double *)(pan + (8 * p + r) * 4) + (c >> 1);
        const double ev = q[2 * ((2 * (c & 1)) ^ (r >> 1))], od = q[2 * ((2 * (c & 1) + 1) ^ (r >> 1))];
        double a1[2] = {0.0, 0.0};
        dmma(a0, ev, ev);
        dmma(a1, od, od);
        a0[0] += a1[0]; a0[1] += a1[1];
      }
      __syncwarp();
      ((double2 *)blk)[lane] = make_double2(a0[0], a0[1]);
      __syncwarp();
      const int w = min(8, n - 8 * p);
      double Lb[8][8], mine = 0.0;
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j <= i; ++j) Lb[i][j] = -blk[i * 8 + j];
      __syncwarp();
#pragma unroll
      for (int q = 0; q < 8; ++q) {          // L D L^T, the columns not yet divided by their pivots
        const double d = Lb[q][q], dg = q < w ? diag0[8 * p + q] : 0.0;
        const bool bad = !(d > t.dead_rel * dg) || !(dg > 0);
        const double inv = bad ? 0.0 : rcp_pos(d);
        if (lane == q) mine = bad ? 0.0 : d;
#pragma unroll
        for (int i = q; i < 8; ++i) if (lane == 0) blk[8 * i + q] = Lb[i][q];
        double u[8];
#pragma unroll
        for (int i = q + 1; i < 8; ++i) u[i] = Lb[i][q] * inv;
#pragma unroll
        for (int j = q + 1; j < 8; ++j)
#pragma unroll
          for (int i = j; i < 8; ++i) Lb[i][j] = fma(-Lb[i][q], u[j], Lb[i][j]);
      }
      const double rs = mine > 0.0 ? rsqrt_pos(mine) : 0.0;
      if (lane < w && mine == 0.0) s_dead = 1;
      if (lane < 8) ipiv[lane] = rs;
      __syncwarp();
      {
        const double2 x = ((const double2 *)blk)[lane], f = ((const double2 *)ipiv)[c];
        ((double2 *)lb)[lane] = make_double2(x.x * f.x, x.y * f.y);
      }
      __syncthreads();                                   // A
      __syncthreads();                                   // B
    }
  }
  mxh = __reduce_max_sync(0xffffffffu, mxh);
  if (lane == 0) s_red[warp] = mxh;
  __syncthreads();
  if (tid == 0 && s_dead && t.status) atomicOr(t.status, 2);
  if (t.L64) {
    for (int j = warp; j < n; j += NW)
      for (int i = lane; i < j; i += 32) t.L64[(size_t)j * n + i] = 0.0;
    if (warp == 0) {     // max |L_ij|^2 <= max G_ii: exponent for the single-precision Jacobi iteration
      double mxd = 0.0;
      for (int i = lane; i < n; i += 32) mxd = fmax(mxd, diag0[i]);
      for (int o = 16; o; o >>= 1) mxd = fmax(mxd, __shfl_xor_sync(0xffffffffu, mxd, o));
      int e2 = 0;
      if (mxd > 0.0 && mxd < 1e300) frexp(mxd, &e2);
      if (lane == 0) t.L64[(size_t)n * n] = (double)((e2 + 1) / 2 + 1);
    }
  }
  if (!t.Lhi) return;
  // ---- L^-1: (L^-1)_ic = X[c][i] for c <= i.  Scaled so that the largest entry lies in [2^9, 2^10).
  mxh = __reduce_max_sync(0xffffffffu, lane < NW ? s_red[lane] : 0);
  const int xe = (mxh >> 20) - 1023, le = mxh > 0 && xe < 1024 ? 9 - xe : 0;
  if (tid == 0) *t.l_exp = le;
  const double sc = ldexp(1.0, le);
  const int nb = kp >> 3;
#pragma unroll 2
  for (int q = warp; q < nb * nb; q += NW) {             // rows 8 I .., columns 8 J .. of L^-1: the transpose of X (J, I)
    const int I = q / nb, J = q - I * nb;
    double2 x = make_double2(0.0, 0.0);
    if (J <= I && I < NT) x = tile[(row_start(I) + J) * 32 + at_lane];
    const float f0 = (float)(x.x * sc), f1 = (float)(x.y * sc);
    // lanes r and r ^ 1 trade: the even one keeps column 2 c of X, the odd one column 2 c + 1, each a pair of rows
    const bool odd = r & 1;
    const float o = __shfl_xor_sync(0xffffffffu, odd ? f0 : f1, 4);
    const __half2 h = odd ? __floats2half2_rn(o, f1) : __floats2half2_rn(f0, o);
    const float2 hf = __half22float2(h);
    const size_t at = (size_t)(8 * I + 2 * c + (odd ? 1 : 0)) * kp + 8 * J + (r & ~1);
    *(__half2 *)(t.Lhi + at) = h;
    *(__half2 *)(t.Llo + at) = odd ? __floats2half2_rn(o - hf.x, f1 - hf.y) : __floats2half2_rn(f0 - hf.x, o - hf.y);
  }
}

// ---------------------------------------------------------------------------------------------- apply
// One CTA per 128 rows of the basis: D[128 rows][kp] = sum_j R[row][j] Linv[c][j].
__global__ void __launch_bounds__(OR_THREADS, 1) orth_apply_kernel(const OrthCell *__restrict__ cells) {
  extern __shared__ unsigned char smem_raw[];
  const OrthCell &c = cells[blockIdx.y];
  const int tpp = c.rpp / 128;                        // 128-row tiles per panel
  if ((int)blockIdx.x >= c.panels * tpp) return;
  const int panel = blockIdx.x / tpp, r0 = (blockIdx.x - panel * tpp) * 128;
  const int kp = c.kp, nkb = (kp + 63) / 64;

  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  unsigned char *sm = smem_raw + (base - raw);
  const uint32_t tile = (uint32_t)kp * 128u;           // [kp rows][64 elements]
  const uint32_t sAhi = base, sAlo = base + 2 * tile, sBhi = base + 4 * tile, sBlo = sBhi + nkb * tile;
  const uint32_t sBar = sBlo + nkb * tile;
  const size_t bar_off = (size_t)(4 + 2 * nkb) * tile;
  volatile int *abort_flag = (volatile int *)(sm + bar_off + 64);
  uint32_t *tmem_slot = (uint32_t *)(sm + bar_off + 72);
  const uint32_t bLoad = sBar, bDone = sBar + 8;

  const int warp = warp_uniform(), lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    *abort_flag = 0;
    mbar_init(bLoad, 1); mbar_init(bDone, 1);
    fence_barrier_init();
  }
  if (warp == 4) { tmem_alloc(smem_u32(tmem_slot), 256); tmem_relinquish(); }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  if (warp == 4 && lane == 0) {
    tma_prefetch_desc(&c.tmHi); tma_prefetch_desc(&c.tmLo); tma_prefetch_desc(&c.tmLhi); tma_prefetch_desc(&c.tmLlo);
    mbar_expect_tx(bLoad, (4 + 2 * nkb) * tile);
    for (int hf = 0; hf < 2; ++hf) {
      tma_load_3d(sAhi + hf * tile, &c.tmHi, bLoad, r0 + hf * 64, 0, panel);
      tma_load_3d(sAlo + hf * tile, &c.tmLo, bLoad, r0 + hf * 64, 0, panel);
    }
    for (int kb = 0; kb < nkb; ++kb) {
      tma_load_2d(sBhi + kb * tile, &c.tmLhi, bLoad, kb * 64, 0);
      tma_load_2d(sBlo + kb * tile, &c.tmLlo, bLoad, kb * 64, 0);
    }
  } else if (warp == 5) {
    if (mbar_wait_warp(bLoad, 0, abort_flag)) {
      tc_fence_after();
      const uint32_t idesc = umma_idesc_f16(128, kp, 1, 0);
      for (int ks = 0; ks < kp / 16; ++ks) {
        // A: MN-major, 16 contraction rows = 2048 B per step, the second 64 rows of the tile `tile` bytes further
        const uint64_t aH = umma_desc_sw128(sAhi + ks * 2048, tile, 1024), aL = umma_desc_sw128(sAlo + ks * 2048, tile, 1024);
        const uint32_t boff = (uint32_t)(ks >> 2) * tile + (uint32_t)(ks & 3) * 32;
        const uint64_t bH = umma_desc_sw128(sBhi + boff, 16, 1024), bL = umma_desc_sw128(sBlo + boff, 16, 1024);
        umma_f16(tmem_base, aH, bH, idesc, ks != 0);
        umma_f16(tmem_base, aH, bL, idesc, 1);
        umma_f16(tmem_base, aL, bH, idesc, 1);
      }
      umma_commit(bDone);
    }
  } else if (warp < 4) {
    const bool ok = __all_sync(0xffffffffu, mbar_wait(bDone, 0, abort_flag));
    if (ok) {
      tc_fence_after();
      const int row = warp * 32 + lane;                       // row of the tile
      const uint32_t t_lane = tmem_base + ((uint32_t)(warp * 32) << 16);
      const float s_in = ldexpf(1.0f, -*c.l_exp), s_out = ldexpf(1.0f, c.out_exp);
      float *orow = c.out32 ? c.out32 + ((size_t)panel * c.rpp + r0 + row) * c.ld : nullptr;
      // the operand tiles are consumed: stage the fp16 result over them in the layout they were loaded in
      unsigned char *hiT = sm + (row >> 6) * tile, *loT = sm + 2 * tile + (row >> 6) * tile;
      const int rr = row & 63;
      for (int ch = 0; ch * 16 < kp; ++ch) {
        float v[16];
        tmem_ld16(t_lane + ch * 16, v);
        tmem_wait_ld();
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          const int col = ch * 16 + i;
          const float q = v[i] * s_in;
          if (orow && col < c.k) orow[col] = q;
          const float qs = col < c.k ? q * s_out : 0.f;
          const __half h = __float2half_rn(qs);
          const uint32_t off = (uint32_t)col * 128u + ((((uint32_t)rr >> 3) ^ ((uint32_t)col & 7u)) << 4) + ((uint32_t)rr & 7u) * 2u;
          *(__half *)(hiT + off) = h;
          *(__half *)(loT + off) = __float2half_rn(qs - __half2float(h));
        }
      }
      fence_proxy_async();
    }
    named_bar_sync(1, 128);
    if (ok && threadIdx.x == 0) {
      for (int hf = 0; hf < 2; ++hf) {
        tma_store_3d(&c.tmHi, sAhi + hf * tile, r0 + hf * 64, 0, panel);
        tma_store_3d(&c.tmLo, sAlo + hf * tile, r0 + hf * 64, 0, panel);
      }
      tma_store_commit_wait();
    }
  }
  tc_fence_before();
  __syncthreads();
  if (*abort_flag) {
    if (threadIdx.x == 0) atomicOr(c.status, 8);
    const long long t0 = clock64();
    while (clock64() - t0 < 2000000) {}
    __syncthreads();
  }
  if (warp == 4) { tc_fence_after(); tmem_dealloc(tmem_base, 256); }
}

// ---------------------------------------------------------------------------------------------- split with a measured scale
// |x| maximum of fp32 arrays (one slot per job, zeroed by the caller); values are non-negative, so the integer
// maximum of the bit patterns is the floating-point maximum.
struct AbsMaxJob { const float *in; long long n; unsigned *slot; };
__global__ void absmax_kernel(const AbsMaxJob *__restrict__ jobs) {
  const AbsMaxJob j = jobs[blockIdx.y];
  float mx = 0.f;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < j.n; i += (long long)gridDim.x * blockDim.x)
    mx = fmaxf(mx, fabsf(j.in[i]));
  for (int o = 16; o; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if ((threadIdx.x & 31) == 0 && mx > 0.f && isfinite(mx)) atomicMax(j.slot, __float_as_uint(mx));
}

}  // namespace tc
}  // namespace jolt
