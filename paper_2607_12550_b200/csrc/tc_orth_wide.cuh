// CholeskyQR on tensor cores for sketch widths beyond one accumulator (k > 152: long contexts with ranks up to 256, and the
// spectrum probe at its cap of 512 directions).  Same operand layout and roles as tc_orth.cuh; the k x k Gram and the product
// with L^-1 are cut into 128 x 128 blocks:
//
//   orthw_gram_kernel    block (rb, cb >= rb) of G = R^T R over a run of 64-row steps: A = rows rb of the transposed basis,
//                        B = rows cb; the accumulator is flushed into fp32 registers after every step
//   chol_cluster_kernel  G = L L^T, L^-1 in fp64 (chol_cluster.cuh)
//   orthw_apply_kernel   Q = R L^-T for 128 rows of the basis, column blocks from the last to the first: block c only needs
//                        the columns j <= c of R, so it may replace its own columns in place
//
// hi hi goes to one accumulator and hi lo + lo hi to another (the fp32 accumulation of tcgen05.mma truncates about 2^-24 of
// the running sum per step, and the cross terms would triple the steps of the main sum); both are added in registers.
// The fp64 CUDA-core path these kernels replace for 16-bit caches (tall Gram, single-CTA Cholesky, row-wise triangular solve) took
// 12 ms per pass and group of four cells of 32768 rows at k = 522: the solve alone is rows x k^2 fp32 operations
// through shared memory.
#pragma once
#include "tc_orth.cuh"

namespace jolt {
namespace tc {

constexpr int OW_THREADS = 192;           // warps 0-3 epilogue, warp 4 TMA, warp 5 MMA
constexpr int OW_GRAM_STEPS = 16;         // 64-row steps per Gram CTA
constexpr int OW_STAGES = 3;
constexpr int OW_STAGE_BYTES = 65536;     // four operand tiles of 16 KB
constexpr int OW_GRAM_SMEM = OW_STAGES * OW_STAGE_BYTES + 1024 + 512;
constexpr int OW_APPLY_SMEM = OW_STAGES * OW_STAGE_BYTES + 32768 + 1024 + 512;      // + output staging (64 columns, hi + lo)

struct alignas(64) OrthWCell {
  CUtensorMap tmHi, tmLo;     // basis [panels][kp][rpp] fp16, box {64 rows, 128 columns, 1}
  CUtensorMap tmAhi, tmAlo;   // the same with box {64, 64, 1} (apply: operand and output)
  CUtensorMap tmLhi, tmLlo;   // L^-1 [kp][kp], box {64 j, 128 c}
  float *part;                // [n_chunks][kp][kp], entries (r, c) with block(c) >= block(r)
  int *l_exp;
  float *out32;
  int ld, k, kp, rpp, panels, n_chunks, out_exp;
  int *status;
  const __half *hi, *lo;      // the basis
  double *unit;               // [k] orthw_norms_kernel
};

// unit[c] = 1 / |column c| of the finished basis (1 for a dead one).  The tensor core's accumulation truncates, which shows where
// every term has one sign: on the diagonal of the Gram, and in Q = R L^-T through the one large term of each entry.  The columns
// come out up to 2e-7 long; what is made of them takes the factor along (UnitJob).  A warp per column, eight rows a lane and
// step; bound by reading the basis once (4 bytes an entry).
__global__ void __launch_bounds__(256) orthw_norms_kernel(const OrthWCell *__restrict__ cells) {
  const OrthWCell &c = cells[blockIdx.y];
  const int col = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (col >= c.k) return;
  const int per = c.rpp / 8, total = c.panels * per;           // pieces of eight rows: of a panel, of the column
  double s0 = 0.0, s1 = 0.0;
#pragma unroll 2
  for (int e = lane; e < total; e += 32) {
    const int panel = e / per;
    const size_t o = ((size_t)panel * c.kp + col) * c.rpp + (size_t)(e - panel * per) * 8;
    const uint4 h = __ldg((const uint4 *)(c.hi + o)), l = __ldg((const uint4 *)(c.lo + o));
    const uint32_t hw[4] = {h.x, h.y, h.z, h.w}, lw[4] = {l.x, l.y, l.z, l.w};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float2 a = __half22float2(*(const __half2 *)&hw[q]), b = __half22float2(*(const __half2 *)&lw[q]);
      const double x = (double)a.x + (double)b.x, y = (double)a.y + (double)b.y;
      s0 = fma(x, x, s0); s1 = fma(y, y, s1);
    }
  }
  s0 += s1;
  for (int o = 16; o; o >>= 1) s0 += __shfl_xor_sync(0xffffffffu, s0, o);
  const double n2 = ldexp(s0, -2 * c.out_exp);
  if (lane == 0) c.unit[col] = n2 > 0.25 ? rsqrt(n2) : 1.0;
}

__global__ void __launch_bounds__(OW_THREADS, 1) orthw_gram_kernel(const OrthWCell *__restrict__ cells) {
  extern __shared__ unsigned char smem_raw[];
  const OrthWCell &c = cells[blockIdx.z];
  if ((int)blockIdx.x >= c.n_chunks) return;
  const int kp = c.kp, nb = (kp + 127) / 128;
  int rb = 0, cb = blockIdx.y;              // block pairs in the order (0,0) (0,1) .. (1,1) ..
  for (; rb < nb && cb >= nb - rb; ++rb) cb -= nb - rb;
  if (rb >= nb) return;
  cb += rb;
  const bool diag = cb == rb;
  const int spp = c.rpp / 64, total = c.panels * spp;
  const int s0 = blockIdx.x * OW_GRAM_STEPS, n_steps = min(OW_GRAM_STEPS, total - s0);
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  unsigned char *sm = smem_raw + (base - raw);
  const uint32_t sBar = base + OW_STAGES * OW_STAGE_BYTES;
  volatile int *abort_flag = (volatile int *)(sm + OW_STAGES * OW_STAGE_BYTES + 256);
  uint32_t *tmem_slot = (uint32_t *)(sm + OW_STAGES * OW_STAGE_BYTES + 264);
  auto bFull = [=](int s) { return sBar + 8 * s; };
  auto bEmpty = [=](int s) { return sBar + 64 + 8 * s; };
  auto bAfull = [=](int b) { return sBar + 128 + 8 * b; };
  auto bAempty = [=](int b) { return sBar + 144 + 8 * b; };
  const int warp = warp_uniform(), lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    *abort_flag = 0;
    for (int s = 0; s < OW_STAGES; ++s) { mbar_init(bFull(s), 1); mbar_init(bEmpty(s), 1); }
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
    for (int j = 0; j < n_steps; ++j) {
      const int s = j % OW_STAGES, n = j / OW_STAGES;
      if (!mbar_wait(bEmpty(s), (n & 1) ^ 1, abort_flag)) break;
      const int step = s0 + j, panel = step / spp, r0 = (step - panel * spp) * 64;
      const uint32_t st = base + s * OW_STAGE_BYTES;
      mbar_expect_tx(bFull(s), diag ? 32768 : 65536);
      tma_load_3d(st, &c.tmHi, bFull(s), r0, cb * 128, panel);
      tma_load_3d(st + 16384, &c.tmLo, bFull(s), r0, cb * 128, panel);
      if (!diag) {
        tma_load_3d(st + 32768, &c.tmHi, bFull(s), r0, rb * 128, panel);
        tma_load_3d(st + 49152, &c.tmLo, bFull(s), r0, rb * 128, panel);
      }
    }
  } else if (warp == 5) {
    const uint32_t idesc = umma_idesc_f16(128, 128, 0, 0);
    for (int j = 0; j < n_steps; ++j) {
      const int s = j % OW_STAGES, n = j / OW_STAGES, b = j & 1, q = j >> 1;
      if (!mbar_wait_warp(bFull(s), n & 1, abort_flag)) break;
      if (!mbar_wait_warp(bAempty(b), (q & 1) ^ 1, abort_flag)) break;
      tc_fence_after();
      const uint32_t bt = base + s * OW_STAGE_BYTES, at = diag ? bt : bt + 32768;
      const uint32_t d0 = tmem_base + b * 256, d1 = d0 + 128;
#pragma unroll
      for (int k4 = 0; k4 < 4; ++k4) {
        const uint64_t aH = umma_desc_sw128(at + k4 * 32, 16, 1024), aL = umma_desc_sw128(at + 16384 + k4 * 32, 16, 1024);
        const uint64_t bH = umma_desc_sw128(bt + k4 * 32, 16, 1024), bL = umma_desc_sw128(bt + 16384 + k4 * 32, 16, 1024);
        umma_f16(d0, aH, bH, idesc, k4 != 0);
        umma_f16(d1, aH, bL, idesc, k4 != 0);
        umma_f16(d1, aL, bH, idesc, 1);
      }
      umma_commit(bEmpty(s));
      umma_commit(bAfull(b));
    }
  } else if (warp < 4) {
    float acc[128];
#pragma unroll
    for (int i = 0; i < 128; ++i) acc[i] = 0.f;
    const uint32_t t_lane = tmem_base + ((uint32_t)(warp * 32) << 16);
    bool ok = true;
    for (int j = 0; j < n_steps; ++j) {
      const int b = j & 1, q = j >> 1;
      ok = __all_sync(0xffffffffu, mbar_wait(bAfull(b), q & 1, abort_flag));
      if (!ok) break;
      tc_fence_after();
#pragma unroll
      for (int ch = 0; ch < 8; ++ch) {
        float v[16], x[16];
        tmem_ld16(t_lane + b * 256 + ch * 16, v);
        tmem_ld16(t_lane + b * 256 + 128 + ch * 16, x);
        tmem_wait_ld();
#pragma unroll
        for (int i = 0; i < 16; ++i) acc[ch * 16 + i] += v[i] + x[i];
      }
      tc_fence_before();
      mbar_arrive(bAempty(b));
    }
    const int row = rb * 128 + warp * 32 + lane;
    if (ok && row < kp) {
      float4 *out = (float4 *)(c.part + (size_t)blockIdx.x * kp * kp + (size_t)row * kp + cb * 128);
#pragma unroll
      for (int i = 0; i < 32; ++i)
        if (cb * 128 + 4 * i < kp) out[i] = make_float4(acc[4 * i], acc[4 * i + 1], acc[4 * i + 2], acc[4 * i + 3]);
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

// One CTA per 128 rows of the basis; column blocks of 128 from the last to the first, two accumulator pairs.
__global__ void __launch_bounds__(OW_THREADS, 1) orthw_apply_kernel(const OrthWCell *__restrict__ cells) {
  extern __shared__ unsigned char smem_raw[];
  const OrthWCell &c = cells[blockIdx.y];
  const int tpp = c.rpp / 128;
  if ((int)blockIdx.x >= c.panels * tpp) return;
  const int panel = blockIdx.x / tpp, r0 = (blockIdx.x - panel * tpp) * 128;
  const int kp = c.kp, nb = (kp + 127) / 128;
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  unsigned char *sm = smem_raw + (base - raw);
  constexpr int OFF_STG = OW_STAGES * OW_STAGE_BYTES, OFF_BAR = OFF_STG + 32768;
  const uint32_t sStg = base + OFF_STG, sBar = base + OFF_BAR;
  volatile int *abort_flag = (volatile int *)(sm + OFF_BAR + 256);
  uint32_t *tmem_slot = (uint32_t *)(sm + OFF_BAR + 264);
  auto bFull = [=](int s) { return sBar + 8 * s; };
  auto bEmpty = [=](int s) { return sBar + 64 + 8 * s; };
  auto bAfull = [=](int b) { return sBar + 128 + 8 * b; };
  auto bAempty = [=](int b) { return sBar + 144 + 8 * b; };
  const int warp = warp_uniform(), lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    *abort_flag = 0;
    for (int s = 0; s < OW_STAGES; ++s) { mbar_init(bFull(s), 1); mbar_init(bEmpty(s), 1); }
    for (int b = 0; b < 2; ++b) { mbar_init(bAfull(b), 1); mbar_init(bAempty(b), 128); }
    fence_barrier_init();
  }
  if (warp == 4) { tmem_alloc(smem_u32(tmem_slot), 512); tmem_relinquish(); }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  // 64-column steps a block needs: the columns j below the end of the block
  auto steps_of = [=](int cbk) { return (min(kp, cbk * 128 + 128) + 63) / 64; };

  if (warp == 4 && lane == 0) {
    tma_prefetch_desc(&c.tmAhi); tma_prefetch_desc(&c.tmAlo); tma_prefetch_desc(&c.tmLhi); tma_prefetch_desc(&c.tmLlo);
    bool ok = true;
    int cnt = 0;
    for (int cbk = nb - 1; ok && cbk >= 0; --cbk)
      for (int j = 0; j < steps_of(cbk); ++j, ++cnt) {
        const int s = cnt % OW_STAGES, n = cnt / OW_STAGES;
        ok = mbar_wait(bEmpty(s), (n & 1) ^ 1, abort_flag);
        if (!ok) break;
        const uint32_t st = base + s * OW_STAGE_BYTES;
        mbar_expect_tx(bFull(s), OW_STAGE_BYTES);
        for (int hf = 0; hf < 2; ++hf) {
          tma_load_3d(st + hf * 8192, &c.tmAhi, bFull(s), r0 + hf * 64, j * 64, panel);
          tma_load_3d(st + 16384 + hf * 8192, &c.tmAlo, bFull(s), r0 + hf * 64, j * 64, panel);
        }
        tma_load_2d(st + 32768, &c.tmLhi, bFull(s), j * 64, cbk * 128);
        tma_load_2d(st + 49152, &c.tmLlo, bFull(s), j * 64, cbk * 128);
      }
  } else if (warp == 5) {
    const uint32_t idesc = umma_idesc_f16(128, 128, 1, 0);
    bool ok = true;
    int cnt = 0;
    for (int i = 0; ok && i < nb; ++i) {
      const int cbk = nb - 1 - i, b = i & 1, q = i >> 1, ns = steps_of(cbk);
      ok = mbar_wait_warp(bAempty(b), (q & 1) ^ 1, abort_flag);
      if (!ok) break;
      tc_fence_after();
      const uint32_t d0 = tmem_base + b * 256, d1 = d0 + 128;
      for (int j = 0; j < ns; ++j, ++cnt) {
        const int s = cnt % OW_STAGES, n = cnt / OW_STAGES;
        ok = mbar_wait_warp(bFull(s), n & 1, abort_flag);
        if (!ok) break;
        tc_fence_after();
        const uint32_t st = base + s * OW_STAGE_BYTES;
#pragma unroll
        for (int k4 = 0; k4 < 4; ++k4) {
          // A: MN-major, 16 contraction rows = 2048 B per step, the second 64 rows 8 KB further
          const uint64_t aH = umma_desc_sw128(st + k4 * 2048, 8192, 1024), aL = umma_desc_sw128(st + 16384 + k4 * 2048, 8192, 1024);
          const uint64_t bH = umma_desc_sw128(st + 32768 + k4 * 32, 16, 1024), bL = umma_desc_sw128(st + 49152 + k4 * 32, 16, 1024);
          umma_f16(d0, aH, bH, idesc, (j | k4) != 0);
          umma_f16(d1, aH, bL, idesc, (j | k4) != 0);
          umma_f16(d1, aL, bH, idesc, 1);
        }
        umma_commit(bEmpty(s));
      }
      if (ok) umma_commit(bAfull(b));
    }
  } else if (warp < 4) {
    const int row = warp * 32 + lane;
    const uint32_t t_lane = tmem_base + ((uint32_t)(warp * 32) << 16);
    const float s_in = ldexpf(1.0f, -*c.l_exp), s_out = ldexpf(1.0f, c.out_exp);
    float *const orow = c.out32 ? c.out32 + ((size_t)panel * c.rpp + r0 + row) * c.ld : nullptr;
    unsigned char *hiT = sm + OFF_STG + (row >> 6) * 8192, *loT = hiT + 16384;
    const int rr = row & 63;
    bool ok = true;
    for (int i = 0; i < nb; ++i) {
      const int cbk = nb - 1 - i, b = i & 1, q = i >> 1;
      // every epilogue thread walks the same barriers whether or not a wait timed out
      ok = __all_sync(0xffffffffu, ok && mbar_wait(bAfull(b), q & 1, abort_flag));
      tc_fence_after();
      for (int g = 0; g < 2; ++g) {                      // 64 columns at a time
        const int col0 = cbk * 128 + g * 64;
        if (col0 >= kp) break;
        if (threadIdx.x == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");    // staging has been read
        named_bar_sync(1, 128);
        if (ok) {
#pragma unroll
          for (int ch = 0; ch < 4; ++ch) {
            float v[16], x[16];
            tmem_ld16(t_lane + b * 256 + g * 64 + ch * 16, v);
            tmem_ld16(t_lane + b * 256 + 128 + g * 64 + ch * 16, x);
            tmem_wait_ld();
#pragma unroll
            for (int e = 0; e < 16; ++e) {
              const int cl = ch * 16 + e, col = col0 + cl;
              const float qv = (v[e] + x[e]) * s_in;
              if (orow && col < c.k) orow[col] = qv;
              const float qs = col < c.k ? qv * s_out : 0.f;
              const __half h = __float2half_rn(qs);
              const uint32_t off = (uint32_t)cl * 128u + ((((uint32_t)rr >> 3) ^ ((uint32_t)cl & 7u)) << 4) + ((uint32_t)rr & 7u) * 2u;
              *(__half *)(hiT + off) = h;
              *(__half *)(loT + off) = __float2half_rn(qs - __half2float(h));
            }
          }
          fence_proxy_async();
        }
        named_bar_sync(1, 128);
        if (ok && threadIdx.x == 0) {
          for (int hf = 0; hf < 2; ++hf) {
            tma_store_3d(&c.tmAhi, sStg + hf * 8192, r0 + hf * 64, col0, panel);
            tma_store_3d(&c.tmAlo, sStg + 16384 + hf * 8192, r0 + hf * 64, col0, panel);
          }
          asm volatile("cp.async.bulk.commit_group;" ::: "memory");
        }
      }
      tc_fence_before();
      mbar_arrive(bAempty(b));
    }
    if (threadIdx.x == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
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

}  // namespace tc
}  // namespace jolt
