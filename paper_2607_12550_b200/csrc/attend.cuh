// Single-step attention computed on the compressed cache, without materialising keys or values.
//
// The paper names this as the route to decode parity ("a fused kernel that runs attention directly on the
// factors, without materializing the cache", Sec. 7 and the closing discussion) and gives no algorithm.  What is
// computed here, per layer group, merged head h and query i (n_q queries per KV head):
//     s_t = scale <q_i, K^[h, t]>,   p = softmax_t(s),   o_i = sum_t p_t V^[h, t],
// with K^, V^ the decoded (not yet rounded) cells  X^ = 2^e U_T P_h + s . H(r^') / sqrt(d),  P_h = fp16(G_h U_F^T).
// Both contractions move to the small side:
//     <q, K^[h, t]>     = 2^e sum_k U_T[t, k] (P_h q)[k]  +  < H(s . q) / sqrt(d), r^'[h, t] >
//     sum_t p_t V^[h,t] = 2^e (p^T U_T) P_h               +  s . H( sum_t p_t r^'[h, t] ) / sqrt(d)
// so a call streams U_T and the packed codes once each (the compressed bytes) instead of the fp16 cache, and the
// Hadamard rotation is applied to one query / one output row per head instead of every token.
//
// Kernels of a call (contractions with a tensor-core shape are warp-level fp16 MMAs with fp32 accumulation, an fp32
// operand entering as hi + lo fp16; the rest is CUDA-core fp32):
//   (P_h = fp16(G_h U_F^T), the projected core the decoder also reads, is kept with the handle since compress)
//   attend_prep_kernel     per (group, head, query): rotated scaled query (fp32, and scaled hi + lo fp16), w = P_h q
//   attend_stream_kernel   per (group, four heads, 128-token chunk): scores, chunk maximum, p = exp(s - max), chunk sum,
//                          sum_t p_t r^'_t and p^T U_T
//   attend_combine_kernel  per (group, head, query): merges the chunks (running-maximum rescaling), applies P_h of the
//                          value cell and the inverse rotation, divides by the softmax denominator
// The portable path has four kernels in place of the streaming one: attend_bscore_kernel (U_T w of all heads of a cell as one
// dense product), attend_scores_kernel, attend_values_kernel (codes on the CUDA cores), attend_bvalue_kernel (p^T U_T).
// Keys compressed before a rotary embedding cannot use the first identity (the rotation differs per token).
#pragma once
#include <cuda_fp16.h>

#include "common.cuh"
#include "rowquant.cuh"

namespace jolt {

constexpr int kAttChunk = 256;      // portable kernels: tokens per chunk = threads per CTA (the streaming kernel: kAttTok)
constexpr int kAttMaxQ = 8;         // queries per KV head (padded to 4 or 8 inside)

struct AttendCell {
  const __half *G, *UT, *UF;        // [m * r_t][r_f], [T][r_t], [128][r_f]
  const int *e;
  const uint32_t *words;            // [m][T][4 * bits]
  const __half *scales;             // [m][T][4]
  int r_t, r_f, bits, cell;
};

struct AttendJob {                  // one per layer group
  AttendCell k, v;
  int m, T;
  const float *q;                   // [m][n_q][128]
  float *out;                       // [m][n_q][128]
  __half *kP, *vP;                  // [m * r_t][128]    P_h = fp16(G_h U_F^T) of the key / value cell (scaled units)
  __half *wh, *wl;                  // [m NQP][k.r_t]    P_h q times 2^-E_n per column n = (head, query), as hi + lo fp16
  float *we;                        // [m NQP]           scale 2^e 2^E_n
  float *qt;                        // [m][128][NQP]     scale H(s . q) / sqrt(d)
  __half *qh, *ql;                  // [m][8][128]       the same, times 2^-E per (head, query), as hi + lo fp16 (MMA operand)
  float *qe;                        // [m][8]            2^E
  float *p;                         // [m][T][NQP]       exp(s - chunk maximum)
  float *ml;                        // [m][n_chunks][2][NQP]  chunk maximum, chunk sum
  float *y;                         // [m][n_chunks][NQP][v.r_t]
  float *a;                         // [m][n_chunks][NQP][128]
};

// The descriptors of a short call travel as a kernel argument (up to 15 layer groups): the copy ahead of it cost more than its
// kernels' ramps (35 -> 31 us at 384 tokens).  A call of more than one wave of CTAs has them in the table arena: the streaming
// kernel that reads them from its argument spills 48 bytes (128.5 against 126.3 us at 4096 tokens).
constexpr int kAttArgJobs = 15;
struct AttendArgs {
  const AttendJob *table;           // null: j
  AttendJob j[kAttArgJobs];
};
__device__ __forceinline__ const AttendJob &att_job(const AttendArgs &a, int i) { return a.table ? a.table[i] : a.j[i]; }

// 128-point Walsh-Hadamard transform by one warp: lane l holds elements 4 l .. 4 l + 3.
__device__ __forceinline__ void att_wht_warp(float (&v)[4]) {
  const int lane = threadIdx.x & 31;
  float a = v[0] + v[1], b = v[0] - v[1], c = v[2] + v[3], d = v[2] - v[3];
  v[0] = a + c; v[1] = b + d; v[2] = a - c; v[3] = b - d;
#pragma unroll
  for (int len = 1; len < 32; len <<= 1)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float o = __shfl_xor_sync(0xffffffffu, v[j], len);
      v[j] = lane & len ? o - v[j] : v[j] + o;
    }
}

// Sums over the warp of N values a lane (4 or 8): the sum of value att_sum_index(lane) on return.
template <int N>
__device__ __forceinline__ float att_warp_sums(float (&v)[N]) {
  const int lane = threadIdx.x & 31;
  int o = 16;
#pragma unroll
  for (int n = N; n > 1; n >>= 1, o >>= 1)
#pragma unroll
    for (int j = 0; j < n / 2; ++j) {
      const float keep = lane & o ? v[j + n / 2] : v[j], give = lane & o ? v[j] : v[j + n / 2];
      v[j] = keep + __shfl_xor_sync(0xffffffffu, give, o);
    }
#pragma unroll
  for (; o > 0; o >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
  return v[0];
}

// A kernel launched while its predecessor still runs waits here before it reads what that one wrote: by plain loads (the read-only
// path, __ldg, is for memory that nobody writes while the kernel is resident, and may be moved across the wait).
__device__ __forceinline__ void att_wait_predecessor() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void att_let_successor_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

__device__ __forceinline__ float att_sign(uint64_t seed, int cell, int f) {
  uint32_t sw[4];
  cell_sign_words(seed, cell, sw);
  return ((sw[f >> 5] >> (f & 31)) & 1u) ? -1.f : 1.f;
}

// grid (m, groups), 256 threads: a warp per query rotates it (four features a lane), then a warp per row of P_h forms w with
// four rows in flight.  Bound by the latency of its few loads: with a CTA per query, block-wide transforms and five shuffles
// per value and row it took 19.6 us at 8 groups of 32 heads, rank 128; now 8.8.
template <int NQ>
__global__ void __launch_bounds__(256) attend_prep_kernel(const __grid_constant__ AttendArgs args, int n_q, float scale, uint64_t seed) {
  const AttendJob &jb = att_job(args, blockIdx.y);
  const int h = blockIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (h >= jb.m) return;
  att_let_successor_start();
  const int kr = jb.k.r_t;
  float q[NQ][4];
#pragma unroll
  for (int c = 0; c < NQ; ++c) {
    const float4 v = c < n_q ? *(const float4 *)(jb.q + ((size_t)h * n_q + c) * 128 + lane * 4) : make_float4(0.f, 0.f, 0.f, 0.f);
    q[c][0] = v.x; q[c][1] = v.y; q[c][2] = v.z; q[c][3] = v.w;
  }
  if (jb.k.bits > 0 && warp < NQ) {
    const int i = warp;
    float v[4];
#pragma unroll
    for (int c = 0; c < NQ; ++c)
      if (c == i) { v[0] = q[c][0]; v[1] = q[c][1]; v[2] = q[c][2]; v[3] = q[c][3]; }
#pragma unroll
    for (int j = 0; j < 4; ++j) v[j] *= att_sign(seed, jb.k.cell, lane * 4 + j);
    att_wht_warp(v);
    float mx = 0.f;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      v[j] = v[j] * kInvSqrtD * scale;
      jb.qt[((size_t)h * 128 + lane * 4 + j) * NQ + i] = v[j];
      mx = fmaxf(mx, fabsf(v[j]));
    }
    // the tensor-core form of the same row: scaled by a power of two so that hi + lo fp16 hold it (|entry| < 2^13)
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    int ex = 0;
    if (mx > 0.f && mx < INFINITY) frexpf(mx, &ex);                  // mx < 2^ex
    const float up = ldexpf(1.f, 13 - ex);
    __half hi[4], lo[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float sv = v[j] * up;
      hi[j] = __float2half_rn(sv);
      lo[j] = __float2half_rn(sv - __half2float(hi[j]));
    }
    *(uint2 *)(jb.qh + ((size_t)h * kAttMaxQ + i) * 128 + lane * 4) = *(const uint2 *)hi;
    *(uint2 *)(jb.ql + ((size_t)h * kAttMaxQ + i) * 128 + lane * 4) = *(const uint2 *)lo;
    if (lane == 0) jb.qe[h * kAttMaxQ + i] = ldexpf(1.f, ex - 13);
  }
  if (kr > 0) {
    // w[n][k] = sum_f P_h[k][f] q[f] for column n = (head, query): a warp per row k, a lane per four features.  Stored as
    // hi + lo fp16 times 2^-E_n with 2^E_n > |q|_2: a row of P_h has norm below 2^14.52 (|G| 2^-e < 2^11, r_f <= 128, U_F
    // orthonormal, fp16 rounding), so every scaled entry is below 2^14.52 in magnitude and fits fp16.
    constexpr int RI = 4;                                              // rows in flight
    const uint2 *pr = (const uint2 *)(jb.kP + (size_t)h * kr * 128) + lane;
    uint2 p4[RI];
#pragma unroll
    for (int r = 0; r < RI; ++r) p4[r] = __ldg(pr + (size_t)min(warp * RI + r, kr - 1) * 32);
    float sq[NQ];
#pragma unroll
    for (int c = 0; c < NQ; ++c) sq[c] = fmaf(q[c][0], q[c][0], fmaf(q[c][1], q[c][1], fmaf(q[c][2], q[c][2], q[c][3] * q[c][3])));
    const float nrm = sqrtf(att_warp_sums<NQ>(sq));
    const int c = lane / (32 / NQ);                                    // this lane's query
    int ex = 0;
    if (nrm > 0.f && nrm < INFINITY) frexpf(nrm, &ex);                 // |q|_2 < 2^ex
    ++ex;                                                              // headroom for the rounding of the norm itself
    const float inv = ldexpf(1.f, -ex);
    const bool first = lane % (32 / NQ) == 0;
    if (warp == 0 && first) jb.we[h * NQ + c] = scale * ldexpf(1.f, *jb.k.e) * ldexpf(1.f, ex);
    for (int k = warp * RI; k < kr; k += 8 * RI) {
      uint2 pc[RI];
#pragma unroll
      for (int r = 0; r < RI; ++r) pc[r] = p4[r];
      if (k + 8 * RI < kr)
#pragma unroll
        for (int r = 0; r < RI; ++r) p4[r] = __ldg(pr + (size_t)min(k + 8 * RI + r, kr - 1) * 32);
#pragma unroll
      for (int r = 0; r < RI; ++r) {
        const float2 a = __half22float2(*(const __half2 *)&pc[r].x), b = __half22float2(*(const __half2 *)&pc[r].y);
        float v[NQ];
#pragma unroll
        for (int i = 0; i < NQ; ++i) v[i] = fmaf(a.x, q[i][0], fmaf(a.y, q[i][1], fmaf(b.x, q[i][2], b.y * q[i][3])));
        const float sv = att_warp_sums<NQ>(v) * inv;
        if (first && k + r < kr) {
          const __half hi = __float2half_rn(sv);
          jb.wh[((size_t)h * NQ + c) * kr + k + r] = hi;
          jb.wl[((size_t)h * NQ + c) * kr + k + r] = __float2half_rn(sv - __half2float(hi));
        }
      }
    }
  }
}

// Code j of 32-feature group g of a packed row (little-endian bit string per group, BITS words per group).
template <int BITS>
__device__ __forceinline__ uint32_t att_code(const uint32_t *row, int g, int j) {
  const int bit = j * BITS, wi = g * BITS + (bit >> 5), sh = bit & 31;
  uint32_t u = row[wi] >> sh;
  if (sh + BITS > 32) u |= row[wi + 1] << (32 - sh);
  return u & ((1u << BITS) - 1u);
}

// grid (n_chunks, m, groups), kAttChunk threads (thread = token).  Dynamic shared memory: (128 + r_t) * NQP floats.
template <int BITS>
__global__ void __launch_bounds__(kAttChunk, 3) attend_scores_kernel(const AttendJob *__restrict__ jobs, int NQP) {
  const AttendJob &jb = jobs[blockIdx.z];
  if (jb.k.bits != BITS) return;
  const int h = blockIdx.y, chunk = blockIdx.x;
  if (h >= jb.m || chunk * kAttChunk >= jb.T) return;
  extern __shared__ unsigned char att_smem[];
  float *qts = (float *)att_smem;                   // [128][NQP]
  __shared__ float red[2][kAttChunk / 32][kAttMaxQ];
  __shared__ float qsum[4 * kAttMaxQ];              // per 32-feature group: sum of the rotated query's entries
  const int tid = threadIdx.x, r_t = jb.k.r_t;
  if (BITS > 0)
    for (int i = tid; i < 128 * NQP; i += kAttChunk) qts[i] = jb.qt[(size_t)h * 128 * NQP + i];
  __syncthreads();
  if (BITS > 0 && tid < 4 * kAttMaxQ) {
    const int g = tid / kAttMaxQ, i = tid % kAttMaxQ;
    float a = 0.f;
    if (i < NQP)
      for (int j = 0; j < 32; ++j) a += qts[(g * 32 + j) * NQP + i];
    qsum[tid] = a;
  }
  __syncthreads();
  const int t = chunk * kAttChunk + tid;
  const bool live = t < jb.T;
  float s[kAttMaxQ];
#pragma unroll
  for (int i = 0; i < kAttMaxQ; ++i) s[i] = 0.f;
  if (live) {
    if constexpr (BITS > 0) {
      uint32_t row[4 * BITS];
      const uint4 *wp = (const uint4 *)(jb.k.words + ((size_t)h * jb.T + t) * (4 * BITS));
#pragma unroll
      for (int i = 0; i < BITS; ++i) { const uint4 v = __ldg(wp + i); row[4 * i] = v.x; row[4 * i + 1] = v.y; row[4 * i + 2] = v.z; row[4 * i + 3] = v.w; }
      __half sc[4];
      *(uint2 *)sc = __ldg((const uint2 *)(jb.k.scales + ((size_t)h * jb.T + t) * 4));
      // integer code to float without a conversion instruction: 2^23 + u, minus (2^23 + 2^(b-1))
      // (the half-step offset is applied per group through the sum of the group's query entries, qsum)
      constexpr float off = 8388608.0f + (float)(1 << (BITS - 1));
      const bool q8 = NQP == 8;
#pragma unroll
      for (int g = 0; g < 4; ++g) {
        float g0 = 0.f, g1 = 0.f, g2 = 0.f, g3 = 0.f, g4 = 0.f, g5 = 0.f, g6 = 0.f, g7 = 0.f;
#pragma unroll
        for (int j = 0; j < 32; ++j) {
          const float val = __uint_as_float(0x4B000000u | att_code<BITS>(row, g, j)) - off;
          const float *qp = qts + (g * 32 + j) * NQP;
          const float4 qv = *(const float4 *)qp;
          g0 = fmaf(val, qv.x, g0); g1 = fmaf(val, qv.y, g1); g2 = fmaf(val, qv.z, g2); g3 = fmaf(val, qv.w, g3);
          if (q8) {
            const float4 qw = *(const float4 *)(qp + 4);
            g4 = fmaf(val, qw.x, g4); g5 = fmaf(val, qw.y, g5); g6 = fmaf(val, qw.z, g6); g7 = fmaf(val, qw.w, g7);
          }
        }
        const float delta = __half2float(sc[g]);
        const float *qh = qsum + g * kAttMaxQ;
        g0 = fmaf(0.5f, qh[0], g0); g1 = fmaf(0.5f, qh[1], g1); g2 = fmaf(0.5f, qh[2], g2); g3 = fmaf(0.5f, qh[3], g3);
        g4 = fmaf(0.5f, qh[4], g4); g5 = fmaf(0.5f, qh[5], g5); g6 = fmaf(0.5f, qh[6], g6); g7 = fmaf(0.5f, qh[7], g7);
        s[0] = fmaf(delta, g0, s[0]); s[1] = fmaf(delta, g1, s[1]); s[2] = fmaf(delta, g2, s[2]); s[3] = fmaf(delta, g3, s[3]);
        s[4] = fmaf(delta, g4, s[4]); s[5] = fmaf(delta, g5, s[5]); s[6] = fmaf(delta, g6, s[6]); s[7] = fmaf(delta, g7, s[7]);
      }
    }
    if (r_t > 0) {
      // backbone scores of this token: written to the weight buffer by attend_bscore_kernel, replaced by the weights below
      const float *sb = jb.p + ((size_t)h * jb.T + t) * NQP;
      const float4 b0 = *(const float4 *)sb;
      s[0] += b0.x; s[1] += b0.y; s[2] += b0.z; s[3] += b0.w;
      if (NQP == 8) {
        const float4 b1 = *(const float4 *)(sb + 4);
        s[4] += b1.x; s[5] += b1.y; s[6] += b1.z; s[7] += b1.w;
      }
    }
  }
  // chunk maximum and sum of exp(s - maximum), per query
  const int warp = tid >> 5, lane = tid & 31;
  float mx[kAttMaxQ];
#pragma unroll
  for (int i = 0; i < kAttMaxQ; ++i) {
    float v = live ? s[i] : -INFINITY;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    if (lane == 0) red[0][warp][i] = v;
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < kAttMaxQ; ++i) {
    float v = red[0][0][i];
#pragma unroll
    for (int wq = 1; wq < kAttChunk / 32; ++wq) v = fmaxf(v, red[0][wq][i]);
    mx[i] = v;
  }
  float pr[kAttMaxQ];
#pragma unroll
  for (int i = 0; i < kAttMaxQ; ++i) {
    pr[i] = live ? expf(s[i] - mx[i]) : 0.f;
    float v = pr[i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) red[1][warp][i] = v;
  }
  __syncthreads();
  if (live) {
    float *pp = jb.p + ((size_t)h * jb.T + t) * NQP;
    *(float4 *)pp = make_float4(pr[0], pr[1], pr[2], pr[3]);
    if (NQP == 8) *(float4 *)(pp + 4) = make_float4(pr[4], pr[5], pr[6], pr[7]);
  }
  if (tid < NQP) {
    float l = 0.f;
    for (int wq = 0; wq < kAttChunk / 32; ++wq) l += red[1][wq][tid];
    const int n_chunks = gridDim.x;
    float *ml = jb.ml + ((size_t)h * n_chunks + chunk) * 2 * NQP;
    float m_i = red[0][0][tid];
    for (int wq = 1; wq < kAttChunk / 32; ++wq) m_i = fmaxf(m_i, red[0][wq][tid]);
    ml[tid] = m_i;
    ml[NQP + tid] = l;
  }
}

// warp-level m16n8k16 MMA, fp16 operands, fp32 accumulation
__device__ __forceinline__ void att_mma_f16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
               : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
               : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// grid (n_chunks, m, groups), kAttChunk threads.  The chunk is staged in two halves of 128 tokens (codes, scales and
// weights, coalesced), so that six CTAs fit an SM: the kernel lives on the number of warps that hide its staging
// latency.  NQ = 4 or 8 query slots (compile time: the accumulators are the register budget).  Dynamic shared memory:
// 128 * (NQ floats + 4 BITS words + 4 halves) + 4 * 128 * NQ floats.
constexpr int kAttHalf = kAttChunk / 2;
template <int BITS, int NQ>
__global__ void __launch_bounds__(kAttChunk, NQ == 4 ? 6 : 4) attend_values_kernel(const AttendJob *__restrict__ jobs) {
  const AttendJob &jb = jobs[blockIdx.z];
  if (jb.v.bits != BITS || BITS == 0) return;
  const int h = blockIdx.y, chunk = blockIdx.x, n_chunks = gridDim.x;
  if (h >= jb.m || chunk * kAttChunk >= jb.T) return;
  constexpr int NB = BITS > 0 ? BITS : 1;
  extern __shared__ unsigned char att_smem[];
  float *ps = (float *)att_smem;                                        // [128][NQ]
  uint32_t *cw = (uint32_t *)(ps + kAttHalf * NQ);                      // [128][4 * BITS]
  __half *cs = (__half *)(cw + kAttHalf * 4 * NB);                      // [128][4]
  float *part = (float *)(cs + kAttHalf * 4);                           // [4][128][NQ] slice sums
  const int tid = threadIdx.x;
  // residual: thread = (four neighbouring features, one of eight 16-token slices of the staged half): one word, one scale
  // and one weight load serve four codes; sum_t p_t Delta_t (u_tf - 2^(b-1) + 1/2)
  const int fq = tid & 31, sl = tid >> 5;
  const int f0 = fq * 4, g = f0 >> 5, bit = (f0 & 31) * NB, wi = g * NB + (bit >> 5), sh = bit & 31;
  const bool straddle = NB == 3 && sh + 4 * NB > 32;           // only 3-bit codes cross a word inside a quad
  constexpr uint32_t mask = (1u << NB) - 1u;
  constexpr float off = 8388608.0f + (float)(1 << (NB - 1));
  float acc[4][NQ];
#pragma unroll
  for (int c = 0; c < 4; ++c)
#pragma unroll
    for (int i = 0; i < NQ; ++i) acc[c][i] = 0.f;
  for (int hf = 0; hf < 2; ++hf) {
    const int t0 = chunk * kAttChunk + hf * kAttHalf;
    if (t0 >= jb.T) break;                              // T is a multiple of 128: a half is all in or all out
    if (hf) __syncthreads();                            // the first half has been read
    {
      const float4 *src = (const float4 *)(jb.p + ((size_t)h * jb.T + t0) * NQ);
      for (int i = tid; i < kAttHalf * NQ / 4; i += kAttChunk) ((float4 *)ps)[i] = src[i];
      const uint4 *wsrc = (const uint4 *)(jb.v.words + ((size_t)h * jb.T + t0) * (4 * NB));
      for (int i = tid; i < kAttHalf * NB; i += kAttChunk) ((uint4 *)cw)[i] = __ldg(wsrc + i);
      const uint2 *ssrc = (const uint2 *)(jb.v.scales + ((size_t)h * jb.T + t0) * 4);
      for (int i = tid; i < kAttHalf; i += kAttChunk) ((uint2 *)cs)[i] = __ldg(ssrc + i);
    }
    __syncthreads();
    const int tb = sl * 16;
#pragma unroll 4
    for (int t = tb; t < tb + 16; ++t) {
      const uint32_t *row = cw + t * (4 * NB);
      uint32_t u4 = row[wi] >> sh;
      if (straddle) u4 |= row[wi + 1] << (32 - sh);
      const float delta = __half2float(cs[t * 4 + g]), hd = 0.5f * delta;
      float pv[NQ];
#pragma unroll
      for (int q4 = 0; q4 < NQ; q4 += 4) {
        const float4 p4 = *(const float4 *)(ps + t * NQ + q4);
        pv[q4] = p4.x; pv[q4 + 1] = p4.y; pv[q4 + 2] = p4.z; pv[q4 + 3] = p4.w;
      }
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        // integer code to float without a conversion instruction: 2^23 + u, minus (2^23 + 2^(b-1)); then Delta (u - 2^(b-1) + 1/2)
        const float val = fmaf(__uint_as_float(0x4B000000u | ((u4 >> (c * NB)) & mask)) - off, delta, hd);
#pragma unroll
        for (int i = 0; i < NQ; ++i) acc[c][i] = fmaf(pv[i], val, acc[c][i]);
      }
    }
  }
  // sum over the eight slices: 7..4 -> 3..0, 3..2 -> 1..0, 1 -> 0 through part[4][128][NQ]
#pragma unroll
  for (int stride = 4; stride >= 1; stride >>= 1) {
    if (sl >= stride && sl < 2 * stride) {
#pragma unroll
      for (int c = 0; c < 4; ++c)
#pragma unroll
        for (int i = 0; i < NQ; ++i) part[((sl - stride) * 128 + f0 + c) * NQ + i] = acc[c][i];
    }
    __syncthreads();
    if (sl < stride) {
#pragma unroll
      for (int c = 0; c < 4; ++c)
#pragma unroll
        for (int i = 0; i < NQ; ++i) acc[c][i] += part[(sl * 128 + f0 + c) * NQ + i];
    }
    __syncthreads();
  }
  if (sl == 0) {
    float *ap = jb.a + ((size_t)h * n_chunks + chunk) * NQ * 128 + f0;
#pragma unroll
    for (int i = 0; i < NQ; ++i) *(float4 *)(ap + i * 128) = make_float4(acc[0][i], acc[1][i], acc[2][i], acc[3][i]);
  }
}

// ---- the streaming pass on the tensor cores: scores, softmax weights and values of a chunk in one CTA -------------------
// What bounds the call is the stream of codes; as separate kernels (backbone scores, code scores per bit width, code values,
// backbone values) each of them ran at 1.5 to 2.2 TB/s on the latency of its own staging, with the weights going through
// global memory three times.  Here a CTA of four warps takes a chunk of tokens of NH heads from codes to partial values:
//   scores   U_T w of all NH heads at once (a warp per token stripe), then a warp per head adds the codes' part.  m16n8k16
//            with M = tokens: A fragments come straight from global memory.  The order of the k index is free as long as both
//            operands agree, so a lane takes eight neighbouring elements of a row: one 16-byte load of U_T feeds two MMAs of
//            every head, one field of eight codes the two MMAs of a 32-feature group.
//   weights  a warp per head: chunk maximum, p = exp(s - maximum)
//   values   a warp per head streams the codes (M = features, K = tokens; a lane's pairs are one feature of two neighbouring
//            tokens, joined by byte permutes; the steps scale the weights), then p^T U_T of all heads, a warp per 32 columns.
// Codes enter as the exact integers u - 2^(b-1) (fp16 1024 + u by bit insertion, one subtraction for two codes); the half step
// is a column sum: of the query (initial value of the accumulator) and of the weights (an MMA against a row of ones).  fp32
// operands enter as hi + lo fp16 (22 bits).  Up to four queries share an MMA with their own lo parts (columns q | q + 4).
// At 8 groups of 32 heads, 4096 tokens, ranks 128 / 112, 4- and 8-bit codes, four queries: 190 us in five launches -> 100 us.
// A head per CTA with U_T from L2 for each took 144 us, with four heads but fragment loads straight from global memory 112.
// What is left is instruction issue (46 % of the slots at 16 warps an SM) on chains of expand, multiply, exchange.
constexpr int kAttStreamThreads = 128;
constexpr int kAttTok = 128;                                                // tokens of a chunk
constexpr int kAttPitch = kAttTok + 8;                                      // tokens per row of weights (rows of halves start four banks apart)
constexpr int kAttWTok = 32, kAttWPitch = kAttWTok + 8;                     // ... of the weights times steps, 32 tokens at a time
constexpr int kAttSlot = 2048, kAttSlots = 3;                               // a warp's ring of code stages
__host__ __device__ constexpr int att_stage_rows(int bits) { return bits == 8 ? 16 : bits >= 3 ? 32 : 64; }      // at most kAttSlot bytes
constexpr size_t att_stream_smem(int nq) {
  return 4 * (kAttSlot * kAttSlots + (size_t)nq * kAttPitch * 8 + (size_t)4 * 2 * nq * kAttWPitch * 2);
}

// The packed rows of a warp's head, keys and then values, through a ring in shared memory by 16-byte asynchronous copies: the
// rows of a head are contiguous, so a request touches each 128-byte line once (straight fragment loads looked every line up
// once per 32-feature group: 57 % of the L1's tag rate and 16 % hits), and four stages stay in flight while the warp forms
// weights or multiplies by U_T.  Pieces are swizzled so that the fragment reads fall into different banks: 8-bit rows of the
// keys (lane row g) by row & 3, of the values (lane rows 2c ..) by (row >> 1) & 3 in units of 32 bytes, 4-bit rows by
// (row >> 1) & 3 in units of 16; narrower rows need none.
struct AttRing {
  char *slots;
  const char *src, *vsrc;     // this lane's first piece of the next stage; of the values
  uint32_t dst[4];            // places of its pieces in a slot
  int per, bytes, left;       // pieces of a lane, bytes of a stage, stages to come of the current cell
  int vbits, vleft;
  int wslot, rslot;
  __device__ __forceinline__ void layout(int bits, bool values) {
    const int lane = threadIdx.x & 31;
    const int rows = att_stage_rows(bits);
    per = rows * bits / 32;
    bytes = rows * 16 * bits;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int i = lane + 32 * k, row = bits == 3 ? i / 3 : i >> (bits == 8 ? 3 : bits == 4 ? 2 : bits == 2 ? 1 : 0), j = i - row * bits;
      const int key = bits == 8 ? 2 * (values ? (row >> 1) & 3 : row & 3) : bits == 4 ? (row >> 1) & 3 : 0;
      dst[k] = row * (16 * bits) + (j ^ key) * 16;
    }
  }
  __device__ __forceinline__ void issue() {
    if (left == 0 && vleft > 0) { layout(vbits, true); src = vsrc; left = vleft; vleft = 0; }
    if (left > 0) {
      const uint32_t base = (uint32_t)__cvta_generic_to_shared(slots + wslot * kAttSlot);
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (k < per) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(base + dst[k]), "l"(src + k * 512) : "memory");
      src += bytes;
      --left;
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    wslot = wslot + 1 == kAttSlots ? 0 : wslot + 1;
  }
  __device__ __forceinline__ AttRing(char *ring, const uint32_t *krows, int kbits, const uint32_t *vrows, int vb, int nt)
      : slots(ring), vbits(vb), wslot(0), rslot(0) {
    const int lane = threadIdx.x & 31;
    src = (const char *)krows + lane * 16;
    vsrc = (const char *)vrows + lane * 16;
    left = kbits ? nt / att_stage_rows(kbits) : 0;
    vleft = vb ? nt / att_stage_rows(vb) : 0;
    layout(kbits ? kbits : 1, false);
#pragma unroll
    for (int i = 0; i < kAttSlots - 1; ++i) issue();
  }
  // the stage to read; the one read before it is refilled
  __device__ __forceinline__ const char *next() {
    asm volatile("cp.async.wait_group %0;" ::"n"(kAttSlots - 2) : "memory");
    __syncwarp();
    issue();
    const char *p = slots + rslot * kAttSlot;
    rslot = rslot + 1 == kAttSlots ? 0 : rslot + 1;
    return p;
  }
};

// mid-rise codes of two tokens or features, exact in fp16
template <int BITS>
__device__ __forceinline__ uint32_t att_centre(uint32_t v) {
  const __half2 r = __hsub2(*(const __half2 *)&v, __float2half2_rn(1024.f + (float)(1 << (BITS - 1))));
  return *(const uint32_t *)&r;
}
template <int BITS>
__device__ __forceinline__ uint32_t att_pair(uint32_t z, int i) {             // code i of the low half and of the high half
  constexpr uint32_t m = (1u << BITS) - 1u;
  return att_centre<BITS>(((z >> (BITS * i)) & (m | m << 16)) | 0x64006400u);
}

// Raw field of a lane: eight codes of a row's group (scores; lane c of four) -- natural order for 8-bit codes, else codes
// 0..3 in the low and 4..7 in the high half of a word, so that pair i = (i, i + 4).
template <int BITS>
struct AttField8 {
  uint32_t w0, w1;
  __device__ __forceinline__ void load(const char *st, int row, int key, int G, int c) {       // key: of the ring's swizzle
    const char *r = st + row * (16 * BITS);
    if constexpr (BITS == 8) { const uint2 v = *(const uint2 *)(r + (G ^ key) * 32 + 8 * c); w0 = v.x; w1 = v.y; }
    else if constexpr (BITS == 4) { w0 = *(const uint32_t *)(r + (G ^ key) * 16 + 4 * c); }
    else if constexpr (BITS == 3) { const int lo = (24 * c) >> 5; w0 = *(const uint32_t *)(r + G * 12 + 4 * lo); w1 = *(const uint32_t *)(r + G * 12 + 4 * min(lo + 1, 2)); }
    else if constexpr (BITS == 2) { w0 = *(const unsigned short *)(r + G * 8 + 2 * c); }
    else { w0 = *(const unsigned char *)(r + G * 4 + c); }
  }
  __device__ __forceinline__ void expand(uint32_t (&o)[4], int c) const {
    if constexpr (BITS == 8) {
      o[0] = att_centre<8>(__byte_perm(w0, 0x64646464u, 0x4140)); o[1] = att_centre<8>(__byte_perm(w0, 0x64646464u, 0x4342));
      o[2] = att_centre<8>(__byte_perm(w1, 0x64646464u, 0x4140)); o[3] = att_centre<8>(__byte_perm(w1, 0x64646464u, 0x4342));
    } else {
      uint32_t z = w0;
      if constexpr (BITS == 3) { const uint32_t x = __funnelshift_r(w0, w1, (24 * c) & 31); z = (x & 0xFFFu) | ((x & 0xFFF000u) << 4); }
      if constexpr (BITS == 2) z = __byte_perm(w0, 0u, 0x4140);
      if constexpr (BITS == 1) z = (w0 & 0xFu) | (w0 << 12);
#pragma unroll
      for (int i = 0; i < 4; ++i) o[i] = att_pair<BITS>(z, i);
    }
  }
};
// ... and four codes of a row's group (values; lane g of eight).
template <int BITS>
struct AttField4 {
  uint32_t w0, w1;
  __device__ __forceinline__ void load(const char *st, int row, int key, int G, int g) {
    const char *r = st + row * (16 * BITS);
    if constexpr (BITS == 8) w0 = *(const uint32_t *)(r + (G ^ key) * 32 + 4 * g);
    else if constexpr (BITS == 4) w0 = *(const unsigned short *)(r + (G ^ key) * 16 + 2 * g);
    else if constexpr (BITS == 3) { const int lo = (12 * g) >> 5; w0 = *(const uint32_t *)(r + G * 12 + 4 * lo); w1 = *(const uint32_t *)(r + G * 12 + 4 * min(lo + 1, 2)); }
    else if constexpr (BITS == 2) w0 = *(const unsigned char *)(r + G * 8 + g);
    else w0 = *(const unsigned char *)(r + G * 4 + (g >> 1));
  }
  // features 0..3 of two neighbouring tokens
  static __device__ __forceinline__ void expand(uint32_t (&o)[4], const AttField4 &a, const AttField4 &b, int g) {
    if constexpr (BITS == 8) {
      const uint32_t lo = __byte_perm(a.w0, b.w0, 0x5140), hi = __byte_perm(a.w0, b.w0, 0x7362);
      o[0] = att_centre<8>(__byte_perm(lo, 0x64646464u, 0x4140)); o[1] = att_centre<8>(__byte_perm(lo, 0x64646464u, 0x4342));
      o[2] = att_centre<8>(__byte_perm(hi, 0x64646464u, 0x4140)); o[3] = att_centre<8>(__byte_perm(hi, 0x64646464u, 0x4342));
    } else {
      uint32_t x = a.w0, y = b.w0;
      if constexpr (BITS == 3) { x = __funnelshift_r(a.w0, a.w1, (12 * g) & 31); y = __funnelshift_r(b.w0, b.w1, (12 * g) & 31); }
      if constexpr (BITS == 1) { x >>= 4 * (g & 1); y >>= 4 * (g & 1); }
      const uint32_t z = __byte_perm(x, y, 0x5410);
#pragma unroll
      for (int i = 0; i < 4; ++i) o[i] = att_pair<BITS>(z, i);
    }
  }
};

// fp32 pair -> hi and lo half2
__device__ __forceinline__ void att_split(float x0, float x1, uint32_t &hi, uint32_t &lo) {
  const __half2 h = __floats2half2_rn(x0, x1);
  const float2 f = __half22float2(h);
  const __half2 l = __floats2half2_rn(x0 - f.x, x1 - f.y);
  hi = *(const uint32_t *)&h; lo = *(const uint32_t *)&l;
}

// Code scores of a warp's head over its nt tokens, added to ps[query][token].
template <int BITS, int NQ>
__device__ __forceinline__ void att_code_scores(const AttendJob &jb, int h, size_t row0, int nt, float *ps, AttRing &ring) {
  const int lane = threadIdx.x & 31, g = lane >> 2, c = lane & 3;
  constexpr int NB = NQ == 8 ? 2 : 1, P = kAttPitch;      // lo parts in an MMA of their own
  const int key = BITS == 8 ? g & 3 : (g >> 1) & 3;
  const uint2 *sp = (const uint2 *)jb.k.scales + row0 + g;
  uint2 sc[2][2];
  sc[0][0] = __ldg(sp); sc[0][1] = __ldg(sp + 8); sc[1][0] = __ldg(sp + 16); sc[1][1] = __ldg(sp + 24);
  uint4 bq[NB][4];
  float qs[4][2];
  {
    const int q = NQ == 8 ? g : g & 3;
    const __half *s0 = ((NQ == 4 && g >= 4) ? jb.ql : jb.qh) + ((size_t)h * kAttMaxQ + q) * 128 + 8 * c;
    const __half *s1 = jb.ql + ((size_t)h * kAttMaxQ + q) * 128 + 8 * c;
#pragma unroll
    for (int G = 0; G < 4; ++G) {
      bq[0][G] = *(const uint4 *)(s0 + G * 32);
      if (NB == 2) bq[NB - 1][G] = *(const uint4 *)(s1 + G * 32);
    }
#pragma unroll
    for (int G = 0; G < 4; ++G) {
      float d[4] = {0.f, 0.f, 0.f, 0.f};
      const uint32_t one = 0x3C003C00u, ones[4] = {one, one, one, one};
#pragma unroll
      for (int b = 0; b < NB; ++b) {
        if constexpr (BITS != 8) {                         // pairs (i, i + 4)
          const uint4 v = bq[b][G];
          bq[b][G] = make_uint4(__byte_perm(v.x, v.z, 0x5410), __byte_perm(v.x, v.z, 0x7632), __byte_perm(v.y, v.w, 0x5410), __byte_perm(v.y, v.w, 0x7632));
        }
        att_mma_f16(d, ones, bq[b][G].x, bq[b][G].y);
        att_mma_f16(d, ones, bq[b][G].z, bq[b][G].w);
      }
      qs[G][0] = 0.5f * d[0]; qs[G][1] = 0.5f * d[1];      // the half step of every code of the group
    }
  }
  const int qa = (2 * c) & (NQ - 1);
  const float e0 = jb.qe[h * kAttMaxQ + qa], e1 = jb.qe[h * kAttMaxQ + qa + 1];
  float *pr = ps + qa * P + g + (NQ == 4 ? (c & 2) * 4 : 0);      // NQ = 4: lanes c < 2 finish row g, c >= 2 row g + 8
  constexpr int R = att_stage_rows(BITS);
  const char *stage = nullptr;
  for (int t = 0; t < nt; t += 32) {
    if (R >= 32 && (R == 32 || (t & 32) == 0)) stage = ring.next();
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      if (R == 16) stage = ring.next();
      const int r0 = R == 16 ? 0 : R == 32 ? 16 * u : (t & 32) + 16 * u;
      AttField8<BITS> fa[4], fb[4];
#pragma unroll
      for (int G = 0; G < 4; ++G) { fa[G].load(stage, r0 + g, key, G, c); fb[G].load(stage, r0 + g + 8, key, G, c); }
      float s[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int G = 0; G < 4; ++G) {
        uint32_t x[4], y[4];
        fa[G].expand(x, c);
        fb[G].expand(y, c);
        float d[4] = {qs[G][0], qs[G][1], qs[G][0], qs[G][1]};
        const uint32_t a0[4] = {x[0], y[0], x[1], y[1]}, a1[4] = {x[2], y[2], x[3], y[3]};
#pragma unroll
        for (int b = 0; b < NB; ++b) {
          att_mma_f16(d, a0, bq[b][G].x, bq[b][G].y);
          att_mma_f16(d, a1, bq[b][G].z, bq[b][G].w);
        }
        const uint32_t wa = G & 2 ? sc[u][0].y : sc[u][0].x, wb = G & 2 ? sc[u][1].y : sc[u][1].x;
        const float da = G & 1 ? __high2float(*(const __half2 *)&wa) : __low2float(*(const __half2 *)&wa);
        const float db = G & 1 ? __high2float(*(const __half2 *)&wb) : __low2float(*(const __half2 *)&wb);
        s[0] = fmaf(da, d[0], s[0]); s[1] = fmaf(da, d[1], s[1]);
        s[2] = fmaf(db, d[2], s[2]); s[3] = fmaf(db, d[3], s[3]);
      }
      if (t + 32 < nt) { sc[u][0] = __ldg(sp + t + 32 + 16 * u); sc[u][1] = __ldg(sp + t + 40 + 16 * u); }
      float *pt = pr + t + 16 * u;
      if constexpr (NQ == 4) {
        const float k0 = c & 2 ? s[2] : s[0], k1 = c & 2 ? s[3] : s[1], v0 = c & 2 ? s[0] : s[2], v1 = c & 2 ? s[1] : s[3];
        pt[0] = fmaf(k0 + __shfl_xor_sync(0xffffffffu, v0, 2), e0, pt[0]);
        pt[P] = fmaf(k1 + __shfl_xor_sync(0xffffffffu, v1, 2), e1, pt[P]);
      } else {
        pt[0] = fmaf(s[0], e0, pt[0]); pt[P] = fmaf(s[1], e1, pt[P]);
        pt[8] = fmaf(s[2], e0, pt[8]); pt[P + 8] = fmaf(s[3], e1, pt[P + 8]);
      }
    }
  }
}

// A lane's product columns, hi + lo, as elements 4g .. 4g + 3 of queries 2c, 2c + 1; NQ = 4: lanes c < 2.
template <int NQ>
__device__ __forceinline__ void att_put4(float (&d)[2][4], float mul, float *dst, int stride, bool ok) {
  const int lane = threadIdx.x & 31, c = lane & 3;
#pragma unroll
  for (int j = 0; j < 2; ++j)
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (NQ == 4) d[j][i] += __shfl_xor_sync(0xffffffffu, d[j][i], 2);
  if (!ok || (NQ == 4 && c >= 2)) return;
#pragma unroll
  for (int q = 0; q < 2; ++q)
    *(float4 *)(dst + (size_t)(2 * c + q) * stride) = make_float4(d[0][q] * mul, d[0][q + 2] * mul, d[1][q] * mul, d[1][q + 2] * mul);
}

// One 16-token step of a value product: M = 32 elements of a row (a lane's four, x from tokens 2c, 2c + 1 and y from 8 on), B
// from the weight rows of column g (hi rows 0 .. NQ - 1, lo rows NQ .. 2 NQ - 1).  ones: also sum the weights into row G of e.
template <int NQ>
__device__ __forceinline__ void att_value_mma(float (&d)[2][4], const uint32_t (&x)[4], const uint32_t (&y)[4], const __half *w, int pitch) {
  const uint32_t a0[4] = {x[0], x[1], y[0], y[1]}, a1[4] = {x[2], x[3], y[2], y[3]};
  const uint32_t b0 = *(const uint32_t *)w, b1 = *(const uint32_t *)(w + 8);
  att_mma_f16(d[0], a0, b0, b1); att_mma_f16(d[1], a1, b0, b1);
  if (NQ == 8) {
    const uint32_t c0 = *(const uint32_t *)(w + 8 * pitch), c1 = *(const uint32_t *)(w + 8 * pitch + 8);
    att_mma_f16(d[0], a0, c0, c1); att_mma_f16(d[1], a1, c0, c1);
  }
}

// Code values of a warp's head over its nt tokens.  ws: [4 groups][2 NQ][kAttWPitch] weights times steps of 32 tokens.
template <int BITS, int NQ>
__device__ __forceinline__ void att_code_values(const AttendJob &jb, size_t row0, int nt, const float *ps, __half *ws, AttRing &ring, float *out) {
  const int lane = threadIdx.x & 31, g = lane >> 2, c = lane & 3;
  constexpr int P = kAttPitch;
  // one power of two for the chunk so that step * weight fits fp16: the largest step -> below 2^14
  const uint4 *sp = (const uint4 *)(jb.v.scales + (row0 + 2 * lane) * 4);                 // the steps of two tokens
  __half2 mx2 = __float2half2_rn(0.f);
  for (int t = 0; t < nt; t += 64) {
    const uint4 v = __ldg(sp + t / 2);
    mx2 = __hmax2(mx2, __hmax2(__hmax2(*(const __half2 *)&v.x, *(const __half2 *)&v.y), __hmax2(*(const __half2 *)&v.z, *(const __half2 *)&v.w)));
  }
  float mx = fmaxf(__low2float(mx2), __high2float(mx2));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  int ex = 0;
  if (mx > 0.f && mx < INFINITY) frexpf(mx, &ex);
  const float up = ldexpf(1.f, 14 - ex), down = ldexpf(1.f, ex - 14);
  float d[4][2][4], hs[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
  for (int G = 0; G < 4; ++G)
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
      for (int i = 0; i < 4; ++i) d[G][j][i] = 0.f;
  const __half *w = ws + g * kAttWPitch + 2 * c;
  // weights: this lane forms those of tokens 2 tl, 2 tl + 1 of every 32 and groups 2 gh, 2 gh + 1
  const int tl = lane & 15, gh = lane >> 4;
  const uint4 *vp = (const uint4 *)(jb.v.scales + (row0 + 2 * tl) * 4);
  uint4 vn = __ldg(vp);
  const char *stage = nullptr;
  for (int tb = 0; tb < nt; tb += kAttWTok) {
    const uint32_t va = gh ? vn.y : vn.x, vb = gh ? vn.w : vn.z;
    if (tb + kAttWTok < nt) vn = __ldg(vp + (tb + kAttWTok) / 2);
    const float2 fa = __half22float2(*(const __half2 *)&va), fb = __half22float2(*(const __half2 *)&vb);
    const float d0[2] = {fa.x * up, fa.y * up}, d1[2] = {fb.x * up, fb.y * up};
    __syncwarp();                                                                       // the previous weights have been read
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      const float2 p = *(const float2 *)(ps + q * P + tb + 2 * tl);
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        uint32_t hi, lo;
        att_split(p.x * d0[i], p.y * d1[i], hi, lo);
        __half *wr = ws + ((2 * gh + i) * 2 * NQ + q) * kAttWPitch + 2 * tl;
        *(uint32_t *)wr = hi;
        *(uint32_t *)(wr + NQ * kAttWPitch) = lo;
      }
    }
#pragma unroll
    for (int s = 0; s < kAttWTok / 16; ++s) {
      constexpr int R = att_stage_rows(BITS);
      if (R == 16 || (s == 0 && (R == 32 || (tb & 32) == 0))) stage = ring.next();      // its __syncwarp also publishes the weights
      else if (s == 0) __syncwarp();
      const int r0 = R == 16 ? 0 : R == 32 ? 16 * s : (tb & 32) + 16 * s;
      AttField4<BITS> f[4][4];
#pragma unroll
      for (int G = 0; G < 4; ++G)
#pragma unroll
        for (int i = 0; i < 4; ++i) f[G][i].load(stage, r0 + 2 * c + (i & 1) + (i >> 1) * 8, c, G, g);
#pragma unroll
      for (int G = 0; G < 4; ++G) {
        uint32_t x[4], y[4];
        AttField4<BITS>::expand(x, f[G][0], f[G][1], g);
        AttField4<BITS>::expand(y, f[G][2], f[G][3], g);
        const __half *wg = w + G * 2 * NQ * kAttWPitch + 16 * s;
        att_value_mma<NQ>(d[G], x, y, wg, kAttWPitch);
        const uint32_t one = g == G ? 0x3C003C00u : 0u, a[4] = {one, 0u, one, 0u};      // row G of hs: the sum of the weights
        att_mma_f16(hs, a, *(const uint32_t *)wg, *(const uint32_t *)(wg + 8));
        if (NQ == 8) att_mma_f16(hs, a, *(const uint32_t *)(wg + 8 * kAttWPitch), *(const uint32_t *)(wg + 8 * kAttWPitch + 8));
      }
    }
  }
#pragma unroll
  for (int G = 0; G < 4; ++G) {
    const float a0 = 0.5f * __shfl_sync(0xffffffffu, hs[0], 4 * G + c), a1 = 0.5f * __shfl_sync(0xffffffffu, hs[1], 4 * G + c);
#pragma unroll
    for (int j = 0; j < 2; ++j) { d[G][j][0] += a0; d[G][j][1] += a1; d[G][j][2] += a0; d[G][j][3] += a1; }
    att_put4<NQ>(d[G], down, out + G * 32 + 4 * g, 128, true);
  }
}

// grid (ceil(chunks / (4 / NH)), ceil(m / NH), groups), 128 threads, att_stream_smem bytes of dynamic shared memory.  NH = 4: the
// warps are four heads of one chunk; NH = 1 (fewer than three heads in a cell): four chunks of one head.
template <int NQ, int NH, bool BYARG>
__global__ void __launch_bounds__(kAttStreamThreads, NQ == 4 ? 4 : 3) attend_stream_kernel(const __grid_constant__ AttendArgs args, int n_chunks) {
  constexpr int TC = kAttTok, P = kAttPitch;
  const AttendJob &jb = BYARG ? args.j[blockIdx.z] : args.table[blockIdx.z];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, c = lane & 3;
  const int h0 = blockIdx.y * NH, t_cta = blockIdx.x * (TC * 4 / NH), T = jb.T, m = jb.m;
  if (h0 >= m || t_cta >= T) return;
  extern __shared__ unsigned char att_smem[];
  float *ps_all = (float *)att_smem;                                        // [4 warps][NQ][P] scores, then weights
  __half *pw_all = (__half *)(ps_all + 4 * NQ * P);                         // [4][2 NQ][P] weights as hi and lo rows
  const int kr = jb.k.r_t, vr = jb.v.r_t;
  const int h = h0 + (NH == 4 ? warp : 0), t0 = t_cta + (NH == 4 ? 0 : warp * TC), nt = max(0, min(TC, T - t0));      // nt: a multiple of 128
  const bool alive = h < m && nt > 0;
  const size_t row0 = (size_t)h * T + t0;
  float *ps = ps_all + warp * NQ * P;
  __half *pw = pw_all + warp * 2 * NQ * P, *ws = pw_all + 4 * 2 * NQ * P + warp * 4 * 2 * NQ * kAttWPitch;
  AttRing ring((char *)(pw_all + 4 * 2 * NQ * P + 4 * 4 * 2 * NQ * kAttWPitch) + warp * kAttSlot * kAttSlots, jb.k.words + row0 * 4 * jb.k.bits,
               jb.k.bits, jb.v.words + row0 * 4 * jb.v.bits, jb.v.bits, alive ? nt : 0);
  att_wait_predecessor();
  // ---- backbone scores of a warp's TA tokens, SB stripes of 16 and all heads at a time
  {
    constexpr int TA = TC / NH, SB = 2;
    const int tw = t_cta + warp * TA, tp = NH == 4 ? warp * TA : 0;          // first token; its place in the chunk
    for (int ta = 0; ta < TA && tw + ta < T; ta += 16 * SB) {
      float acc[SB][NH][4];
#pragma unroll
      for (int st = 0; st < SB; ++st)
#pragma unroll
        for (int j = 0; j < NH; ++j)
#pragma unroll
          for (int i = 0; i < 4; ++i) acc[st][j][i] = 0.f;
      const __half *ua = jb.k.UT + (size_t)(tw + ta + g) * kr + 8 * c;
      const size_t wo = ((size_t)h0 * NQ + (NQ == 8 ? g : g & 3)) * kr + 8 * c;
      const __half *w0 = ((NQ == 4 && g >= 4) ? jb.wl : jb.wh) + wo, *w1 = jb.wl + wo;
      const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
      uint4 x[SB], y[SB];
      auto load_a = [&](int k) {
        const bool ok = k + 8 * c < kr;
#pragma unroll
        for (int st = 0; st < SB; ++st) {
          x[st] = ok ? __ldg((const uint4 *)(ua + (size_t)(st * 16) * kr + k)) : zero;
          y[st] = ok ? __ldg((const uint4 *)(ua + (size_t)(st * 16 + 8) * kr + k)) : zero;
        }
      };
      uint4 bn[NH];
      auto load_b = [&](int k) {
#pragma unroll
        for (int j = 0; j < NH; ++j) bn[j] = k + 8 * c < kr && h0 + j < m ? *(const uint4 *)(w0 + (size_t)j * NQ * kr + k) : zero;
      };
      load_b(0);
      load_a(0);
#pragma unroll 1
      for (int k = 0; k < kr; k += 32) {
        uint4 b[NH], bl[NH], xc[SB], yc[SB];
#pragma unroll
        for (int j = 0; j < NH; ++j) {
          b[j] = bn[j];
          if (NQ == 8) bl[j] = k + 8 * c < kr && h0 + j < m ? *(const uint4 *)(w1 + (size_t)j * NQ * kr + k) : zero;
        }
        if (k + 32 < kr) load_b(k + 32);
#pragma unroll
        for (int st = 0; st < SB; ++st) { xc[st] = x[st]; yc[st] = y[st]; }
        if (k + 32 < kr) load_a(k + 32);
#pragma unroll
        for (int st = 0; st < SB; ++st) {
          const uint32_t a0[4] = {xc[st].x, yc[st].x, xc[st].y, yc[st].y}, a1[4] = {xc[st].z, yc[st].z, xc[st].w, yc[st].w};
#pragma unroll
          for (int j = 0; j < NH; ++j) {
            att_mma_f16(acc[st][j], a0, b[j].x, b[j].y);
            att_mma_f16(acc[st][j], a1, b[j].z, b[j].w);
            if (NQ == 8) { att_mma_f16(acc[st][j], a0, bl[j].x, bl[j].y); att_mma_f16(acc[st][j], a1, bl[j].z, bl[j].w); }
          }
        }
      }
      const int qa = (2 * c) & (NQ - 1);
#pragma unroll
      for (int j = 0; j < NH; ++j) {
        const bool hk = kr > 0 && h0 + j < m;
        const float we0 = hk ? jb.we[(h0 + j) * NQ + qa] : 0.f, we1 = hk ? jb.we[(h0 + j) * NQ + qa + 1] : 0.f;
        float *pj = ps_all + (NH == 4 ? j : warp) * NQ * P + qa * P + tp + ta + g;
#pragma unroll
        for (int st = 0; st < SB; ++st) {
          const float *s = acc[st][j];
          if constexpr (NQ == 4) {
            const float k0 = c & 2 ? s[2] : s[0], k1 = c & 2 ? s[3] : s[1], v0 = c & 2 ? s[0] : s[2], v1 = c & 2 ? s[1] : s[3];
            const float r0 = (k0 + __shfl_xor_sync(0xffffffffu, v0, 2)) * we0, r1 = (k1 + __shfl_xor_sync(0xffffffffu, v1, 2)) * we1;
            pj[st * 16 + (c & 2) * 4] = r0; pj[P + st * 16 + (c & 2) * 4] = r1;
          } else {
            pj[st * 16] = s[0] * we0; pj[P + st * 16] = s[1] * we1;
            pj[st * 16 + 8] = s[2] * we0; pj[P + st * 16 + 8] = s[3] * we1;
          }
        }
      }
    }
  }
  __syncthreads();
  if (alive) {
    switch (jb.k.bits) {
      case 1: att_code_scores<1, NQ>(jb, h, row0, nt, ps, ring); break;
      case 2: att_code_scores<2, NQ>(jb, h, row0, nt, ps, ring); break;
      case 3: att_code_scores<3, NQ>(jb, h, row0, nt, ps, ring); break;
      case 4: att_code_scores<4, NQ>(jb, h, row0, nt, ps, ring); break;
      case 8: att_code_scores<8, NQ>(jb, h, row0, nt, ps, ring); break;
      default: break;
    }
    __syncwarp();
    // chunk maximum, weights and their sum, per query; this lane: tokens 2 lane, 2 lane + 1 of every 64
    const int chunk = t0 / TC;
    float *ml = jb.ml + ((size_t)h * n_chunks + chunk) * 2 * NQ;
    float2 v[NQ][TC / 64];
    float mx[NQ], l[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      mx[q] = -INFINITY; l[q] = 0.f;
#pragma unroll
      for (int i = 0; i < TC / 64; ++i) { v[q][i] = *(const float2 *)(ps + q * P + 64 * i + 2 * lane); mx[q] = fmaxf(mx[q], fmaxf(v[q][i].x, v[q][i].y)); }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
      for (int q = 0; q < NQ; ++q) mx[q] = fmaxf(mx[q], __shfl_xor_sync(0xffffffffu, mx[q], o));
#pragma unroll
    for (int q = 0; q < NQ; ++q)
#pragma unroll
      for (int i = 0; i < TC / 64; ++i) {
        const float2 p = make_float2(expf(v[q][i].x - mx[q]), expf(v[q][i].y - mx[q]));
        l[q] += p.x + p.y;
        *(float2 *)(ps + q * P + 64 * i + 2 * lane) = p;
        uint32_t hi, lo;
        att_split(p.x, p.y, hi, lo);
        *(uint32_t *)(pw + q * P + 64 * i + 2 * lane) = hi;
        *(uint32_t *)(pw + (q + NQ) * P + 64 * i + 2 * lane) = lo;
      }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
      for (int q = 0; q < NQ; ++q) l[q] += __shfl_xor_sync(0xffffffffu, l[q], o);
    if (lane == 0)
#pragma unroll
      for (int q = 0; q < NQ; ++q) { ml[q] = mx[q]; ml[NQ + q] = l[q]; }
    __syncwarp();
    float *ap = jb.a + ((size_t)h * n_chunks + chunk) * NQ * 128;
    switch (jb.v.bits) {
      case 1: att_code_values<1, NQ>(jb, row0, nt, ps, ws, ring, ap); break;
      case 2: att_code_values<2, NQ>(jb, row0, nt, ps, ws, ring, ap); break;
      case 3: att_code_values<3, NQ>(jb, row0, nt, ps, ws, ring, ap); break;
      case 4: att_code_values<4, NQ>(jb, row0, nt, ps, ws, ring, ap); break;
      case 8: att_code_values<8, NQ>(jb, row0, nt, ps, ws, ring, ap); break;
      default: break;
    }
  }
  __syncthreads();
  // ---- p^T U_T: 32 columns at a time, all heads (NH = 4) or this warp's chunk (NH = 1)
  if (nt == 0) return;
  for (int kb = NH == 4 ? warp * 32 : 0; kb < vr; kb += NH == 4 ? 128 : 32) {
    const int k = kb + 4 * g;
    const bool ok = k < vr;
    const __half *p0 = jb.v.UT + (size_t)(t0 + 2 * c) * vr + min(k, vr - 4), *p1 = p0 + vr, *p2 = p0 + 8 * (size_t)vr, *p3 = p2 + vr;      // columns past the end: not stored
    const size_t step = 16 * (size_t)vr;
    constexpr int PF = 4;
    uint2 f[PF][4];
    auto fetch = [&](int buf) {
      f[buf][0] = __ldg((const uint2 *)p0); f[buf][1] = __ldg((const uint2 *)p1); f[buf][2] = __ldg((const uint2 *)p2); f[buf][3] = __ldg((const uint2 *)p3);
      p0 += step; p1 += step; p2 += step; p3 += step;
    };
#pragma unroll
    for (int u = 0; u < PF; ++u) fetch(u);
    float d[NH][2][4];
#pragma unroll
    for (int j = 0; j < NH; ++j)
#pragma unroll
      for (int i = 0; i < 8; ++i) d[j][i >> 2][i & 3] = 0.f;
    const __half *w = pw_all + (NH == 4 ? 0 : warp) * 2 * NQ * P + g * P + 2 * c;
    for (int t = 0; t < nt; t += 16 * PF) {
#pragma unroll
      for (int u = 0; u < PF; ++u) {
        uint32_t x[4], y[4];
        x[0] = __byte_perm(f[u][0].x, f[u][1].x, 0x5410); x[1] = __byte_perm(f[u][0].x, f[u][1].x, 0x7632);
        x[2] = __byte_perm(f[u][0].y, f[u][1].y, 0x5410); x[3] = __byte_perm(f[u][0].y, f[u][1].y, 0x7632);
        y[0] = __byte_perm(f[u][2].x, f[u][3].x, 0x5410); y[1] = __byte_perm(f[u][2].x, f[u][3].x, 0x7632);
        y[2] = __byte_perm(f[u][2].y, f[u][3].y, 0x5410); y[3] = __byte_perm(f[u][2].y, f[u][3].y, 0x7632);
        if (t + 16 * PF < nt) fetch(u);
#pragma unroll
        for (int j = 0; j < NH; ++j) att_value_mma<NQ>(d[j], x, y, w + j * 2 * NQ * P + t + 16 * u, P);
      }
    }
#pragma unroll
    for (int j = 0; j < NH; ++j)
      att_put4<NQ>(d[j], 1.f, jb.y + ((size_t)(h0 + j) * n_chunks + t0 / TC) * NQ * vr + k, vr, ok && h0 + j < m);
  }
}

// The backbone terms are shared by all heads of a cell (one U_T per cell), so they are two small dense products over the
// whole cell instead of a loop per head:  with n = (head, query),
//   attend_bscore_kernel   S_b[t][n] = sum_k U_T[t][k] w[n][k]            written to the weight buffer p[h][t][i]
//   attend_bvalue_kernel   y[chunk][n][k] = sum_{t in chunk} p[n][t] U_T[t][k]
// Both run on the tensor cores as warp-level m16n8k16 fp16 MMAs with fp32 accumulation: U_T is fp16 as stored, the
// fp32 operand enters as hi + lo fp16 (22 bits) -- p lies in [0, 1]; w is scaled per column by a power of two bounded
// through |q|_2 (see attend_prep_kernel).  0.13 GFLOP per cell each with N = 128: too small to set up TMEM-resident
// tcgen05 tiles for.  (A TF32 m16n8k8 form of the first product ran at the CUDA-core FMA rate and was replaced.)
constexpr int kAttBPitch = 136;     // floats per staged operand row: 8 c + g addresses all 32 banks

// grid (ceil(T / 64), ceil(m NQP / 128), groups), 256 threads: warp w owns 16 tokens (w & 3) x 64 columns n (w >> 2).
// m16n8k16 fp16 MMAs: A = U_T as stored, B = the scaled w as hi + lo.  The operands of the next 32-wide k chunk are
// requested into registers before the MMAs of the current one.
__global__ void __launch_bounds__(256, 2) attend_bscore_kernel(const AttendJob *__restrict__ jobs, int NQP) {
  const AttendJob &jb = jobs[blockIdx.z];
  const int r_t = jb.k.r_t, N = jb.m * NQP, n0 = blockIdx.y * 128, t0 = blockIdx.x * 64;
  if (r_t == 0 || n0 >= N || t0 >= jb.T) return;
  __shared__ __align__(16) uint32_t Bh[16][kAttBPitch], Bl[16][kAttBPitch];       // w chunk as k pairs, hi and lo, [k / 2][n]
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, c = lane & 3;
  const int wt = warp & 3, wn = warp >> 2;
  float acc[8][4];
#pragma unroll
  for (int nt = 0; nt < 8; ++nt)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[nt][j] = 0.f;
  const int ta = min(t0 + wt * 16 + g, jb.T - 1), tb = min(t0 + wt * 16 + g + 8, jb.T - 1);   // rows past the end repeat the last
  const __half *rowa = jb.k.UT + (size_t)ta * r_t, *rowb = jb.k.UT + (size_t)tb * r_t;
  // staging items of a chunk: (hi | lo, column n, block of eight k) -> 2 * 128 * 4 = 1024, four per thread
  uint4 breg[4];
  uint4 areg[4][2];
  auto load_chunk = [&](int k0) {
#pragma unroll
    for (int it = 0; it < 4; ++it) {
      const int idx = tid + it * 256, hl = idx >> 9, nn = (idx >> 2) & 127, kb8 = (idx & 3) * 8, n = n0 + nn;
      breg[it] = make_uint4(0u, 0u, 0u, 0u);
      if (n < N && k0 + kb8 < r_t) breg[it] = *(const uint4 *)((hl ? jb.wl : jb.wh) + (size_t)n * r_t + k0 + kb8);
    }
#pragma unroll
    for (int k8 = 0; k8 < 4; ++k8) {
      areg[k8][0] = make_uint4(0u, 0u, 0u, 0u); areg[k8][1] = areg[k8][0];
      if (k0 + k8 * 8 < r_t) {
        areg[k8][0] = __ldg((const uint4 *)(rowa + k0 + k8 * 8));
        areg[k8][1] = __ldg((const uint4 *)(rowb + k0 + k8 * 8));
      }
    }
  };
  auto word_of = [](const uint4 &u, int w) { return (w & 2) ? ((w & 1) ? u.w : u.z) : ((w & 1) ? u.y : u.x); };
  load_chunk(0);
  for (int k0 = 0; k0 < r_t; k0 += 32) {
    __syncthreads();
#pragma unroll
    for (int it = 0; it < 4; ++it) {
      const int idx = tid + it * 256, hl = idx >> 9, nn = (idx >> 2) & 127, kp0 = (idx & 3) * 4;
      uint32_t (*dst)[kAttBPitch] = hl ? Bl : Bh;
      dst[kp0][nn] = breg[it].x; dst[kp0 + 1][nn] = breg[it].y; dst[kp0 + 2][nn] = breg[it].z; dst[kp0 + 3][nn] = breg[it].w;
    }
    uint4 acur[4][2];
#pragma unroll
    for (int k8 = 0; k8 < 4; ++k8) { acur[k8][0] = areg[k8][0]; acur[k8][1] = areg[k8][1]; }
    __syncthreads();
    if (k0 + 32 < r_t) load_chunk(k0 + 32);
#pragma unroll
    for (int s16 = 0; s16 < 2; ++s16) {
      // A: rows g, g + 8; k = 16 s16 + 2c, +1 (word c of the first eight halves) and + 8 (word c of the next eight)
      const uint32_t a[4] = {word_of(acur[2 * s16][0], c), word_of(acur[2 * s16][1], c), word_of(acur[2 * s16 + 1][0], c), word_of(acur[2 * s16 + 1][1], c)};
#pragma unroll
      for (int nt = 0; nt < 8; ++nt) {
        const int col = wn * 64 + nt * 8 + g;
        att_mma_f16(acc[nt], a, Bh[s16 * 8 + c][col], Bh[s16 * 8 + c + 4][col]);
        att_mma_f16(acc[nt], a, Bl[s16 * 8 + c][col], Bl[s16 * 8 + c + 4][col]);
      }
    }
  }
  const int t_lo = t0 + wt * 16 + g, t_hi = t_lo + 8;
#pragma unroll
  for (int nt = 0; nt < 8; ++nt) {
    const int n = n0 + wn * 64 + nt * 8 + 2 * c;
    if (n >= N) continue;
    const float2 we = *(const float2 *)(jb.we + n);
    const size_t col = (size_t)(n / NQP) * jb.T * NQP + n % NQP;
    if (t_lo < jb.T) *(float2 *)(jb.p + col + (size_t)t_lo * NQP) = make_float2(acc[nt][0] * we.x, acc[nt][1] * we.y);
    if (t_hi < jb.T) *(float2 *)(jb.p + col + (size_t)t_hi * NQP) = make_float2(acc[nt][2] * we.x, acc[nt][3] * we.y);
  }
}

// grid (n_chunks * KT, ceil(m NQP / 128), groups) with KT = ceil(max r_t / 64), 256 threads: 128 columns n x 64 columns k
// of one 256-token chunk; warp w owns 16 n x 64 k.  m16n8k16 fp16 MMAs: U_T is fp16 as stored, a weight p in [0, 1]
// enters as hi + lo fp16 (22 bits; the lo part of a tiny weight may be subnormal, an absolute error below 2^-25).  The
// next 32 tokens' operands are requested into registers before the MMAs of the current 32.
__global__ void __launch_bounds__(256) attend_bvalue_kernel(const AttendJob *__restrict__ jobs, int NQP, int n_chunks, int KT) {
  const AttendJob &jb = jobs[blockIdx.z];
  const int r_t = jb.v.r_t, N = jb.m * NQP, n0 = blockIdx.y * 128;
  const int chunk = blockIdx.x / KT, kb = (blockIdx.x % KT) * 64, t0 = chunk * kAttChunk;
  if (r_t == 0 || n0 >= N || kb >= r_t || t0 >= jb.T) return;
  // token pairs (2 tp, 2 tp + 1) packed as half2, low half = the even token
  __shared__ __align__(16) uint32_t Ph[16][kAttBPitch], Pl[16][kAttBPitch];     // weights hi / lo, [tp][n]
  __shared__ __align__(16) uint32_t Us[16][64 + 8];                             // U_T, [tp][k]
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, c = lane & 3;
  float acc[8][4];
#pragma unroll
  for (int nt = 0; nt < 8; ++nt)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[nt][j] = 0.f;
  const int nt_tok = min(kAttChunk, jb.T - t0);          // a multiple of 128
  float4 preg[2][2];
  uint4 ureg[2];
  const int u_tp = (tid & 127) >> 3, u_k8 = (tid & 7) * 8;
  auto load_step = [&](int tt0) {
#pragma unroll
    for (int it = 0; it < 2; ++it) {
      const int idx = tid + it * 256, tp = idx >> 5, q4 = idx & 31, n = n0 + q4 * 4;
      preg[it][0] = make_float4(0.f, 0.f, 0.f, 0.f); preg[it][1] = preg[it][0];
      if (n < N) {
        const float *src = jb.p + ((size_t)(n / NQP) * jb.T + t0 + tt0 + 2 * tp) * NQP + n % NQP;
        preg[it][0] = *(const float4 *)src;
        preg[it][1] = *(const float4 *)(src + NQP);
      }
    }
    ureg[0] = make_uint4(0u, 0u, 0u, 0u); ureg[1] = ureg[0];
    if (tid < 128 && kb + u_k8 < r_t) {
      const __half *src = jb.v.UT + (size_t)(t0 + tt0 + 2 * u_tp) * r_t + kb + u_k8;
      ureg[0] = __ldg((const uint4 *)src);
      ureg[1] = __ldg((const uint4 *)(src + r_t));
    }
  };
  load_step(0);
  for (int tt0 = 0; tt0 < nt_tok; tt0 += 32) {
    __syncthreads();
#pragma unroll
    for (int it = 0; it < 2; ++it) {
      const int idx = tid + it * 256, tp = idx >> 5, q4 = idx & 31;
      const float4 v0 = preg[it][0], v1 = preg[it][1];
      const float x0[4] = {v0.x, v0.y, v0.z, v0.w}, x1[4] = {v1.x, v1.y, v1.z, v1.w};
      uint32_t hi[4], lo[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const __half2 h2 = __floats2half2_rn(x0[j], x1[j]);
        const float2 hf = __half22float2(h2);
        const __half2 l2 = __floats2half2_rn(x0[j] - hf.x, x1[j] - hf.y);
        hi[j] = *(const uint32_t *)&h2; lo[j] = *(const uint32_t *)&l2;
      }
      *(uint4 *)&Ph[tp][q4 * 4] = make_uint4(hi[0], hi[1], hi[2], hi[3]);
      *(uint4 *)&Pl[tp][q4 * 4] = make_uint4(lo[0], lo[1], lo[2], lo[3]);
    }
    if (tid < 128) {
      const uint32_t w0[4] = {ureg[0].x, ureg[0].y, ureg[0].z, ureg[0].w}, w1[4] = {ureg[1].x, ureg[1].y, ureg[1].z, ureg[1].w};
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        Us[u_tp][u_k8 + 2 * j] = (w0[j] & 0xFFFFu) | (w1[j] << 16);
        Us[u_tp][u_k8 + 2 * j + 1] = (w0[j] >> 16) | (w1[j] & 0xFFFF0000u);
      }
    }
    __syncthreads();
    if (tt0 + 32 < nt_tok) load_step(tt0 + 32);
#pragma unroll
    for (int s16 = 0; s16 < 2; ++s16) {
      const int nr = warp * 16 + g;
      const uint32_t ah[4] = {Ph[s16 * 8 + c][nr], Ph[s16 * 8 + c][nr + 8], Ph[s16 * 8 + c + 4][nr], Ph[s16 * 8 + c + 4][nr + 8]};
      const uint32_t al[4] = {Pl[s16 * 8 + c][nr], Pl[s16 * 8 + c][nr + 8], Pl[s16 * 8 + c + 4][nr], Pl[s16 * 8 + c + 4][nr + 8]};
#pragma unroll
      for (int nt = 0; nt < 8; ++nt) {
        const uint32_t b0 = Us[s16 * 8 + c][nt * 8 + g], b1 = Us[s16 * 8 + c + 4][nt * 8 + g];
        att_mma_f16(acc[nt], ah, b0, b1);
        att_mma_f16(acc[nt], al, b0, b1);
      }
    }
  }
#pragma unroll
  for (int half = 0; half < 2; ++half) {
    const int n = n0 + warp * 16 + g + half * 8;
    if (n >= N) continue;
    float *yr = jb.y + (((size_t)(n / NQP) * n_chunks + chunk) * NQP + n % NQP) * r_t;
#pragma unroll
    for (int nt = 0; nt < 8; ++nt) {
      const int k = kb + nt * 8 + 2 * c;
      if (k < r_t) yr[k] = acc[nt][half * 2];
      if (k + 1 < r_t) yr[k + 1] = acc[nt][half * 2 + 1];
    }
  }
}

// grid (m, groups, n_q), 128 threads; CTA z finishes query z.  Dynamic shared memory: (n_chunks + v.r_t + 128) floats.
__global__ void __launch_bounds__(128) attend_combine_kernel(const __grid_constant__ AttendArgs args, int n_q, int NQP, int n_chunks,
                                                             uint64_t seed) {
  const AttendJob &jb = att_job(args, blockIdx.y);
  const int h = blockIdx.x, f = threadIdx.x, i = blockIdx.z, warp = f >> 5, lane = f & 31;
  if (h >= jb.m) return;
  extern __shared__ unsigned char att_smem[];
  const int r_t = jb.v.r_t;
  float *coef = (float *)att_smem;                                   // [n_chunks]
  float *ys = coef + ((n_chunks + 3) & ~3);                          // [r_t]
  float *buf = ys + r_t;                                             // [128]
  __shared__ float4 part[4][32];
  __shared__ float Ls;
  const float *ml = jb.ml + (size_t)h * n_chunks * 2 * NQP + i;
  const float esc = r_t > 0 ? ldexpf(1.f, *jb.v.e) : 0.f;
  att_wait_predecessor();
  // running-maximum merge of the chunks: warp 0 finds the maximum and the rescaled sum
  if (warp == 0) {
    float M = -INFINITY;
    for (int c = lane; c < n_chunks; c += 32) M = fmaxf(M, ml[(size_t)c * 2 * NQP]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, o));
    float L = 0.f;
    for (int c = lane; c < n_chunks; c += 32) {
      const float cf = expf(ml[(size_t)c * 2 * NQP] - M);
      coef[c] = cf;
      L = fmaf(cf, ml[(size_t)c * 2 * NQP + NQP], L);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) L += __shfl_xor_sync(0xffffffffu, L, o);
    if (lane == 0) Ls = L;
  }
  __syncthreads();
  auto merge = [&](const float *p, size_t stride) {
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
    int c = 0;
    for (; c + 16 <= n_chunks; c += 16) {
      float v[16];
#pragma unroll
      for (int u = 0; u < 16; ++u) v[u] = p[(size_t)(c + u) * stride];
#pragma unroll
      for (int u = 0; u < 16; ++u) acc[u & 3] = fmaf(coef[c + u], v[u], acc[u & 3]);
    }
    for (; c < n_chunks; ++c) acc[0] = fmaf(coef[c], p[(size_t)c * stride], acc[0]);
    return (acc[0] + acc[1]) + (acc[2] + acc[3]);
  };
  if (jb.v.bits > 0) buf[f] = merge(jb.a + ((size_t)h * n_chunks * NQP + i) * 128 + f, (size_t)NQP * 128);
  for (int k = f; k < r_t; k += 128) ys[k] = merge(jb.y + ((size_t)h * n_chunks * NQP + i) * r_t + k, (size_t)NQP * r_t);
  __syncthreads();
  // y P_h: a lane per four features, a warp per fourth row
  float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
  const uint2 *P = (const uint2 *)(jb.vP + (size_t)h * r_t * 128) + lane;
#pragma unroll 8
  for (int k = warp; k < r_t; k += 4) {
    const uint2 p = __ldg(P + (size_t)k * 32);
    const float2 a = __half22float2(*(const __half2 *)&p.x), b = __half22float2(*(const __half2 *)&p.y);
    const float y = ys[k];
    o.x = fmaf(y, a.x, o.x); o.y = fmaf(y, a.y, o.y); o.z = fmaf(y, b.x, o.z); o.w = fmaf(y, b.y, o.w);
  }
  part[warp][lane] = o;
  __syncthreads();
  if (warp) return;
  float res[4] = {0.f, 0.f, 0.f, 0.f};
  if (jb.v.bits > 0) {
    const float4 v = *(const float4 *)(buf + 4 * lane);
    res[0] = v.x; res[1] = v.y; res[2] = v.z; res[3] = v.w;
    att_wht_warp(res);
#pragma unroll
    for (int j = 0; j < 4; ++j) res[j] *= kInvSqrtD * att_sign(seed, jb.v.cell, 4 * lane + j);
  }
  const float4 p1 = part[1][lane], p2 = part[2][lane], p3 = part[3][lane];
  const float L = Ls;
  *(float4 *)(jb.out + ((size_t)h * n_q + i) * 128 + 4 * lane) =
      make_float4((((o.x + p1.x) + (p2.x + p3.x)) * esc + res[0]) / L, (((o.y + p1.y) + (p2.y + p3.y)) * esc + res[1]) / L,
                  (((o.z + p1.z) + (p2.z + p3.z)) * esc + res[2]) / L, (((o.w + p1.w) + (p2.w + p3.w)) * esc + res[3]) / L);
}

}  // namespace jolt
