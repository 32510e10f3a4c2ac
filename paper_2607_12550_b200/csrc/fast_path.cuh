// Hooks through which the tcgen05 / TMA kernels replace stages of the portable pipeline.  A cell takes
// the tensor-core kernels when its shape fits them (fp16 data, r_t a multiple of 16 up to 256, r_f a
// multiple of 8); every other cell stays on the portable kernels, in the same call.
#pragma once
#include "tc_backbone.cuh"
#include "tc_decode.cuh"
#include "tc_decode_p.cuh"
#include "tc_gemm.cuh"
#include "tc_orth.cuh"
#include "tc_orth_wide.cuh"
#include "chol_cluster.cuh"

namespace {

inline bool tc_shape_ok(const CellDesc &c) {
  return c.r_t > 0 && c.r_t % 16 == 0 && c.r_t <= 256 && c.r_f % 8 == 0 && c.r_f >= 8 && c.T % 128 == 0;
}

// Tensor maps of the stored factors (constant for the life of a handle).
inline bool encode_store_maps(CellStore &cs) {
  const CellDesc &c = cs.c;
  cs.tc_ok = false;
  if (!tc_shape_ok(c)) return false;
  {
    const uint64_t dims[2] = {(uint64_t)c.r_t, (uint64_t)c.T};
    const uint64_t str[1] = {(uint64_t)c.r_t * 2};
    const uint32_t box[2] = {64, 128};
    if (!make_tmap_f16(&cs.tmUT, cs.UT16, 2, dims, str, box)) return false;
  }
  {  // projected core P[m * r_t][128]: a box is one head's r_t rows by 64 features (one MN-major operand panel)
    if (!cs.P16) return false;
    const uint64_t dims[2] = {(uint64_t)kD, (uint64_t)c.m * c.r_t};
    const uint64_t str[1] = {(uint64_t)kD * 2};
    const uint32_t box[2] = {64, (uint32_t)c.r_t};
    if (!make_tmap_f16(&cs.tmP, cs.P16, 2, dims, str, box)) return false;
  }
  cs.tc_ok = true;
  return true;
}

// Launch with an explicit execution priority (the least one for the kernels that fill the machine: a cell group's
// cache-wide sweeps and its residual pass then yield to the other groups' small latency-bound kernels, whose side
// streams run at a higher priority).  Outside the concurrent cell groups the priority has nothing to compete with.
inline int heavy_kernel_priority() {
  static int lo = 0, hi = 0;
  static bool have = false;
  if (!have) { cudaDeviceGetStreamPriorityRange(&lo, &hi); have = true; }
  return lo;
}
template <typename... KArgs, typename... Args>
inline void launch_heavy(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, Args... args) {
  cudaLaunchConfig_t cfg;
  memset(&cfg, 0, sizeof cfg);
  cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = s;
  cudaLaunchAttribute at;
  memset(&at, 0, sizeof at);
  at.id = cudaLaunchAttributePriority; at.val.priority = heavy_kernel_priority();
  cfg.attrs = &at; cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, kernel, KArgs(args)...);
}

inline void bb_split(int total_heads, int n_tiles, int &tiles_per_item, int &items_per_head) {
  int per_head = (888 + total_heads / 2) / std::max(total_heads, 1);
  per_head = std::max(1, std::min(per_head, n_tiles));
  tiles_per_item = (n_tiles + per_head - 1) / per_head;
  items_per_head = (n_tiles + tiles_per_item - 1) / tiles_per_item;
}

inline void add_backbone_tc(Program &P, int stage, const std::vector<tc::BBCell> &cells, uint64_t seed) {
  if (cells.empty()) return;
  static DeviceOnce once;
  once([] { cudaFuncSetAttribute(tc::backbone_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, tc::BB_SMEM_BYTES); });
  int gx = 0;
  for (auto &c : cells) gx = std::max(gx, c.m * c.items_per_head);
  const size_t off = P.push(cells);
  const int n = (int)cells.size();
  P.add(stage, [=](char *dev_t, cudaStream_t s) {
    launch_heavy(tc::backbone_kernel, dim3(gx, n), dim3(tc::BB_THREADS), (size_t)tc::BB_SMEM_BYTES, s, (const tc::BBCell *)(dev_t + off), seed);
    LAUNCHED();
  });
}

inline void fill_bb_common(tc::BBCell &b, const CellStore &cs, int *status) {
  memset(&b, 0, sizeof b);
  b.tmUT = cs.tmUT; b.tmP = cs.tmP;
  b.words = cs.words; b.scales = cs.scales; b.e = cs.e;
  const CellDesc &c = cs.c;
  b.m = c.m; b.n_heads = c.n_heads; b.T = c.T; b.r_t = c.r_t; b.r_f = c.r_f; b.bits = c.bits; b.cell = c.cell;
  b.status = status;
}


// A launch that may begin while the kernel before it on the stream drains (on the device it waits for that kernel).
template <typename... P, typename... A>
inline void launch_overlapped(void (*kernel)(P...), dim3 grid, int threads, size_t shm, cudaStream_t s, const A &...args) {
  cudaLaunchConfig_t cfg;
  memset(&cfg, 0, sizeof cfg);
  cfg.gridDim = grid; cfg.blockDim = dim3(threads); cfg.dynamicSmemBytes = shm; cfg.stream = s;
  cudaLaunchAttribute at;
  memset(&at, 0, sizeof at);
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &at; cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}

// Per-item decode kernel over descriptors [first, first + n).  overlap: behind a launch of the persistent kernel, which writes other
// cells: this one's CTAs take the SMs that come free.
inline void launch_decode_items(const jolt_handle *H, int first, int n, const tc::DecOut &out, const float2 *rope, long long *dbg, bool overlap, cudaStream_t s) {
  using LY = tc::DecLayout;
  static DeviceOnce once;
  once([] {
    cudaFuncSetAttribute(tc::decode_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, LY::SMEM_BYTES);
    cudaFuncSetAttribute(tc::decode_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, LY::SMEM_BYTES);
  });
  tc::DecIArgs a;
  memset(&a, 0, sizeof a);
  a.out = out; a.cells = (const tc::BBCell *)H->d_dec + first; a.rope = rope; a.seed = H->seed;
#ifdef JOLT_DEBUG
  a.dbg = dbg;
#else
  (void)dbg;
#endif
  int heads = 0, m_max = 0;
  for (int i = first; i < first + n; ++i) { heads += H->dec.m[i]; m_max = std::max(m_max, H->dec.m[i]); }
  bb_split(heads, H->T / 128, a.tiles_per_item, a.items_per_head);
  const dim3 grid(m_max * a.items_per_head, n);
  const auto kernel = rope ? tc::decode_kernel<true> : tc::decode_kernel<false>;
  if (overlap) launch_overlapped(kernel, grid, LY::THREADS, LY::SMEM_BYTES, s, a);
  else kernel<<<grid, LY::THREADS, LY::SMEM_BYTES, s>>>(a);
  LAUNCHED();
}

template <bool TMA_ONLY, unsigned BITMASK, bool ROPE = false>
inline void launch_decode_p(const tc::DecPArgs &a, int grid, cudaStream_t s, bool overlap = false) {
  using LY = tc::DecLayout;
  static DeviceOnce once;
  once([] { cudaFuncSetAttribute(tc::decode_persistent_kernel<TMA_ONLY, BITMASK, ROPE>, cudaFuncAttributeMaxDynamicSharedMemorySize, LY::SMEM_BYTES); });
  if (overlap) launch_overlapped(tc::decode_persistent_kernel<TMA_ONLY, BITMASK, ROPE>, dim3(grid), LY::THREADS, LY::SMEM_BYTES, s, a);
  else tc::decode_persistent_kernel<TMA_ONLY, BITMASK, ROPE><<<grid, LY::THREADS, LY::SMEM_BYTES, s>>>(a);
}

// The persistent kernel is instantiated per output mode and per set of bit widths: with at most two tile loops compiled
// in (and fp16 output through bulk tensor stores only) ptxas keeps the whole epilogue in registers; with three or more
// it spills 50-60 bytes, and a spill reload inside the tile loop costs several per cent of the launch.
inline void launch_decode_widths(const tc::DecPArgs &a, unsigned bitmask, int grid, cudaStream_t s) {
  const bool tma_only = a.out.tma_out != 0 && a.out.out_dtype == DT_F16;
  if (!tma_only) launch_decode_p<false, 0x11Fu>(a, grid, s);
  else if (bitmask == 0x010u) launch_decode_p<true, 0x010u>(a, grid, s);
  else if (bitmask == 0x100u) launch_decode_p<true, 0x100u>(a, grid, s);
  else if ((bitmask & ~0x110u) == 0) launch_decode_p<true, 0x110u>(a, grid, s);
  else if ((bitmask & ~0x014u) == 0) launch_decode_p<true, 0x014u>(a, grid, s);
  else if ((bitmask & ~0x018u) == 0) launch_decode_p<true, 0x018u>(a, grid, s);
  else launch_decode_p<true, 0x11Fu>(a, grid, s);
}

// Descriptors of the cells that take the tensor-core decode, in the order [values, r_t <= 128][keys, r_t <= 128][r_t > 128] and in each
// class the costliest first (most residual bits, then largest r_t: the last wave of per-item CTAs is then the cheapest), for the
// persistent kernel; then all of them once more, the costliest first, for one launch of the per-item kernel.
inline void make_decode_table(jolt_handle &H, std::vector<tc::BBCell> &table) {
  table.clear();
  H.dec = jolt_handle::DecTable();
  auto costlier = [](const tc::BBCell &x, const tc::BBCell &y) { return x.bits != y.bits ? x.bits > y.bits : x.r_t > y.r_t; };
  long long total = 0;
  for (int cls = 0; cls < 3; ++cls) {
    std::vector<tc::BBCell> v;
    for (size_t i = 0; i < H.cells.size(); ++i) {
      const CellStore &cs = H.cells[i];
      if (!cs.tc_ok || cls != (cs.c.r_t > 128 ? 2 : (i % 2 == 0 ? 1 : 0))) continue;
      tc::BBCell b;
      fill_bb_common(b, cs, H.d_status + 4 * i);
      b.layer0 = H.group_start[i / 2];
      v.push_back(b);
    }
    std::stable_sort(v.begin(), v.end(), costlier);
    for (auto &b : v) {
      b.tile_base = (int)std::min<long long>(total, 1 << 30);
      total += (long long)b.m * (b.T / 128);
      if (cls < 2) H.dec.bitmask[cls] |= 1u << b.bits;
      H.dec.m.push_back(b.m);
    }
    table.insert(table.end(), v.begin(), v.end());
    H.dec.end[cls] = (int)table.size();
    H.dec.tiles[cls] = total;
  }
  std::vector<tc::BBCell> all = table;
  std::stable_sort(all.begin(), all.end(), costlier);
  for (auto &b : all) H.dec.m.push_back(b.m);
  table.insert(table.end(), all.begin(), all.end());
}

// ------------------------------------------------------------------ tensor-core sweeps of the factor stage

inline bool make_x_map(CUtensorMap *tm, const CellDesc &c, uint32_t box_tok) {
  const uint64_t dims[4] = {(uint64_t)kD, (uint64_t)c.T, (uint64_t)c.n_heads, (uint64_t)(c.m / c.n_heads)};
  const uint64_t str[3] = {(uint64_t)c.st * 2, (uint64_t)c.sh * 2, (uint64_t)c.sl * 2};
  const uint32_t box[4] = {64, box_tok, 1, 1};
  return make_tmap_f16(tm, c.X, 4, dims, str, box);
}

inline bool x_tma_ok(const CellDesc &c) {
  return c.dtype == DT_F16 && c.st % 8 == 0 && c.sh % 8 == 0 && c.sl % 8 == 0 && ((uintptr_t)c.X % 16 == 0) && c.T % 128 == 0;
}

// A cell's factor-stage sweeps can run on tensor cores: fp16 data TMA can address.  One MMA takes N <= 256
// columns; wider sketches are swept in column chunks (one more read of X per chunk).
constexpr int kTcMaxSketch = 768;
inline bool tc_sweep_ok(const CellDesc &c, bool staged_from_host) {
  if (c.dtype != DT_F16 || c.st % 8 || c.sh % 8 || c.sl % 8 || c.T % 128) return false;
  if (!staged_from_host && ((uintptr_t)c.X % 16)) return false;
  return c.k >= 1 && c.k <= kTcMaxSketch;
}

// column chunks of a padded sketch width: equal multiples of 16, each <= 256
inline void sketch_chunks(int kp, std::vector<std::pair<int, int>> &out) {
  const int n = (kp + 255) / 256;
  const int w = (((kp + n - 1) / n) + 15) & ~15;
  out.clear();
  for (int c0 = 0; c0 < kp; c0 += w) out.push_back({c0, std::min(w, kp - c0)});
}

inline int ilog2_floor(long long v) { int e = 0; while ((1ll << (e + 1)) <= v) ++e; return e; }

template <int MODE>
inline void launch_tc_gemm(Program &P, int stage, std::vector<tc::GemmCell> &cells) {
  if (cells.empty()) return;
  uint32_t max_stage = 0;
  int gx = 0;
  for (auto &c : cells) {
    const uint32_t b_bytes = MODE == tc::GM_GRAM ? 0u : (uint32_t)c.kp * 128u;
    const uint32_t b_pitch = (b_bytes + 1023u) & ~1023u;
    max_stage = std::max(max_stage, 16384u + ((c.has_lo && MODE != tc::GM_GRAM) ? 2 * b_pitch : b_pitch));
    gx = std::max(gx, MODE == tc::GM_TOK ? c.T / 128 : c.m);
  }
  int n_stages = std::min(8, (int)((tc::GM_SMEM_LIMIT - 1536) / max_stage));
  const size_t smem = (size_t)n_stages * max_stage + 1024 + 512;
  static DeviceOnce once;
  once([] { cudaFuncSetAttribute(tc::tc_gemm_kernel<MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, tc::GM_SMEM_LIMIT); });
  const size_t off = P.push(cells);
  const int n = (int)cells.size();
  P.add(stage, [=](char *dev_t, cudaStream_t s) {
    launch_heavy(tc::tc_gemm_kernel<MODE>, dim3(gx, n), dim3(tc::GM_THREADS), smem, s, (const tc::GemmCell *)(dev_t + off), n_stages);
    LAUNCHED();
  });
}

template <int MODE>
inline void launch_tc_gemm2(Program &P, int stage, std::vector<tc::Gemm2Cell> &cells) {
  if (cells.empty()) return;
  uint32_t max_stage = 0;
  int gx = 0;
  for (auto &c : cells) {
    const uint32_t b_pitch = ((uint32_t)c.kp * 128u + 1023u) & ~1023u;
    max_stage = std::max(max_stage, 32768u + (c.has_lo ? 2 * b_pitch : b_pitch));
    gx = std::max(gx, MODE == tc::GM_TOK ? (c.T / 128 + 1) / 2 : c.m / 2);
  }
  const int n_stages = std::min(8, (int)((tc::GM_SMEM_LIMIT - 1536) / max_stage));
  const size_t smem = (size_t)n_stages * max_stage + 1024 + 512;
  static DeviceOnce once;
  once([] { cudaFuncSetAttribute(tc::tc_gemm2_kernel<MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, tc::GM_SMEM_LIMIT); });
  const size_t off = P.push(cells);
  const int n = (int)cells.size();
  P.add(stage, [=](char *dev_t, cudaStream_t s) {
    launch_heavy(tc::tc_gemm2_kernel<MODE>, dim3(gx, n), dim3(tc::GM_THREADS), smem, s, (const tc::Gemm2Cell *)(dev_t + off), n_stages);
    LAUNCHED();
  });
}

inline bool make_x_map4(CUtensorMap *tm, const CellDesc &c, uint32_t box_tok, uint32_t box_heads) {
  const uint64_t dims[4] = {(uint64_t)kD, (uint64_t)c.T, (uint64_t)c.n_heads, (uint64_t)(c.m / c.n_heads)};
  const uint64_t str[3] = {(uint64_t)c.st * 2, (uint64_t)c.sh * 2, (uint64_t)c.sl * 2};
  const uint32_t box[4] = {64, box_tok, box_heads, 1};
  return make_tmap_f16(tm, c.X, 4, dims, str, box);
}

inline void launch_split(Program &P, int stage, const std::vector<tc::SplitJob> &jobs) {
  if (jobs.empty()) return;
  const size_t off = P.push(jobs);
  const int n = (int)jobs.size();
  P.add(stage, [=](char *dev_t, cudaStream_t s) {
    tc::split_transpose_kernel<<<dim3(296, 1, n), 256, 0, s>>>((const tc::SplitJob *)(dev_t + off));
    LAUNCHED();
  });
}

// mode-3 Gram of the tensor-core cells: fp32 partial per head, summed in fp64.
inline void add_gram_tc(Program &P, int stage, std::vector<CellWork> &ws) {
  std::vector<tc::GemmCell> gc;
  std::vector<const float *> parts; std::vector<double *> outs; std::vector<int> counts;
  for (auto &w : ws) {
    if (!w.active || !w.tc_gram) continue;
    tc::GemmCell g;
    memset(&g, 0, sizeof g);
    make_x_map(&g.tmX, w.c, 64);
    g.ldc = kD; g.ncols = kD; g.kp = kD; g.has_lo = 0; g.scale_exp = 0;
    g.m = w.c.m; g.n_heads = w.c.n_heads; g.T = w.c.T; g.status = w.status;
    const int nseg = tok_segments(w.c.T);
    for (int sg = 0; sg < nseg; ++sg) {
      g.C = (float *)w.gram_part + (size_t)sg * w.c.m * kD * kD;
      g.t0 = sg * kTokSegment; g.n_tok = std::min(kTokSegment, w.c.T - g.t0);
      gc.push_back(g);
    }
    parts.push_back((const float *)w.gram_part); outs.push_back(w.C); counts.push_back(w.c.m * nseg);
  }
  if (gc.empty()) return;
  launch_tc_gemm<tc::GM_GRAM>(P, stage, gc);
  const size_t o1 = P.push(parts), o2 = P.push(outs), o3 = P.push(counts);
  const int n = (int)parts.size();
  P.add(stage, [=](char *dev_t, cudaStream_t s) {
    tc::reduce_gram_partials_kernel<<<dim3(kD * kD / 256, n), 256, 0, s>>>((const float *const *)(dev_t + o1),
                                                                        (double *const *)(dev_t + o2), (const int *)(dev_t + o3));
    LAUNCHED();
  });
}

// S = sum_h X_h W_h for the tensor-core cells.  src: 0 = fp16 sketch already in Bhi, 1 = split W (fp32,
// [h][128][k]), 2 = split Z (fp32, [h][128][k], orthonormal columns over N rows).
inline bool orth_tc_ok(const CellWork &w);
inline void add_tok_tc(Program &P, int stage, std::vector<CellWork> &ws, const std::vector<int> &src) {
  std::vector<tc::SplitJob> sp;
  std::vector<tc::GemmCell> gc;
  std::vector<tc::Gemm2Cell> gc2;
  for (size_t i = 0; i < ws.size(); ++i) {
    CellWork &w = ws[i];
    if (!w.active || !w.tc) continue;
    const CellDesc &c = w.c;
    int se = 0;
    if (src[i] == 2 && w.ufI && w.split_ready == 2) {
      se = ilog2_floor((long long)c.N) / 2;          // the triangular solve of orth(Z) has written the operand already
      w.split_ready = 0;
    } else if (src[i] != 0) {
      const float *in = w.W;
      if (src[i] == 2) { in = w.ufI ? w.Z : w.W; se = ilog2_floor((long long)c.N) / 2; }
      tc::SplitJob j;
      j.in = in; j.hi = w.Bhi; j.lo = w.Blo; j.batch = c.m; j.rows = kD; j.cols = c.k; j.ld_in = c.k;
      j.kp = w.kp; j.scale_exp = se; j.absmax = nullptr; j.top = 0;
      sp.push_back(j);
    }
    std::vector<std::pair<int, int>> ch;
    sketch_chunks(w.kp, ch);
    if (g_fast.load() & 64) {
      // two token tiles per CTA share every operand tile
      if (orth_tc_ok(w)) w.absmax_ready = true;
      for (auto &cc : ch) {
        const int c0 = cc.first, kc = cc.second;
        if (c0 >= c.k) break;
        tc::Gemm2Cell g;
        memset(&g, 0, sizeof g);
        const uint64_t dims[3] = {(uint64_t)kD, (uint64_t)kc, (uint64_t)c.m};
        const uint64_t str[2] = {(uint64_t)kD * 2, (uint64_t)w.kp * kD * 2};
        const uint32_t box[3] = {64, (uint32_t)kc, 1};
        bool okm = make_x_map4(&g.tmX, c, 256, 1) && make_tmap_f16(&g.tmBhi, w.Bhi + (size_t)c0 * kD, 3, dims, str, box) &&
                   make_tmap_f16(&g.tmBlo, w.Blo + (size_t)c0 * kD, 3, dims, str, box);
        (void)okm;
        g.C = w.S + c0; g.ldc = c.k; g.ncols = std::min(kc, c.k - c0); g.kp = kc; g.has_lo = src[i] != 0; g.scale_exp = se;
        g.m = c.m; g.n_heads = c.n_heads; g.T = c.T; g.status = w.status;
        if (w.absmax_ready) g.absmax = w.orthMax + (w.orthMaxUsed % kOrthMaxSlots);
        gc2.push_back(g);
      }
      continue;
    }
    for (auto &cc : ch) {
      const int c0 = cc.first, kc = cc.second;
      if (c0 >= c.k) break;
      tc::GemmCell g;
      memset(&g, 0, sizeof g);
      const uint64_t dims[3] = {(uint64_t)kD, (uint64_t)kc, (uint64_t)c.m};
      const uint64_t str[2] = {(uint64_t)kD * 2, (uint64_t)w.kp * kD * 2};
      const uint32_t box[3] = {64, (uint32_t)kc, 1};
      bool okm = make_x_map(&g.tmX, c, 128) && make_tmap_f16(&g.tmBhi, w.Bhi + (size_t)c0 * kD, 3, dims, str, box) &&
                 make_tmap_f16(&g.tmBlo, w.Blo + (size_t)c0 * kD, 3, dims, str, box);
      (void)okm;
      g.C = w.S + c0; g.ldc = c.k; g.ncols = std::min(kc, c.k - c0); g.kp = kc; g.has_lo = src[i] != 0; g.scale_exp = se;
      g.m = c.m; g.n_heads = c.n_heads; g.T = c.T; g.status = w.status;
      gc.push_back(g);
    }
  }
  launch_split(P, stage, sp);
  launch_tc_gemm<tc::GM_TOK>(P, stage, gc);
  launch_tc_gemm2<tc::GM_TOK>(P, stage, gc2);
}

// Z'_h = X_h^T Q for the tensor-core cells (Q = w.S, T x k with orthonormal columns).
inline void add_feat_tc(Program &P, int stage, std::vector<CellWork> &ws) {
  std::vector<tc::SplitJob> sp;
  std::vector<tc::GemmCell> gc;
  std::vector<tc::Gemm2Cell> gc2;
  std::vector<tc::SumJob> sums;
  for (auto &w : ws) {
    if (!w.active || !w.tc) continue;
    const CellDesc &c = w.c;
    const int se = ilog2_floor(c.T) / 2;
    if (w.split_ready != 1) {      // else the triangular solve of orth(S) has written the operand already
      tc::SplitJob j;
      j.in = w.S; j.hi = w.Bhi; j.lo = w.Blo; j.batch = 1; j.rows = c.T; j.cols = c.k; j.ld_in = c.k; j.kp = w.kp; j.scale_exp = se; j.absmax = nullptr; j.top = 0;
      sp.push_back(j);
    }
    w.split_ready = 0;
    std::vector<std::pair<int, int>> ch;
    sketch_chunks(w.kp, ch);
    if (c.n_heads % 2 == 0 && (g_fast.load() & 64)) {
      // two heads of a layer per CTA share every tile of Q
      const int nseg = tok_segments(c.T);
      if (orth_tc_ok(w)) w.absmax_ready = true;
      unsigned *slot = w.absmax_ready ? w.orthMax + (w.orthMaxUsed % kOrthMaxSlots) : nullptr;
      for (auto &cc : ch) {
        const int c0 = cc.first, kc = cc.second;
        if (c0 >= c.k) break;
        tc::Gemm2Cell g;
        memset(&g, 0, sizeof g);
        const uint64_t dims[2] = {(uint64_t)c.T, (uint64_t)kc};
        const uint64_t str[1] = {(uint64_t)c.T * 2};
        const uint32_t box[2] = {64, (uint32_t)kc};
        bool okm = make_x_map4(&g.tmX, c, 64, 2) && make_tmap_f16(&g.tmBhi, w.Bhi + (size_t)c0 * c.T, 2, dims, str, box) &&
                   make_tmap_f16(&g.tmBlo, w.Blo + (size_t)c0 * c.T, 2, dims, str, box);
        (void)okm;
        g.ldc = c.k; g.ncols = std::min(kc, c.k - c0); g.kp = kc; g.has_lo = 1; g.scale_exp = se;
        g.m = c.m; g.n_heads = c.n_heads; g.T = c.T; g.status = w.status;
        g.absmax = nseg == 1 ? slot : nullptr;
        for (int sg = 0; sg < nseg; ++sg) {
          g.C = (nseg > 1 ? w.Zpart + (size_t)sg * c.m * kD * c.k : w.Zp) + c0;
          g.t0 = sg * kTokSegment; g.n_tok = std::min(kTokSegment, c.T - g.t0);
          gc2.push_back(g);
        }
      }
      if (nseg > 1) sums.push_back({w.Zpart, w.Zp, (long long)c.m * kD * c.k, (long long)c.m * kD * c.k, nseg, slot});
      continue;
    }
    for (auto &cc : ch) {
      const int c0 = cc.first, kc = cc.second;
      if (c0 >= c.k) break;
      tc::GemmCell g;
      memset(&g, 0, sizeof g);
      const uint64_t dims[2] = {(uint64_t)c.T, (uint64_t)kc};
      const uint64_t str[1] = {(uint64_t)c.T * 2};
      const uint32_t box[2] = {64, (uint32_t)kc};
      bool okm = make_x_map(&g.tmX, c, 64) && make_tmap_f16(&g.tmBhi, w.Bhi + (size_t)c0 * c.T, 2, dims, str, box) &&
                 make_tmap_f16(&g.tmBlo, w.Blo + (size_t)c0 * c.T, 2, dims, str, box);
      (void)okm;
      g.ldc = c.k; g.ncols = std::min(kc, c.k - c0); g.kp = kc; g.has_lo = 1; g.scale_exp = se;
      g.m = c.m; g.n_heads = c.n_heads; g.T = c.T; g.status = w.status;
      const int nseg = tok_segments(c.T);
      for (int sg = 0; sg < nseg; ++sg) {
        g.C = (nseg > 1 ? w.Zpart + (size_t)sg * c.m * kD * c.k : w.Zp) + c0;
        g.t0 = sg * kTokSegment; g.n_tok = std::min(kTokSegment, c.T - g.t0);
        gc.push_back(g);
      }
    }
    if (tok_segments(c.T) > 1) sums.push_back({w.Zpart, w.Zp, (long long)c.m * kD * c.k, (long long)c.m * kD * c.k, tok_segments(c.T), nullptr});
  }
  launch_split(P, stage, sp);
  launch_tc_gemm<tc::GM_FEAT>(P, stage, gc);
  launch_tc_gemm2<tc::GM_FEAT>(P, stage, gc2);
  if (!sums.empty()) {
    const size_t off = P.push(sums);
    const int n = (int)sums.size();
    P.add(stage, [=](char *dev_t, cudaStream_t s) {
      tc::sum_partials_f32_kernel<<<dim3(296, n), 256, 0, s>>>((const tc::SumJob *)(dev_t + off));
      LAUNCHED();
    });
  }
}

// fp16 sketch of the r_f = d tensor-core cells, written straight into the TOK operand layout.
inline void add_sketch_gen_tc(Program &P, int stage, std::vector<CellWork> &ws, int stream_id, uint64_t seed) {
  std::vector<tc::SketchJob> jobs;
  for (auto &w : ws)
    if (w.active && w.tc && w.ufI) jobs.push_back({w.Bhi, w.c.m, w.c.k, w.kp, w.c.cell});
  if (jobs.empty()) return;
  const size_t off = P.push(jobs);
  const int n = (int)jobs.size();
  P.add(stage, [=](char *dev_t, cudaStream_t s) {
    launch_heavy(tc::gen_sketch_f16_kernel, dim3(148, n), dim3(256), (size_t)0, s, (const tc::SketchJob *)(dev_t + off), stream_id, seed);
    LAUNCHED();
  });
}

// ------------------------------------------------------------------ CholeskyQR on tensor cores
// Cells whose basis is already kept as the hi + lo operand of the sweeps (tensor-core cells with r_f = d) orthonormalise
// it there: Gram and Q = R L^-T are tcgen05 GEMMs, the Cholesky factor and its inverse one fp64 CTA per cell up to
// OR_MAX_K columns (one accumulator, one shared memory), a cluster per cell beyond.
inline bool orth_tc_ok(const CellWork &w) {
  return w.active && w.tc && w.ufI && w.c.T % 128 == 0 && w.orthPart != nullptr;
}
inline bool orth_is_wide(const CellWork &w) { return w.c.k > tc::OR_MAX_K || w.kp > tc::OR_MAX_KP; }

// The sweep left the raw basis as fp32 rows: measure its magnitude (unless the sweep's epilogue did), split it into the
// operand layout.  After a power iteration the columns are graded like the spectrum: with the largest entry below 1 the lo part of
// an entry 1e-4 of it is a subnormal of three or four bits, and the weak directions of the span were lost with them.
// Wide sketches, which reach furthest down the spectrum, use all of fp16's range (kOrthWideTop).  Distance of the span from an
// fp64 one, key caches: 7.1e-4 -> 1.04e-4 at k = 160, 1.3e-2 -> 5.0e-4 at k = 522 (fp64 Gram and CUDA-core solve: 1.05e-4, 5.0e-4).
constexpr int kOrthWideTop = 15;
inline void add_orth_split(Program &P, int stage, std::vector<CellWork> &ws, const std::vector<int> &idx, bool token_side) {
  std::vector<tc::AbsMaxJob> am;
  std::vector<tc::SplitJob> sp;
  for (int i : idx) {
    CellWork &w = ws[i];
    const CellDesc &c = w.c;
    const int rpp = token_side ? c.T : kD, panels = token_side ? 1 : c.m;
    float *src = token_side ? w.S : w.Z;
    unsigned *slot = w.orthMax + (w.orthMaxUsed++ % kOrthMaxSlots);
    if (!w.absmax_ready) am.push_back({src, (long long)rpp * panels * c.k, slot});
    w.absmax_ready = false;
    tc::SplitJob j;
    j.in = src; j.hi = w.Bhi; j.lo = w.Blo; j.batch = panels; j.rows = rpp; j.cols = c.k; j.ld_in = c.k; j.kp = w.kp; j.scale_exp = 0;
    j.absmax = slot; j.top = orth_is_wide(w) ? kOrthWideTop : 0;
    sp.push_back(j);
  }
  const size_t o_am = P.push(am), o_sp = P.push(sp);
  const int n = (int)idx.size(), n_am = (int)am.size();
  P.add(stage, [=](char *dev_t, cudaStream_t s) {
    if (n_am) { tc::absmax_kernel<<<dim3(32, n_am), 256, 0, s>>>((const tc::AbsMaxJob *)(dev_t + o_am)); LAUNCHED(); }
    tc::split_transpose_kernel<<<dim3(296, 1, n), 256, 0, s>>>((const tc::SplitJob *)(dev_t + o_sp)); LAUNCHED();
  });
}

// Wide sketches (k > OR_MAX_K): blocked Gram and apply, cluster Cholesky.
constexpr double kOrthRedoRel = 5e-7;      // about eight times the error of a single-precision Gram relative to its diagonal
inline void add_orth_wide(Program &P, int stage, std::vector<CellWork> &ws, const std::vector<int> &idx, bool token_side, int passes,
                          bool want_fp32) {
  if (idx.empty()) return;
  static DeviceOnce once;
  once([] {
    cudaFuncSetAttribute(tc::orthw_gram_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, tc::OW_GRAM_SMEM);
    cudaFuncSetAttribute(tc::orthw_apply_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, tc::OW_APPLY_SMEM);
  });
  add_orth_split(P, stage, ws, idx, token_side);
  std::vector<tc::OrthWCell> oc, oc_last;
  std::vector<CholTask> ct, ct_redo;
  std::vector<TallGram> tg;
  int max_chunks = 0, max_tiles = 0, max_pairs = 0, max_k = 0;
  for (int i : idx) {
    CellWork &w = ws[i];
    const CellDesc &c = w.c;
    const int rpp = token_side ? c.T : kD, panels = token_side ? 1 : c.m;
    tc::OrthWCell o;
    memset(&o, 0, sizeof o);
    {
      const uint64_t dims[3] = {(uint64_t)rpp, (uint64_t)w.kp, (uint64_t)panels};
      const uint64_t str[2] = {(uint64_t)rpp * 2, (uint64_t)w.kp * rpp * 2};
      const uint32_t box[3] = {64, 128, 1}, boxa[3] = {64, 64, 1};
      make_tmap_f16(&o.tmHi, w.Bhi, 3, dims, str, box);
      make_tmap_f16(&o.tmLo, w.Blo, 3, dims, str, box);
      make_tmap_f16(&o.tmAhi, w.Bhi, 3, dims, str, boxa);
      make_tmap_f16(&o.tmAlo, w.Blo, 3, dims, str, boxa);
    }
    {
      const uint64_t dims[2] = {(uint64_t)w.kp, (uint64_t)w.kp};
      const uint64_t str[1] = {(uint64_t)w.kp * 2};
      const uint32_t box[2] = {64, 128};
      make_tmap_f16(&o.tmLhi, w.orthLhi, 2, dims, str, box);
      make_tmap_f16(&o.tmLlo, w.orthLlo, 2, dims, str, box);
    }
    const int steps = panels * (rpp / 64), nb = (w.kp + 127) / 128;
    o.part = w.orthPart; o.l_exp = w.orthExp; o.out32 = nullptr; o.ld = c.k; o.k = c.k; o.kp = w.kp; o.rpp = rpp; o.panels = panels;
    o.n_chunks = (steps + tc::OW_GRAM_STEPS - 1) / tc::OW_GRAM_STEPS;
    o.out_exp = ilog2_floor((long long)rpp * panels) / 2;
    o.status = w.status;
    o.hi = w.Bhi; o.lo = w.Blo; o.unit = w.Gs;      // (the fp64 Gram of the first pass is used up by then)
    if (want_fp32) w.unit = w.Gs;
    oc.push_back(o);
    o.out32 = want_fp32 ? (token_side ? w.S : w.Z) : nullptr;
    oc_last.push_back(o);
    ct.push_back({w.orthPart, o.n_chunks, c.k, w.kp, w.cholW, w.cholW + (size_t)c.k * c.k, w.orthLhi, w.orthLlo, w.orthExp, w.status, 1e-10, nullptr, 0.0, nullptr, nullptr});
    {
      // the raw basis may be as ill-conditioned as the cache: where the single-precision Gram is too coarse for a pivot, the
      // Gram is taken again in fp64 from the fp32 rows the sweep left (the second pass starts from a conditioned basis)
      CholTask r = ct.back();
      ct.back().redo = w.orthExp + 1; ct.back().redo_rel = kOrthRedoRel;
      r.only = w.orthExp + 1; r.A64 = w.Gs;
      ct_redo.push_back(r);
      tg.push_back({token_side ? w.S : w.Z, rpp * panels, c.k, w.gpart, w.Gs, w.orthExp + 1});
    }
    max_chunks = std::max(max_chunks, o.n_chunks);
    max_tiles = std::max(max_tiles, panels * (rpp / 128));
    max_pairs = std::max(max_pairs, nb * (nb + 1) / 2); max_k = std::max(max_k, c.k);
    w.split_ready = token_side ? 1 : 2;
  }
  const size_t o_oc = P.push(oc), o_ocl = P.push(oc_last), o_ct = P.push(ct), o_ctr = P.push(ct_redo);
  const int n = (int)idx.size();
  for (int pass = 0; pass < passes; ++pass) {
    const size_t o_app = pass + 1 == passes ? o_ocl : o_oc;
    P.add(stage, [=](char *dev_t, cudaStream_t s) {
      tc::orthw_gram_kernel<<<dim3(max_chunks, max_pairs, n), tc::OW_THREADS, tc::OW_GRAM_SMEM, s>>>((const tc::OrthWCell *)(dev_t + o_oc)); LAUNCHED();
      chol_cluster_launch((const CholTask *)(dev_t + o_ct), n, max_k, s); g_launches += 2;
    });
    if (pass == 0) {
      add_tall_gram(P, stage, tg);
      P.add(stage, [=](char *dev_t, cudaStream_t s) { chol_cluster_launch((const CholTask *)(dev_t + o_ctr), n, max_k, s); g_launches += 2; });
    }
    P.add(stage, [=](char *dev_t, cudaStream_t s) {
      tc::orthw_apply_kernel<<<dim3(max_tiles, n), tc::OW_THREADS, tc::OW_APPLY_SMEM, s>>>((const tc::OrthWCell *)(dev_t + o_app)); LAUNCHED();
    });
  }
  if (want_fp32)
    P.add(stage, [=](char *dev_t, cudaStream_t s) {
      tc::orthw_norms_kernel<<<dim3((max_k + 7) / 8, n), 256, 0, s>>>((const tc::OrthWCell *)(dev_t + o_oc)); LAUNCHED();
    });
}

inline void add_orth_tc(Program &P, int stage, std::vector<CellWork> &ws, const std::vector<int> &idx, bool token_side, int passes,
                        bool want_fp32) {
  if (idx.empty()) return;
  static DeviceOnce once;
  once([] {
    cudaFuncSetAttribute(tc::orth_gram_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, tc::OR_SMEM_LIMIT);
    cudaFuncSetAttribute(tc::orth_apply_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, tc::OR_SMEM_LIMIT);
    cudaFuncSetAttribute(tc::cholinv_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)tc::cholinv_smem_bytes(tc::kCholInvMaxN));
  });
  add_orth_split(P, stage, ws, idx, token_side);
  std::vector<tc::OrthCell> oc, oc_last;      // the fp32 rows of Q are only written by the last pass, and only if someone reads them
  std::vector<tc::CholInvTask> ci;
  int max_chunks = 0, max_tiles = 0, max_kp = 0, max_k = 0;
  for (int i : idx) {
    CellWork &w = ws[i];
    const CellDesc &c = w.c;
    const int rpp = token_side ? c.T : kD, panels = token_side ? 1 : c.m;
    float *src = token_side ? w.S : w.Z;
    tc::OrthCell o;
    memset(&o, 0, sizeof o);
    {
      const uint64_t dims[3] = {(uint64_t)rpp, (uint64_t)w.kp, (uint64_t)panels};
      const uint64_t str[2] = {(uint64_t)rpp * 2, (uint64_t)w.kp * rpp * 2};
      const uint32_t box[3] = {64, (uint32_t)w.kp, 1};
      make_tmap_f16(&o.tmHi, w.Bhi, 3, dims, str, box);
      make_tmap_f16(&o.tmLo, w.Blo, 3, dims, str, box);
    }
    {
      const uint64_t dims[2] = {(uint64_t)w.kp, (uint64_t)w.kp};
      const uint64_t str[1] = {(uint64_t)w.kp * 2};
      const uint32_t box[2] = {64, (uint32_t)w.kp};
      make_tmap_f16(&o.tmLhi, w.orthLhi, 2, dims, str, box);
      make_tmap_f16(&o.tmLlo, w.orthLlo, 2, dims, str, box);
    }
    const int steps = panels * (rpp / 64);
    o.part = w.orthPart; o.Lhi = w.orthLhi; o.Llo = w.orthLlo; o.l_exp = w.orthExp;
    o.out32 = nullptr; o.ld = c.k; o.k = c.k; o.kp = w.kp; o.rpp = rpp; o.panels = panels;
    o.n_chunks = (steps + tc::OR_STEPS_PER_CTA - 1) / tc::OR_STEPS_PER_CTA;
    o.out_exp = ilog2_floor((long long)rpp * panels) / 2;
    o.status = w.status;
    oc.push_back(o);
    o.out32 = want_fp32 ? src : nullptr;
    oc_last.push_back(o);
    ci.push_back({w.orthPart, o.n_chunks, w.kp, nullptr, c.k, w.orthLhi, w.orthLlo, w.orthExp, nullptr, w.status, 1e-10});
    max_chunks = std::max(max_chunks, o.n_chunks);
    max_tiles = std::max(max_tiles, panels * (rpp / 128));
    max_kp = std::max(max_kp, w.kp); max_k = std::max(max_k, c.k);
    w.split_ready = token_side ? 1 : 2;
  }
  const size_t o_oc = P.push(oc), o_ocl = P.push(oc_last), o_ci = P.push(ci);
  const int n = (int)idx.size();
  const uint32_t tile = (uint32_t)max_kp * 128u;
  const int g_stages = std::max(2, std::min(6, (int)((tc::OR_SMEM_LIMIT - 16384 - 2048) / (2 * tile))));
  const size_t g_smem = (size_t)g_stages * 2 * tile + 16384 + 1024 + 1024;
  const size_t a_smem = (size_t)(4 + 2 * ((max_kp + 63) / 64)) * tile + 1024 + 1024;
  const size_t c_smem = tc::cholinv_smem_bytes(max_k);
  for (int pass = 0; pass < passes; ++pass) {
    const size_t o_app = pass + 1 == passes ? o_ocl : o_oc;
    P.add(stage, [=](char *dev_t, cudaStream_t s) {
      tc::orth_gram_kernel<<<dim3(max_chunks, n), tc::OR_THREADS, g_smem, s>>>((const tc::OrthCell *)(dev_t + o_oc), g_stages); LAUNCHED();
      tc::cholinv_kernel<<<n, tc::kCholInvThreads, c_smem, s>>>((const tc::CholInvTask *)(dev_t + o_ci)); LAUNCHED();
      tc::orth_apply_kernel<<<dim3(max_tiles, n), tc::OR_THREADS, a_smem, s>>>((const tc::OrthCell *)(dev_t + o_app)); LAUNCHED();
    });
  }
}

}  // namespace
