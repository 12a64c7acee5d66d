// Host side of the tensor-core projection: TMA tensor maps, K-split planning and launches.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <math.h>

#include <algorithm>
#include <map>
#include <mutex>
#include <tuple>

#include "gemm_wide.cuh"
#include "host.hpp"

namespace bpd {
namespace tc {

// Resident CTA slots the planner aims to fill: 2 CTAs on each of the 148 SMs of a B200.  Constants of that chip, as are the
// cluster counts in wide_tiling: a plan fixes the order of sums, which a model's results should not owe to the device asked.
constexpr int kSms = 148;
constexpr int kSlots = 2 * kSms;
constexpr int kMinChunksPerSplit = 2;

struct Plan {
  int tiles, chunks, splits, chunks_per_split;
  int groups, group_chunks;   // of a split's chunks, see TcParams
};
// Launches of at most 16 token rows (gemm_tc.cuh): one token tile, two CTAs per SM, K split finely.  Depends on (N, K)
// only -- never on the number of tokens -- so that a position scored alone and the same position scored inside a
// block add up in the same order.
inline Plan plan_splits(int N, int K) {
  Plan pl;
  pl.tiles = (N + kBM - 1) / kBM;
  pl.chunks = (K + kBK - 1) / kBK;
  const int splits = std::max(1, std::min(pl.chunks / kMinChunksPerSplit, kSlots / pl.tiles));
  pl.chunks_per_split = (pl.chunks + splits - 1) / splits;
  pl.splits = (pl.chunks + pl.chunks_per_split - 1) / pl.chunks_per_split;
  pl.groups = pl.chunks_per_split >= 32 ? 8 : 1;
  pl.group_chunks = (pl.chunks_per_split + pl.groups - 1) / pl.groups;
  return pl;
}
// CTAs that share a split in a launch of `tiles` feature tiles: as many as the slots hold.
inline int plan_fine(const Plan& pl, int tiles) {
  int fine = 1;
  while (fine < pl.groups && tiles * pl.splits * fine * 2 <= kSlots) fine *= 2;
  return fine;
}

// Launches of the wide kernel (gemm_wide.cuh).  A tiling is (tokens per tile, CTAs per cluster = K splits); its cost in
// microseconds is estimated from what bounds these launches: shared-memory fill (every CTA stages 16 KB of weights and
// bn x planes x 128 bytes of activations per K chunk) and the exchange of the partial tiles inside the cluster.
struct WidePlan {
  int tiles, chunks, splits, chunks_per_split, bn, ttiles, stages;
  float cost;
};
constexpr size_t kWideSmemHalf = 108 * 1024;    // dynamic shared memory with two CTAs per SM (static: 4.3 KB, reserved: 1 KB)
constexpr size_t kWideSmemFull = 221 * 1024;
inline WidePlan wide_tiling(int N, int K, int T, int z, int planes, int splits, int ttiles) {
  WidePlan w;
  w.tiles = (N + kBM - 1) / kBM;
  w.chunks = (K + kBK - 1) / kBK;
  w.splits = splits;
  w.chunks_per_split = (w.chunks + splits - 1) / splits;
  w.ttiles = ttiles;
  w.bn = std::max(16, ((T + ttiles - 1) / ttiles + 15) / 16 * 16);
  // two CTAs per SM where at least two stages of each fit, else one with as many stages as there is room for
  int per_sm = 2;
  size_t room = kWideSmemHalf;
  if (wide_smem_bytes(w.bn, planes, std::min(2, w.chunks_per_split)) > kWideSmemHalf) { per_sm = 1; room = kWideSmemFull; }
  w.stages = 1;
  while (w.stages < kWideStages && w.stages < w.chunks_per_split && wide_smem_bytes(w.bn, planes, w.stages + 1) <= room) ++w.stages;
  // Fitted to 2300 timings of dependent launches (N 256..40960, K 512..40960, T 10..2560; the tiling it picks is on
  // average 2.6 % slower than the best one measured): a first round trip, the bytes of a chunk at what one SM takes in,
  // a refill of the ring per chunk beyond its depth, the exchange inside the cluster; all CTA slots of the GPU (clusters
  // of 4 and 8 do not fill every SM) in waves, and no faster than L2 and HBM deliver.
  const double ctas = (double)w.tiles * w.splits * w.ttiles * z;
  const double kb = wide_stage_bytes(w.bn, planes) / 1024.0;
  // (15 clusters of 8 are resident at one CTA per SM, 33 at two)
  const int full = kSms * per_sm, slots = splits >= 8 ? (per_sm == 1 ? 120 : 264) : (splits == 4 ? full * 11 / 12 : full);
  const double waves = ceil(ctas / slots), resident = std::min<double>(per_sm, ceil(ctas / kSms));
  const double in = 2.26 + w.chunks_per_split * kb * resident / 165.0 + std::max(0, w.chunks_per_split - w.stages) * 1.2 / w.stages;
  const double out = 0.0017 * w.bn / splits + (splits > 1 ? 0.022 * w.bn * (splits - 1) / splits : 0.0);
  const double deliver = std::max(ctas * w.chunks_per_split * kb / 13200.0, (double)z * w.tiles * w.chunks * 16.0 / 7600.0);
  w.cost = (float)std::max(waves * (in + out) * (per_sm == 1 ? 1.2 : 1.0), deliver + 2.26 + out);
  return w;
}
// The split of a matrix: chosen for `rows` token rows (the session's widest pass) and kept for every launch on it.
inline int wide_splits(int N, int K, int rows, int z, int planes) {
  int best = 1;
  float cost = 0;
  for (int s = 1; s <= 8; s *= 2) {
    if (s > 1 && s > (K + kBK - 1) / kBK) break;
    for (int tt = (rows + kWideBN - 1) / kWideBN; tt <= (rows + 31) / 32 || tt == 1; ++tt) {
      const WidePlan w = wide_tiling(N, K, rows, z, planes, s, tt);
      if ((long)(tt - 1) * w.bn >= rows) continue;                   // its last tile would be empty
      if (cost == 0 || w.cost < cost) { cost = w.cost; best = s; }
    }
  }
  return best;
}
// The token tiling of a launch of T rows, its split given.
inline WidePlan wide_plan(int N, int K, int T, int z, int planes, int splits) {
  WidePlan best;
  best.cost = -1;
  for (int tt = (T + kWideBN - 1) / kWideBN; tt <= (T + 31) / 32 || tt == 1; ++tt) {
    const WidePlan w = wide_tiling(N, K, T, z, planes, splits, tt);
    if ((long)(tt - 1) * w.bn >= T) continue;
    if (best.cost < 0 || w.cost < best.cost) best = w;
  }
  return best;
}

// The same with the split chosen for (plan_n, rows); a thread that repeats a launch keeps its plan (an operator call is
// a few microseconds, the search over tilings one or two).
inline WidePlan wide_plan_for(int N, int K, int T, int z, int planes, int plan_n, int rows) {
  struct Last { int key[7]; WidePlan plan; };
  static thread_local Last last = {{0, 0, 0, 0, 0, 0, 0}, {}};
  const int key[7] = {N, K, T, z, planes, plan_n, rows};
  if (memcmp(key, last.key, sizeof(key)) != 0) {
    last.plan = wide_plan(N, K, T, z, planes, wide_splits(plan_n, K, rows, z, planes));
    memcpy(last.key, key, sizeof(key));
  }
  return last.plan;
}

// fp32 elements of split-K workspace and arrival counters a launch of the few-row kernel needs.
constexpr int kNarrowBN = 16;
inline size_t ws_floats(int N, int K, int zslices) {
  const Plan pl = plan_splits(N, K);
  // launches of fewer tiles may split finer, up to kSlots CTAs
  return pl.splits == 1 && pl.groups == 1 ? 0 : std::max((size_t)zslices * pl.tiles * pl.splits, (size_t)kSlots) * kNarrowBN * kBM;
}
inline size_t counters_needed(int N, int zslices) { return (size_t)zslices * ((N + kBM - 1) / kBM); }

struct Scratch {
  float* ws; size_t ws_floats;
  unsigned* tile_counters; size_t n_counters;
  unsigned* done_counter;
  unsigned long long* best; size_t best_elems;
  int* error;
  int wide_rows;     // > 0: the wide kernel, its splits chosen for this many token rows; 0: the few-row kernel
  int l2_hints;      // 1: weights that a launch reads once are loaded "evict first"
  int error_on_host; // 1: `error` lies in pinned host memory (wide kernel only)
};

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

inline int get_encode_fn(EncodeTiledFn* out) {
  static EncodeTiledFn fn = nullptr;
  static std::mutex mu;
  std::lock_guard<std::mutex> lock(mu);
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    cudaError_t e = cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q);
    if (e != cudaSuccess || q != cudaDriverEntryPointSuccess || !p)
      return fail(BPD_E_CUDA, "cuTensorMapEncodeTiled is not available: %s", cudaGetErrorString(e));
    fn = reinterpret_cast<EncodeTiledFn>(p);
  }
  *out = fn;
  return BPD_OK;
}

constexpr size_t kMapCacheMax = 4096;   // descriptors kept per process (128 bytes each)

// bf16 matrix [rows, cols] with `ld` elements between rows; boxes of (64 columns, box_rows rows), 128-byte swizzle.
inline int make_map(const void* ptr, uint64_t rows, uint64_t cols, uint64_t ld, uint32_t box_rows, CUtensorMap* out) {
  typedef std::tuple<const void*, uint64_t, uint64_t, uint64_t, uint32_t> Key;
  static std::map<Key, CUtensorMap> cache;
  static std::mutex mu;
  const Key key(ptr, rows, cols, ld, box_rows);
  {
    std::lock_guard<std::mutex> lock(mu);
    auto it = cache.find(key);
    if (it != cache.end()) { *out = it->second; return BPD_OK; }
  }
  if ((uintptr_t)ptr % 16 || (ld * 2) % 16) return fail(BPD_E_INVALID, "tensor-map operand is not 16-byte aligned");
  if (box_rows < 1 || box_rows > 256) return fail(BPD_E_INVALID, "tensor-map box of %u rows", box_rows);
  EncodeTiledFn enc;
  int rc = get_encode_fn(&enc);
  if (rc) return rc;
  const cuuint64_t dims[2] = {cols, rows};
  const cuuint64_t strides[1] = {ld * 2};
  const cuuint32_t box[2] = {(cuuint32_t)kBK, box_rows};
  const cuuint32_t estr[2] = {1, 1};
  CUresult r = enc(out, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(ptr), dims, strides, box, estr,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return fail(BPD_E_CUDA, "cuTensorMapEncodeTiled failed with code %d", (int)r);
  std::lock_guard<std::mutex> lock(mu);
  // A descriptor is a pure function of its key, so an entry never goes stale (a freed and reused address yields
  // the same descriptor); the cache only saves the encode call.  Keep it bounded: sessions come and go in a
  // long-lived process, each with its own activation buffers.
  if (cache.size() >= kMapCacheMax) cache.clear();
  cache[key] = *out;
  return BPD_OK;
}

// A 3-D map (not cached): `layers` matrices of `rows` x `cols` elements of `elem_bytes` (2: bf16, 4: fp32), `ld` elements
// between rows and `layer_stride_bytes` between matrices; boxes of box_cols x box_rows x 1, swizzle chosen by the box's
// inner extent in bytes (128 -> 128-byte mode, 64 -> 64-byte mode).
inline int make_map_3d(const void* ptr, int elem_bytes, uint64_t layers, uint64_t layer_stride_bytes, uint64_t rows, uint64_t cols,
                       uint64_t ld, uint32_t box_cols, uint32_t box_rows, bool swizzle, CUtensorMap* out) {
  if ((uintptr_t)ptr % 16 || (ld * elem_bytes) % 16 || layer_stride_bytes % 16)
    return fail(BPD_E_INVALID, "tensor-map operand is not 16-byte aligned");
  if (box_rows < 1 || box_rows > 256 || box_cols < 1 || box_cols > 256) return fail(BPD_E_INVALID, "tensor-map box %u x %u", box_cols, box_rows);
  EncodeTiledFn enc;
  int rc = get_encode_fn(&enc);
  if (rc) return rc;
  const uint32_t inner = box_cols * (uint32_t)elem_bytes;
  CUtensorMapSwizzle sw = CU_TENSOR_MAP_SWIZZLE_NONE;
  if (swizzle && inner == 128) sw = CU_TENSOR_MAP_SWIZZLE_128B;
  else if (swizzle && inner == 64) sw = CU_TENSOR_MAP_SWIZZLE_64B;
  else if (swizzle) return fail(BPD_E_INVALID, "no swizzle mode for boxes of %u bytes per row", inner);
  const cuuint64_t dims[3] = {cols, rows, layers};
  const cuuint64_t strides[2] = {ld * (uint64_t)elem_bytes, layers > 1 ? layer_stride_bytes : ld * (uint64_t)elem_bytes * rows};
  const cuuint32_t box[3] = {box_cols, box_rows, 1};
  const cuuint32_t estr[3] = {1, 1, 1};
  CUresult r = enc(out, elem_bytes == 2 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3,
                   const_cast<void*>(ptr), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, sw,
                   CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return fail(BPD_E_CUDA, "cuTensorMapEncodeTiled (3-D) failed with code %d", (int)r);
  return BPD_OK;
}

struct Operands {
  const void* w; int w_rows;            // weights [w_rows, K] (all slices stacked)
  const void* x; long long x_plane;     // activation planes: hi at x, lo at x + x_plane (elements); 0: one plane (wide kernel only)
  long long ldx; int x_rows; int x_cols;  // allocated rows, total columns per row
};

// plan_n: the feature count the K split is planned for.  A launch that computes only the first features of a matrix
// (fewer heads) passes the full count so that every feature is summed in the same order either way.
// plan_rows: in a session with many rows, the row count the split is planned for when its results need not agree bit
// for bit with any other launch (the second stage of the lazy heads).
template <int EPI>
int launch(const Operands& op, int N, int K, int T, TcParams p, const Scratch& sc, cudaStream_t st, int zslices = 1,
           int a_rows_per_slice = 0, int b_cols_per_slice = 0, bool pdl = false, int plan_n = 0, int plan_rows = 0) {
  const int pn = plan_n > 0 ? plan_n : N;
  const int planes = op.x_plane > 0 ? 2 : 1;
  const bool wide = sc.wide_rows > 0;
  if (!wide && (T > kNarrowBN || planes != 2)) return fail(BPD_E_UNSUPPORTED, "%d token rows in a launch of the few-row projection kernel", T);
  if (EPI == kTcArgmax && (size_t)T > sc.best_elems) return fail(BPD_E_NOMEM, "top-1 workspace too small");
  WidePlan wp;
  Plan pl;
  int bn = kNarrowBN;
  if (wide) {
    wp = wide_plan_for(N, K, T, zslices, planes, pn, plan_rows > 0 ? plan_rows : sc.wide_rows);
    bn = wp.bn;
  } else {
    pl = plan_splits(pn, K);
    pl.tiles = (N + kBM - 1) / kBM;
    p.fine = plan_fine(pl, pl.tiles * zslices);
    p.groups = pl.groups; p.group_chunks = pl.group_chunks;
    pl.splits *= p.fine;
    const size_t need_ws = pl.splits == 1 ? 0 : (size_t)zslices * pl.tiles * pl.splits * bn * kBM;
    const size_t need_cnt = (size_t)zslices * pl.tiles;
    if (need_ws > sc.ws_floats || need_cnt > sc.n_counters)
      return fail(BPD_E_NOMEM, "split-K workspace too small (%zu floats, %zu counters needed)", need_ws, need_cnt);
  }
  CUtensorMap ma, mh, ml;
  int rc = make_map(op.w, (uint64_t)op.w_rows, (uint64_t)K, (uint64_t)K, kBM, &ma);
  if (rc) return rc;
  rc = make_map(op.x, (uint64_t)op.x_rows, (uint64_t)op.x_cols, (uint64_t)op.ldx, (uint32_t)bn, &mh);
  if (rc) return rc;
  ml = mh;
  if (planes == 2) rc = make_map(static_cast<const bf16*>(op.x) + op.x_plane, (uint64_t)op.x_rows, (uint64_t)op.x_cols, (uint64_t)op.ldx, (uint32_t)bn, &ml);
  if (rc) return rc;
  p.T = T; p.N = N; p.K = K; p.bn = bn;
  p.splits = wide ? wp.splits : pl.splits; p.chunks_per_split = wide ? wp.chunks_per_split : pl.chunks_per_split;
  p.ws = sc.ws; p.tile_counters = sc.tile_counters; p.done_counter = sc.done_counter;
  p.best = sc.best; p.error = sc.error; p.error_on_host = sc.error_on_host;
  p.stream_weights = ((!wide || wp.ttiles == 1) && sc.l2_hints) ? 1 : 0;
  if (!wide) {
    if (p.stat_in || p.stat_out) return fail(BPD_E_UNSUPPORTED, "per-tile layer-norm statistics in a launch of the few-row projection kernel");
    if constexpr (EPI == kTcArgmax) {
      return fail(BPD_E_UNSUPPORTED, "the few-row projection kernel has no top-1 epilogue");
    } else {
      if ((rc = ensure_smem_limit(reinterpret_cast<const void*>(gemm_tc_kernel<EPI>), smem_bytes(bn)))) return rc;
      BPD_CUDA(launch_k(gemm_tc_kernel<EPI>, dim3(pl.tiles, pl.splits, zslices), dim3(kThreads), smem_bytes(bn), st, pdl, ma, mh, ml, p,
                        zslices, a_rows_per_slice, b_cols_per_slice));
      return BPD_OK;
    }
  }
  {
    // vector stores in the epilogue: every row offset and pointer involved must allow them
    auto al = [](const void* q, size_t a) { return q == nullptr || (uintptr_t)q % a == 0; };
    p.vec = (N % 4 == 0 && p.ldo % 4 == 0 && p.plane % 4 == 0 && p.xg_plane % 4 == 0 && p.zofs_n % 4 == 0 && p.zofs_ln % 4 == 0 && p.zofs_out % 4 == 0 &&
             (p.d % 4 == 0) && al(p.out_f32, 16) && al(p.out_hi, 8) && al(p.xg_hi, 8) && al(p.h, 16) && al(p.bias, 8) &&
             al(p.g_next, 8) && al(p.kcache, 8) && al(p.vcache, 8)) ? 1 : 0;
  }
  if (p.ln_x || (!p.vec && EPI != kTcF32 && EPI != kTcArgmax)) return fail(BPD_E_UNSUPPORTED, "operands of the wide projection kernel are misaligned");
  if ((p.stat_in || p.stat_out) && !(p.vec && N % kBM == 0 && EPI != kTcArgmax))
    return fail(BPD_E_UNSUPPORTED, "per-tile layer-norm statistics need whole, aligned feature tiles (N = %d)", N);
  const void* kernel = planes == 2 && !p.ln_parts && !p.centred ? reinterpret_cast<const void*>(gemm_wide_kernel<EPI, 2, false>) : nullptr;
  if constexpr (EPI == kTcF32 || EPI == kTcArgmax) {
    if (planes == 1 && !p.ln_parts) kernel = reinterpret_cast<const void*>(gemm_wide_kernel<EPI, 1, false>);
  }
  if constexpr (EPI == kTcF32 || EPI == kTcPlanes || EPI == kTcResidual) {
    if (planes == 2 && (EPI == kTcResidual ? p.centred && p.stat_out : p.ln_parts && p.stat_in)) kernel = reinterpret_cast<const void*>(gemm_wide_kernel<EPI, 2, true>);
  }
  if (p.ln_parts && p.stat_parts > 8) return fail(BPD_E_UNSUPPORTED, "centred activations of %d tiles", p.stat_parts);
  if (!kernel) return fail(BPD_E_UNSUPPORTED, "single-plane or centred activations with this epilogue");
  const size_t smem = wide_smem_bytes(bn, planes, wp.stages, p.ln_parts != nullptr);
  if ((rc = ensure_smem_limit(kernel, smem))) return rc;
  BPD_CUDA(launch_cluster(kernel, dim3(wp.ttiles * zslices, wp.splits, wp.tiles), dim3(kWideThreads), smem, st, pdl, wp.splits,
                          ma, mh, ml, p, wp.ttiles, wp.stages, a_rows_per_slice, b_cols_per_slice));
  return BPD_OK;
}

#define BPD_TC_LAUNCH(EPI) \
  template int launch<EPI>(const Operands&, int, int, int, TcParams, const Scratch&, cudaStream_t, int, int, int, bool, int, int)
// instantiated in gemm_tc.cu
extern BPD_TC_LAUNCH(kTcPlanes);
extern BPD_TC_LAUNCH(kTcF32);
extern BPD_TC_LAUNCH(kTcResidual);
extern BPD_TC_LAUNCH(kTcQkv);
extern BPD_TC_LAUNCH(kTcHeadOut);
extern BPD_TC_LAUNCH(kTcArgmax);

}  // namespace tc
}  // namespace bpd
