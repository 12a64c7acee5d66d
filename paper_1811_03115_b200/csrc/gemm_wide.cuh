// Projections of many token rows on the 5th-generation tensor cores (sm_100a): sessions whose passes carry more than
// 16 rows, the encoder, and the single operators.  Same operands and orientation as gemm_tc.cuh -- the weights are the
// MMA's M operand (128 features per tile), the tokens its N operand (16 to 256 per tile), activations as two bf16
// planes (PL = 2) or as one (PL = 1: the operators' plain bf16 inputs) -- but a different way of splitting K.
//
// What bounds these launches is not the tensor pipe: a layer projection of 20 to 320 rows is a few hundred KB to a few
// MB of shared-memory fill per SM and a chain of latencies around it.  K is therefore split over the CTAs of a
// cluster (up to 8 along grid.y), which puts every byte of a launch in flight at once, and the partial tiles never
// leave the chip: each CTA lays its tile out in its own shared memory, one cluster barrier later every CTA adds the
// S partial tiles of its share of the tokens through distributed shared memory, in rank order, and finishes them from
// registers with 8- and 16-byte stores.  (A partial tile in global memory, an arrival counter and a merge by the
// CTA that comes last took 7 us after the last MMA; this takes about 2.)
//
// The order of a sum is fixed by (features, K, split): the split is a property of the session and of the matrix, never
// of the number of rows in a launch.
#pragma once
#include "gemm_tc.cuh"

namespace bpd {
namespace tc {

constexpr int kWideThreads = 320;   // warp 0: TMA, warp 1: MMA + tensor-memory allocation, warps 2-9: epilogue
constexpr int kEpiWarps = 8;
constexpr int kWideBN = 256;        // tokens per tile at most
constexpr int kWidePitch = kBM + 4; // floats between the rows (tokens) of a tile in shared memory: 16-byte reads of a
                                    // warp and 4-byte writes of a warp both hit all banks once
constexpr int kWideStages = 8;

__host__ __device__ inline size_t wide_stage_bytes(int bn, int planes) { return (size_t)kBM * 128 + (size_t)planes * bn * 128; }
// (centred: 32 bytes per token behind the tile, see centre_shares; they change neither the stages nor the CTAs per SM:
// a tile with them is 80 KB at the 144 tokens that two CTAs take, 140 KB at 256)
__host__ __device__ inline size_t wide_smem_bytes(int bn, int planes, int stages, bool centred = false) {
  const size_t ring = stages * wide_stage_bytes(bn, planes), tile = (size_t)bn * (kWidePitch * sizeof(float) + (centred ? 32 : 0));
  return (ring > tile ? ring : tile) + 1024 /*alignment*/ + 256 /*barriers, control words*/;
}

__device__ __forceinline__ uint32_t map_to_rank(uint32_t saddr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(saddr), "r"(rank));
  return r;
}
__device__ __forceinline__ float4 ld_cluster_v4(uint32_t addr) {
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }

__device__ __forceinline__ uint2 pack4_bf16(const bf16 (&b)[4]) {
  return make_uint2((uint32_t)__bfloat16_as_ushort(b[0]) | ((uint32_t)__bfloat16_as_ushort(b[1]) << 16),
                    (uint32_t)__bfloat16_as_ushort(b[2]) | ((uint32_t)__bfloat16_as_ushort(b[3]) << 16));
}
// A 16-byte load from L2 that stays where it is written: the compiler otherwise sinks such loads to their first use,
// which turns a batch of independent loads into a chain of round trips.
__device__ __forceinline__ float4 ld_cg_v4_here(const float* ptr) {
  float4 v;
  asm volatile("ld.global.cg.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(ptr) : "memory");
  return v;
}

// Error code of a launch: a device word that keeps the first code, or (single operators) a word of pinned host memory.
__device__ __forceinline__ void report(const TcParams& p, int code) {
  if (p.error_on_host) *reinterpret_cast<volatile int*>(p.error) = code;
  else atomicCAS(p.error, 0, code);
}

// ---------------------------------------------------------------- finishing (token, four features) items
// A warp finishes the 128 features of a token, four consecutive ones per lane.  Per-thread constants of the four:
struct FinishCtx {
  float bias[4], gn[4], lns[4];
  bool folded;     // y = rstd * (acc - mean * ln_s) + ln_c; ln_c holds the bias (ln_s: 0 with centred planes, see centre_terms)
  int n, g;
};
template <int EPI>
__device__ __forceinline__ void finish_setup(const TcParams& p, int z, int tile, int lane, FinishCtx& c) {
  c.g = lane;
  c.n = tile * kBM + lane * 4;                       // first of the lane's four features (within the slice)
#pragma unroll
  for (int e = 0; e < 4; ++e) { c.bias[e] = 0.f; c.gn[e] = 0.f; c.lns[e] = 0.f; }
  c.folded = (p.stat_in != nullptr);
  if (c.n >= p.N) return;
  if (c.folded) {
    const float4 c4 = *reinterpret_cast<const float4*>(p.ln_c + c.n + p.zofs_ln * z);
    if (!p.ln_parts) {
      const float4 s4 = *reinterpret_cast<const float4*>(p.ln_s + c.n + p.zofs_ln * z);
      c.lns[0] = s4.x; c.lns[1] = s4.y; c.lns[2] = s4.z; c.lns[3] = s4.w;
    }
    c.bias[0] = c4.x; c.bias[1] = c4.y; c.bias[2] = c4.z; c.bias[3] = c4.w;
  } else if (p.bias && p.vec) {
    const uint2 bw = *reinterpret_cast<const uint2*>(p.bias + c.n + p.zofs_n * z);
    c.bias[0] = __uint_as_float(bw.x << 16); c.bias[1] = __uint_as_float(bw.x & 0xffff0000u);
    c.bias[2] = __uint_as_float(bw.y << 16); c.bias[3] = __uint_as_float(bw.y & 0xffff0000u);
  } else if (p.bias) {
#pragma unroll
    for (int e = 0; e < 4; ++e) if (c.n + e < p.N) c.bias[e] = __bfloat162float(p.bias[c.n + e]);
  }
  if (EPI == kTcResidual && p.g_next) {
    const uint2 gw = *reinterpret_cast<const uint2*>(p.g_next + c.n);
    c.gn[0] = __uint_as_float(gw.x << 16); c.gn[1] = __uint_as_float(gw.x & 0xffff0000u);
    c.gn[2] = __uint_as_float(gw.y << 16); c.gn[3] = __uint_as_float(gw.y & 0xffff0000u);
  }
}
// Planes of the updated stream, less `centre`, times the next layer norm's gain.
__device__ __forceinline__ void store_planes_next(const TcParams& p, const FinishCtx& c, int t, const float4& x, float centre) {
  const float v[4] = {x.x - centre, x.y - centre, x.z - centre, x.w - centre};
  bf16 hi[4], lo[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) split_bf16(v[e] * c.gn[e], hi[e], lo[e]);
  bf16* at = p.xg_hi + (long long)t * p.ldo + c.n;
  *reinterpret_cast<uint2*>(at) = pack4_bf16(hi);
  *reinterpret_cast<uint2*>(at + p.xg_plane) = pack4_bf16(lo);
}
// One item: token t (row tr of the tile), features c.n .. c.n + 3, accumulated values a; `old` is the residual stream's
// content, fetched by the caller (kTcResidual only), and returns the new content.
template <int EPI, bool CENTRED>
__device__ __forceinline__ void finish_item(const TcParams& p, const FinishCtx& c, int z, int t, int tr, const float4& a,
                                            float4& old, const unsigned long long* s_slot, const float* s_mean,
                                            const float* s_rstd) {
  const int n = c.n;
  float v[4] = {a.x + c.bias[0], a.y + c.bias[1], a.z + c.bias[2], a.w + c.bias[3]};
  if (c.folded) {
    const float mu = s_mean[tr], rs = s_rstd[tr];
    v[0] = rs * (a.x - mu * c.lns[0]) + c.bias[0]; v[1] = rs * (a.y - mu * c.lns[1]) + c.bias[1];
    v[2] = rs * (a.z - mu * c.lns[2]) + c.bias[2]; v[3] = rs * (a.w - mu * c.lns[3]) + c.bias[3];
  }
  if (p.relu) {
#pragma unroll
    for (int e = 0; e < 4; ++e) v[e] = fmaxf(v[e], 0.f);
  }
  if (EPI == kTcPlanes || EPI == kTcHeadOut) {
    const int nz = n + p.zofs_n * z;
    if (EPI == kTcHeadOut) {
      const float4 h = __ldg(reinterpret_cast<const float4*>(p.h + (size_t)t * p.d + (n % p.d)));
      const float pre[4] = {h.x, h.y, h.z, h.w};
#pragma unroll
      for (int e = 0; e < 4; ++e) v[e] = (p.head_identity && nz < p.d) ? pre[e] : v[e] + pre[e];
    }
    bf16 hi[4], lo[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) split_bf16(v[e], hi[e], lo[e]);
    const long long o = (long long)t * p.ldo + nz;
    *reinterpret_cast<uint2*>(p.out_hi + o) = pack4_bf16(hi);
    *reinterpret_cast<uint2*>(p.out_hi + o + p.plane) = pack4_bf16(lo);
  } else if (EPI == kTcF32) {
    float* y = p.out_f32 + p.zofs_out * z + (long long)t * p.ldo + n;
    if (p.vec) {
      *reinterpret_cast<float4*>(y) = make_float4(v[0], v[1], v[2], v[3]);
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e) if (n + e < p.N) y[e] = v[e];
    }
  } else if (EPI == kTcResidual) {
    const float xn[4] = {old.x + v[0], old.y + v[1], old.z + v[2], old.w + v[3]};
    old = make_float4(xn[0], xn[1], xn[2], xn[3]);
    *reinterpret_cast<float4*>(p.out_f32 + (long long)t * p.ldo + n) = old;
    if (!CENTRED && p.g_next) store_planes_next(p, c, t, old, 0.f);      // centred: by tile_stats
  } else if (EPI == kTcQkv) {
    const int d = p.d;
    if (n < d) {
      *reinterpret_cast<float4*>(p.out_f32 + (long long)t * p.ldo + n) = make_float4(v[0], v[1], v[2], v[3]);
    } else {
      const bf16 b4[4] = {__float2bfloat16_rn(v[0]), __float2bfloat16_rn(v[1]), __float2bfloat16_rn(v[2]), __float2bfloat16_rn(v[3])};
      bf16* dst = (n < 2 * d) ? p.kcache + s_slot[tr] + (n - d) : p.vcache + s_slot[tr] + (n - 2 * d);
      *reinterpret_cast<uint2*>(dst) = pack4_bf16(b4);
    }
  }
}
// Per-tile statistics of TB tokens at once (kTcResidual with stat_out): the warp holds the tile's 128 new values of
// each token, four per lane (N is a multiple of 128 here: every lane is live).  Sums of deviations from the token's
// first value in the tile, and of their squares, are reduced for all TB tokens together so that the shuffles of one
// token hide behind those of the others; mean and squared deviations about the mean follow exactly from the two.
template <int TB, bool CENTRED>
__device__ __forceinline__ void tile_stats(const TcParams& p, const FinishCtx& c, int t0, int tb, int hi, const float4 (&xn)[TB]) {
  float s1[TB], s2[TB], pivot[TB];
#pragma unroll
  for (int i = 0; i < TB; ++i) {
    pivot[i] = __shfl_sync(0xffffffffu, xn[i].x, 0);
    const float d0 = xn[i].x - pivot[i], d1 = xn[i].y - pivot[i], d2 = xn[i].z - pivot[i], d3 = xn[i].w - pivot[i];
    s1[i] = (d0 + d1) + (d2 + d3);
    s2[i] = (d0 * d0 + d1 * d1) + (d2 * d2 + d3 * d3);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
    for (int i = 0; i < TB; ++i) {
      s1[i] += __shfl_xor_sync(0xffffffffu, s1[i], o);
      s2[i] += __shfl_xor_sync(0xffffffffu, s2[i], o);
    }
  }
#pragma unroll
  for (int i = 0; i < TB; ++i) {
    const int tr = tb + kEpiWarps * i;
    if (tr < hi) {
      const float dm = s1[i] * (1.0f / kBM), mean = pivot[i] + dm;   // dm: mean - pivot
      if (c.g == 0) reinterpret_cast<float2*>(p.stat_out)[(size_t)(c.n / kBM) * p.stat_T + t0 + tr] = make_float2(mean, fmaxf(s2[i] - s1[i] * dm, 0.f));
      if (CENTRED) store_planes_next(p, c, t0 + tr, xn[i], mean);
    }
  }
}
// Centred planes (TcParams::ln_parts) leave out of a token's sum: over the up to eight tiles (d_model 1024), (tile mean -
// row mean) times the tile's share of ln_s.  A lane keeps the shares of its four features; the differences of a token are
// eight words of shared memory behind the tile.
__device__ __forceinline__ void centre_shares(const TcParams& p, const FinishCtx& c, int z, float4 (&share)[8]) {
#pragma unroll
  for (int q = 0; q < 8; ++q)
    share[q] = q < p.stat_parts ? __ldg(reinterpret_cast<const float4*>(p.ln_parts + (size_t)q * p.N + c.n + p.zofs_ln * z)) : make_float4(0.f, 0.f, 0.f, 0.f);
}
__device__ __forceinline__ void add_centre(const float4 (&share)[8], const float4* diff, float4& v) {
  const float4 a = diff[0], b = diff[1];
  const float w[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    v.x = fmaf(w[q], share[q].x, v.x); v.y = fmaf(w[q], share[q].y, v.y);
    v.z = fmaf(w[q], share[q].z, v.z); v.w = fmaf(w[q], share[q].w, v.w);
  }
}

// ---------------------------------------------------------------- the tokens of one CTA
// Tokens lo .. hi - 1 of the tile, whose S partial tiles lie in the shared memories of the cluster's CTAs (`tile_addr`:
// this CTA's, the same offset in every CTA).  Warp w takes tokens lo + w, lo + w + 8, ..., TB of them at a time:
// S x TB 16-byte reads (and the old residual values) are in flight per lane; the partial tiles are added in rank order.
template <int EPI, bool CENTRED, int S, int TB>
__device__ __forceinline__ void finish_tokens(const TcParams& p, int z, int t0, int lo, int hi, int tile, uint32_t tile_addr,
                                              const unsigned long long* s_slot, int warp, int lane, const float* s_mean,
                                              const float* s_rstd, const float4* s_diff) {
  FinishCtx c;
  finish_setup<EPI>(p, z, tile, lane, c);
  const bool live = c.n < p.N;                         // lanes beyond the last feature only keep the warp together
  constexpr bool TERMS = CENTRED && EPI != kTcResidual;
  float4 share[TERMS ? 8 : 1];
  if constexpr (TERMS) centre_shares(p, c, z, share);
  uint32_t part[S];
#pragma unroll
  for (int s = 0; s < S; ++s) part[s] = (S > 1 ? map_to_rank(tile_addr, s) : tile_addr) + lane * 16;
  for (int tb = lo + warp; tb < hi; tb += kEpiWarps * TB) {
    float4 old[TB], v[S][TB];
    int tok[TB];
    float thr[TB];
#pragma unroll
    for (int i = 0; i < TB; ++i) {
      const int tr = tb + kEpiWarps * i;
      old[i] = make_float4(0.f, 0.f, 0.f, 0.f);
      tok[i] = -1;
      if (tr < hi && live) {
        if (EPI == kTcResidual) old[i] = ld_cg_v4_here(p.out_f32 + (long long)(t0 + tr) * p.ldo + c.n);
        if (EPI == kTcArgmax && p.rank.cnt && (t0 + tr) % p.rank_kh == 0) {
          tok[i] = __ldg(&p.rank.tok[(t0 + tr) / p.rank_kh]);
          thr[i] = __ldg(&p.rank.thr[(t0 + tr) / p.rank_kh]);
        }
      }
    }
#pragma unroll
    for (int s = 0; s < S; ++s)
#pragma unroll
      for (int i = 0; i < TB; ++i) {
        const int tr = min(tb + kEpiWarps * i, hi - 1);
        v[s][i] = ld_cluster_v4(part[s] + (uint32_t)tr * (kWidePitch * 4));
      }
#pragma unroll
    for (int i = 0; i < TB; ++i) {
#pragma unroll
      for (int s = 1; s < S; ++s) {
        v[0][i].x += v[s][i].x; v[0][i].y += v[s][i].y; v[0][i].z += v[s][i].z; v[0][i].w += v[s][i].w;
      }
    }
    if constexpr (TERMS) {
#pragma unroll
      for (int i = 0; i < TB; ++i) add_centre(share, s_diff + 2 * min(tb + kEpiWarps * i, hi - 1), v[0][i]);
    }
    if constexpr (EPI == kTcArgmax) {
#pragma unroll
      for (int i = 0; i < TB; ++i) {
        const int tr = tb + kEpiWarps * i;
        if (tr >= hi) break;                           // uniform over the warp
        const float x[4] = {v[0][i].x, v[0][i].y, v[0][i].z, v[0][i].w};
        float best = -INFINITY;
        int at = 0x7fffffff;
#pragma unroll
        for (int e = 0; e < 4; ++e)
          if (c.n + e < p.N && (x[e] > best || at == 0x7fffffff)) { best = x[e]; at = c.n + e; }
        const unsigned b = __float_as_uint(best), ord = (b & 0x80000000u) ? ~b : (b | 0x80000000u);
        const unsigned m = __reduce_max_sync(0xffffffffu, at == 0x7fffffff ? 0u : ord);
        const int ix = __reduce_min_sync(0xffffffffu, (ord == m) ? at : 0x7fffffff);
        // one 64-bit atomic max per (tile, token): larger value wins, equal values go to the lower index; max is
        // order independent, so the result does not depend on which tile arrives first
        if (lane == 0)
          atomicMax(&p.best[(size_t)(t0 + tr) * kBestStride], ((unsigned long long)m << 32) | (unsigned long long)(0xffffffffu - (unsigned)ix));
        if (p.logits) {
#pragma unroll
          for (int e = 0; e < 4; ++e) if (c.n + e < p.N) p.logits[(size_t)(t0 + tr) * p.N + c.n + e] = x[e];
        }
        if (p.rank.cnt && (t0 + tr) % p.rank_kh == 0) {
          // top-n acceptance: how many of the tile's features beat the proposal that follows this position
          unsigned beats = 0;
          if (live && tok[i] >= 0) {
#pragma unroll
            for (int e = 0; e < 4; ++e)
              beats += (c.n + e < p.N && c.n + e != tok[i] && better(x[e], c.n + e, thr[i], tok[i])) ? 1u : 0u;
          }
          beats = __reduce_add_sync(0xffffffffu, beats);
          if (lane == 0 && beats) atomicAdd(&p.rank.cnt[(t0 + tr) / p.rank_kh], (int)beats);
        }
      }
    } else {
#pragma unroll
      for (int i = 0; i < TB; ++i) {
        const int tr = tb + kEpiWarps * i;
        if (tr < hi && live) finish_item<EPI, CENTRED>(p, c, z, t0 + tr, tr, v[0][i], old[i], s_slot, s_mean, s_rstd);
      }
      if (EPI == kTcResidual && p.stat_out) tile_stats<TB, CENTRED>(p, c, t0, tb, hi, old);
    }
  }
}

// ---------------------------------------------------------------- the kernel
// grid = (token tiles x slices, K splits, feature tiles), clusters of (1, K splits, 1): the CTAs that share a weight tile
// are neighbours in x.  tmA: weights [N, K]; tmBh / tmBl: activation planes [rows, K]; boxes (64, 128) and (64, bn).
// CENTRED: the planes read (kTcResidual: written) are, see
// TcParams::ln_parts.  Kernels of their own, because the code costs the decoder's launches more than it does the encoder's:
// in one kernel a pass of 320 rows took 1 % longer.
template <int EPI, int PL, bool CENTRED>
__global__ void __launch_bounds__(kWideThreads, 2)
gemm_wide_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmBh,
                 const __grid_constant__ CUtensorMap tmBl, const __grid_constant__ TcParams p, int ttiles, int stages,
                 int a_rows_per_slice, int b_cols_per_slice) {
  pdl_launch_dependents();
  extern __shared__ uint8_t smem_raw[];
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;      // swizzled tiles need 1024-byte alignment
  uint8_t* gen_base = smem_raw + (base - smem_u32(smem_raw));
  __shared__ __align__(8) unsigned long long s_bar[2 * kWideStages + 1];
  __shared__ uint32_t s_ctl[2];                                     // tensor-memory base, "this CTA merges the top-1"
  __shared__ float s_mean[kWideBN], s_rstd[kWideBN];
  __shared__ unsigned long long s_slot[EPI == kTcQkv ? kWideBN : 1];
  constexpr bool TERMS = CENTRED && EPI != kTcResidual;
  const int bn = p.bn;
  const uint32_t stage_sz = (uint32_t)wide_stage_bytes(bn, PL);
  const uint32_t bars = smem_u32(s_bar);                             // full[stages], empty[stages], accumulator
  const uint32_t acc_bar = bars + 8 * 2 * kWideStages;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int tile = blockIdx.z, split = blockIdx.y, S = p.splits;
  const int ttile = blockIdx.x % ttiles, slice = blockIdx.x / ttiles;
  const int t0 = ttile * bn;
  const int nt = min(bn, p.T - t0);                                  // live tokens in this tile
  const int total_chunks = (p.K + kBK - 1) / kBK;
  const int c0 = split * p.chunks_per_split;
  const int c1 = min(total_chunks, c0 + p.chunks_per_split);
  const int nchunks = max(0, c1 - c0);
  uint32_t ncols = 32;
  while ((int)ncols < bn) ncols <<= 1;

  if (threadIdx.x == 0) {
    for (int s = 0; s < stages; ++s) {
      mbar_init(bars + 8 * s, 1);
      mbar_init(bars + 8 * (kWideStages + s), 1);
    }
    mbar_init(acc_bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) tmem_alloc(smem_u32(&s_ctl[0]), ncols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = s_ctl[0];
  bool ok = true;

  if (warp == 0) {
    if (lane == 0) {
      // weights do not depend on the preceding kernel: the first stages' weight tiles are requested before the wait
      const int a_row = slice * a_rows_per_slice + tile * kBM;
      const int npre = min(nchunks, stages);
      const unsigned long long policy = l2_evict_first();
      auto load_w = [&](int it, int s) {
        mbar_expect_tx(bars + 8 * s, stage_sz);
        if (p.stream_weights) tma_load_2d_hint(base + s * stage_sz, &tmA, bars + 8 * s, (c0 + it) * kBK, a_row, policy);
        else tma_load_2d(base + s * stage_sz, &tmA, bars + 8 * s, (c0 + it) * kBK, a_row);
      };
      auto load_x = [&](int it, int s) {
        const uint32_t sx = base + s * stage_sz + kBM * 128;
        const int kx = slice * b_cols_per_slice + (c0 + it) * kBK;
        tma_load_2d(sx, &tmBh, bars + 8 * s, kx, t0);
        if (PL == 2) tma_load_2d(sx + bn * 128, &tmBl, bars + 8 * s, kx, t0);
      };
      for (int it = 0; it < npre; ++it) load_w(it, it);
      pdl_wait();
      const bool skip = p.all_done && *p.all_done;
      for (int it = 0; it < npre; ++it) load_x(it, it);
      int issued = npre;
      for (int it = npre; it < nchunks && !skip; ++it) {
        const int s = it % stages;
        if (!mbar_wait(bars + 8 * (kWideStages + s), ((it / stages) & 1) ^ 1)) { ok = false; break; }
        issued = it + 1;
        load_w(it, s);
        load_x(it, s);
      }
      if (!ok) report(p, 101);
      if (!ok || skip) {
        // nobody will consume what is in flight: give it a bounded chance to land before shared memory goes away
        for (int it = max(0, issued - stages); it < issued; ++it) mbar_wait(bars + 8 * (it % stages), (it / stages) & 1);
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    if (lane == 0) {
      const uint32_t idesc = instr_desc_bf16(bn);
      pdl_wait();
      const bool skip = p.all_done && *p.all_done;
      for (int it = 0; it < nchunks && !skip; ++it) {
        const int s = it % stages;
        if (!mbar_wait(bars + 8 * s, (it / stages) & 1)) { ok = false; break; }
        tc_fence_after();
        const uint32_t sa = base + s * stage_sz;
#pragma unroll
        for (int kk = 0; kk < kBK / 16; ++kk) {
          const uint64_t ad = smem_desc_sw128(sa + kk * 32);
          umma_f16(tmem, ad, smem_desc_sw128(sa + kBM * 128 + kk * 32), idesc, (it > 0 || kk > 0) ? 1u : 0u);
          if (PL == 2) umma_f16(tmem, ad, smem_desc_sw128(sa + kBM * 128 + bn * 128 + kk * 32), idesc, 1u);
        }
        umma_commit(bars + 8 * (kWideStages + s));    // frees the stage once these MMAs have read it
      }
      umma_commit(acc_bar);                           // accumulator complete
      if (!ok) report(p, 102);
    }
    __syncwarp();
  } else {
    pdl_wait();
    const bool skip = p.all_done && *p.all_done;
    const int et = threadIdx.x - 64, ew = warp - 2;   // 0..255, 0..7
    // this CTA's share of the tile's tokens
    const int per = (nt + S - 1) / S, lo = min(nt, split * per), hi = min(nt, lo + per);
    float diff[TERMS ? 8 : 1] = {};                  // tile means less the row's mean, of this thread's token
    if (EPI == kTcQkv && !skip) {
      const int tr = lo + et;
      if (tr < hi) {
        const int t = t0 + tr, b = t / p.rows_per_b, i = t % p.rows_per_b;
        const int pos = p.st.len[b] + i;
        const int page = p.st.page_table[b * p.st.pages_per_row + pos / kPage];
        s_slot[tr] = ((unsigned long long)page * kPage + (pos % kPage)) * p.d;
      }
    }
    if (EPI != kTcArgmax && p.stat_in && !skip && lo + et < hi) {
      // per-token statistics from the per-tile partial results of the kernel that wrote the stream: merged in tile
      // order (pairwise update of mean and sum of squared deviations), the same for every consumer
      const int tr = lo + et;
      const float2* sp = reinterpret_cast<const float2*>(p.stat_in) + (t0 + tr);
      float2 part[8];
      float mean = 0.f, m2 = 0.f, cnt = 0.f;
      for (int i0 = 0; i0 < p.stat_parts; i0 += 8) {
#pragma unroll
        for (int i = 0; i < 8; ++i)
          if (i0 + i < p.stat_parts) part[i] = __ldcg(sp + (size_t)(i0 + i) * p.stat_T);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          if (i0 + i < p.stat_parts) {
            const float nb = (float)kBM, tot = cnt + nb;
            const float delta = part[i].x - mean;
            mean += delta * (nb / tot);
            m2 += part[i].y + delta * delta * (cnt * nb / tot);
            cnt = tot;
          }
        }
      }
      s_mean[tr] = mean;
      s_rstd[tr] = rsqrtf(m2 / cnt + p.ln_eps);
      if constexpr (TERMS) {
#pragma unroll
        for (int i = 0; i < 8; ++i) diff[i] = i < p.stat_parts ? part[i].x - mean : 0.f;
      }
    }
    bool done = !skip;
    if (done && nchunks > 0) done = mbar_wait(acc_bar, 0);
    if (!done && !skip && lane == 0) report(p, 103);
    tc_fence_after();
    // the stages are free once the accumulator is complete: the tile goes there, one row per token.  A warp reads the
    // 32 tensor-memory lanes (features) its number allows; two warps share them and take every other 16 tokens.
    if (done) {
      const int q = warp & 3, row = q * 32 + lane;
      float* s_t = reinterpret_cast<float*>(gen_base);
      for (int cb = (ew >> 2) * 16; cb < bn; cb += 32) {
        float v[16];
        if (nchunks > 0) tmem_ld16(tmem + ((uint32_t)(q * 32) << 16) + cb, v);
        else {
#pragma unroll
          for (int c = 0; c < 16; ++c) v[c] = 0.f;
        }
#pragma unroll
        for (int c = 0; c < 16; ++c) s_t[(cb + c) * kWidePitch + row] = v[c];
      }
      if constexpr (TERMS) {
        float4* at = reinterpret_cast<float4*>(s_t + bn * kWidePitch) + 2 * (lo + et);
        if (lo + et < hi) {
          at[0] = make_float4(diff[0], diff[1], diff[2], diff[3]);
          at[1] = make_float4(diff[4], diff[5], diff[6], diff[7]);
        }
      }
    }
    s_ctl[1] = 0;
  }
  // every thread of every CTA takes part in the cluster barriers, whatever happened to it before
  const bool skip_all = p.all_done && *p.all_done;
  tc_fence_before();
  if (S > 1) { cluster_arrive(); cluster_wait(); } else __syncthreads();
  if (warp >= 2 && !skip_all) {
    const int et = threadIdx.x - 64, ew = warp - 2;
    const int per = (nt + S - 1) / S, lo = min(nt, split * per), hi = min(nt, lo + per);
    const float4* s_diff = reinterpret_cast<const float4*>(gen_base + (size_t)bn * kWidePitch * sizeof(float));
    if (S == 1) finish_tokens<EPI, CENTRED, 1, 4>(p, slice, t0, lo, hi, tile, base, s_slot, ew, lane, s_mean, s_rstd, s_diff);
    else if (S == 2) finish_tokens<EPI, CENTRED, 2, 4>(p, slice, t0, lo, hi, tile, base, s_slot, ew, lane, s_mean, s_rstd, s_diff);
    else if (S == 4) finish_tokens<EPI, CENTRED, 4, 2>(p, slice, t0, lo, hi, tile, base, s_slot, ew, lane, s_mean, s_rstd, s_diff);
    else finish_tokens<EPI, CENTRED, 8, 1>(p, slice, t0, lo, hi, tile, base, s_slot, ew, lane, s_mean, s_rstd, s_diff);
    if (EPI == kTcArgmax) {
      // the CTA that completes the last tile hands the winners out
      asm volatile("bar.sync 1, 256;" ::: "memory");
      if (et == 0) {
        const unsigned prev = atom_add_acq_rel(p.done_counter, 1u);
        s_ctl[1] = (prev == gridDim.x * gridDim.y * gridDim.z - 1) ? 1u : 0u;
      }
      asm volatile("bar.sync 1, 256;" ::: "memory");
      if (s_ctl[1]) {
        for (int t = et; t < p.T; t += 256) {
          const unsigned long long key = __ldcg(&p.best[(size_t)t * kBestStride]);
          p.out_idx[t] = (int)(0xffffffffu - (unsigned)(key & 0xffffffffull));
          if (p.out_val) p.out_val[t] = unpack_value(key);
          p.best[(size_t)t * kBestStride] = 0ull;                       // ready for the next launch
        }
        if (et == 0) *p.done_counter = 0;
      }
    }
  }
  if (S > 1) { cluster_arrive(); cluster_wait(); }    // a CTA's shared memory stays until its peers have read it
  else __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, ncols);
  }
}

}  // namespace tc
}  // namespace bpd
