// Weight-streaming projection on the 5th-generation tensor cores (sm_100a):
//   y[t][n] = sum_c x[t][c] * w[n][c]        t < T tokens (few), n < N features (many)
// The weight matrix is the MMA's M operand (128 features per tile), the tokens are
// its N operand.  Weights (bf16, [N, K] row-major) and activations (two bf16
// planes hi + lo that together carry an fp32 value, [rows, K] row-major) are
// brought into 128-byte-swizzled shared memory by TMA; one elected thread issues
// tcgen05.mma with the fp32 accumulator in tensor memory; four warps read it
// back with tcgen05.ld and run the fused epilogue.  K can be split over CTAs
// (grid.y): partial tiles go to a workspace and the CTA that arrives last for a
// tile adds them in split order, so the summation order is fixed by (N, K) alone.
//
// Every wait on an mbarrier is bounded; on expiry the CTA records an error code,
// skips its remaining work, waits (bounded) for copies in flight, frees its
// tensor memory and returns.
#pragma once
#include <type_traits>
#include <cuda.h>

#include "common.cuh"

namespace bpd {
namespace tc {

constexpr int kBM = 128;          // features per tile (MMA M)
constexpr int kBK = 64;           // K elements per pipeline stage (128 bytes of bf16: one swizzle row)
constexpr int kThreads = 192;     // warp 0: TMA, warp 1: MMA + tensor-memory allocation, warps 2-5: epilogue
constexpr int kMaxBN = 16;        // tokens per CTA (MMA N); wider launches take gemm_wide.cuh
constexpr unsigned long long kSpinCycles = 2000000000ull;   // about a second

enum TcEpilogue {
  kTcPlanes = 0,    // out planes (hi, lo) = split(act(v + bias))
  kTcF32 = 1,       // out fp32 = act(v + bias)
  kTcResidual = 2,  // x fp32 += v + bias
  kTcQkv = 3,       // n < d: q fp32; else key / value (bf16) into the paged cache
  kTcHeadOut = 4,   // out planes = split(v + bias + h[t][n mod d])
  kTcArgmax = 5     // per-token top-1 over all features (two-level merge), optional logits dump
};

struct TcParams {
  int T, N, K;                 // tokens in this launch, features, reduction length
  int bn;                      // MMA N: T rounded up to 16 (per token tile)
  int splits;                  // grid.y
  int chunks_per_split;        // K chunks (of kBK) each split owns
  // few-row kernel: a split's chunks are summed in `groups` (1 or 8) groups of group_chunks, the groups' sums as a binary
  // tree; `fine` CTAs share a split, each a subtree, so a launch of few feature tiles can use more CTAs and still
  // add up in the order of the launch it was planned for
  int groups, group_chunks, fine;
  const bf16* bias;            // [N] or null
  int relu;
  // outputs
  bf16* out_hi; long long plane; long long ldo;   // planes: lo plane = hi + plane
  float* out_f32;              // kTcF32 / kTcResidual / kTcQkv(q): [T, ldo]
  const float* h; int d;       // kTcHeadOut residual; kTcQkv model width
  int head_identity;
  int zofs_n;                  // column offset of this z-slice inside the output row (block-diagonal heads)
  int zofs_ln; long long zofs_out;   // wide kernel: offset of a z-slice in ln_s / ln_c, and in out_f32 (kTcF32)
  bf16* kcache; bf16* vcache;  // kTcQkv
  RowState st; int rows_per_b;
  // split-K workspace
  float* ws;                   // [z][tile][split][bn][128]
  unsigned* tile_counters;     // [z][tiles]
  // top-1
  unsigned long long* best;         // [T][kBestStride] packed (orderable value, ~index) in the first word of each
                                    // token's 128 bytes, zero between launches
  unsigned* done_counter;           // [1]
  int* out_idx; float* out_val; float* logits;
  RankState rank; int rank_kh;      // top-n acceptance: count entries beating each proposal (rank.cnt null = off)
  // layer norm folded into the projection: the activation planes hold x * gain (not normalised); the
  // epilogue finishes y = rstd * (acc - mean * ln_s[n]) + ln_c[n] with per-token statistics of ln_x
  const float* ln_x; int ln_d; float ln_eps;   // residual stream [rows, ln_d] fp32, or null
  const float* ln_s; const float* ln_c;        // [N]: sum_c gain_c w[n][c]  and  sum_c shift_c w[n][c] + bias[n]
  // wide kernel, `centred`: the planes hold (x - m) * gain, m the mean of the token's 128 features of the tile (stat_in),
  // and y = rstd * (acc + sum_i (m_i - mean) ln_parts[i][n]) + ln_c[n]: a row's mean, however large against its
  // deviations, costs the planes no bits
  const float* ln_parts; int centred;          // [stat_parts][N] shares of ln_s (consumer); 1: write such planes (producer)
  // kTcResidual: also write planes of the updated stream times the next layer norm's gain
  const bf16* g_next; bf16* xg_hi; long long xg_plane;
  // Wide token tiles (more than 16 tokens) cannot afford to read whole rows of the residual stream for the folded
  // layer norm.  There the kernel that updates the stream also writes, per (128-feature tile, token), the mean and
  // the sum of squared deviations of its 128 new values (stat_out, [tiles][stat_T][2]); the projection that
  // consumes the normalised stream merges the stat_parts tiles of a token in tile order (stat_in).
  float* stat_out; const float* stat_in; int stat_parts; int stat_T;
  int* error;                  // error word
  int error_on_host;           // 1 (wide kernel only): the word lies in pinned host memory
  const int* all_done;
  int stream_weights;          // 1: the weights are read once per launch (one token tile): load them "evict first"
  int vec;                     // 1: wide token tiles finish through shared memory with 8- and 16-byte stores (the
                               // host has checked sizes and alignment)
};

// ---------------------------------------------------------------- PTX wrappers
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ uint32_t mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
  return ok;
}
// The same without waiting at all: try_wait may put the thread to sleep first.
__device__ __forceinline__ uint32_t mbar_test(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
  return ok;
}
// Bounded wait: false if the phase did not complete within about a second.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, unsigned long long limit_cycles = kSpinCycles) {
  if (mbar_try_wait(bar, parity)) return true;
  const unsigned long long t0 = clock64();
  for (;;) {
#pragma unroll 1
    for (int i = 0; i < 256; ++i)
      if (mbar_try_wait(bar, parity)) return true;
    if ((unsigned long long)(clock64() - t0) > limit_cycles) return false;
  }
}
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int x, int y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
      ::"r"(dst), "l"(map), "r"(bar), "r"(x), "r"(y) : "memory");
}
// Same with an L2 policy: weights that are read once per pass are marked "evict first", so that streaming
// hundreds of MB through the 126 MB L2 does not push out what every pass reads again (caches, small vectors).
__device__ __forceinline__ unsigned long long l2_evict_first() {
  unsigned long long pol;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
  return pol;
}
__device__ __forceinline__ void tma_load_2d_hint(uint32_t dst, const CUtensorMap* map, uint32_t bar, int x, int y,
                                                 unsigned long long policy) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%3, %4}], [%2], %5;"
      ::"r"(dst), "l"(map), "r"(bar), "r"(x), "r"(y), "l"(policy) : "memory");
}
__device__ __forceinline__ void tmem_alloc(uint32_t dst_smem, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst_smem), "r"(ncols) : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void umma_f16(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate) : "memory");
}
__device__ __forceinline__ void umma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
// 16 consecutive fp32 columns of this thread's tensor-memory lane.
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16]) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr) : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// Shared-memory operand descriptor: K-major rows of 128 bytes, 128-byte swizzle,
// 8-row groups 1024 bytes apart.
__device__ __forceinline__ uint64_t smem_desc_sw128(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3ffff) >> 4);          // start address, 16-byte units
  d |= (uint64_t)1 << 16;                           // leading byte offset (unused for swizzled K-major)
  d |= (uint64_t)(1024 >> 4) << 32;                 // stride byte offset between 8-row groups
  d |= (uint64_t)1 << 46;                           // descriptor version
  d |= (uint64_t)2 << 61;                           // layout: 128-byte swizzle
  return d;
}
// Instruction descriptor: bf16 x bf16 -> fp32, both operands K-major, M = 128.
__device__ __forceinline__ uint32_t instr_desc_bf16(int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(kBM >> 4) << 24);
}

__device__ __forceinline__ void split_bf16(float v, bf16& hi, bf16& lo) {
  hi = __float2bfloat16_rn(v);
  lo = __float2bfloat16_rn(v - __bfloat162float(hi));
}

// Shared-memory footprint of one CTA.
__host__ __device__ inline size_t stage_bytes(int bn) { return (size_t)kBM * 128 + 2 * (size_t)bn * 128; }
constexpr int kStages = 5;        // K chunks in flight; 101 KB at 16 tokens, so two CTAs fit on an SM
__host__ __device__ inline size_t smem_bytes(int bn) { return kStages * stage_bytes(bn) + 1024 /*alignment*/ + 256; }

// ---------------------------------------------------------------- final epilogue for one (feature, token)
// Finishes up to 8 tokens of one feature.  Everything that has to be read (old residual values, the head
// residual, cache slots) is fetched for all tokens first, so the loads overlap instead of queueing behind
// the stores of the previous token.
template <int EPI>
__device__ __forceinline__ void tc_store8(const TcParams& p, int z, int t_first, int ntok, int n, const float (&vin)[8],
                                          const float* s_mean, const float* s_rstd, int stat0,
                                          const unsigned long long* s_slot) {
  float lns = 0.f, lnc = 0.f, bias = 0.f, gnext = 0.f;
  if (p.ln_x) { lns = p.ln_s[n]; lnc = p.ln_c[n]; }
  else if (p.bias) bias = __bfloat162float(p.bias[n + p.zofs_n * z]);
  if (EPI == kTcResidual && p.g_next) gnext = __bfloat162float(p.g_next[n]);
  float pre[8];
  const bool need_old = (EPI == kTcResidual) && p.g_next != nullptr;   // otherwise the add is a fire-and-forget reduction
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    pre[c] = 0.f;
    if (c < ntok) {
      const int t = t_first + c;
      if (need_old) pre[c] = p.out_f32[(long long)t * p.ldo + n];
      if (EPI == kTcHeadOut) pre[c] = __ldg(&p.h[(size_t)t * p.d + (n % p.d)]);
    }
  }
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    if (c < ntok) {
      const int t = t_first + c;
      float v = vin[c];
      if (p.ln_x) v = s_rstd[(stat0 + c) & 15] * (v - s_mean[(stat0 + c) & 15] * lns) + lnc;
      else v += bias;
      if (p.relu) v = fmaxf(v, 0.f);
      if (EPI == kTcPlanes) {
        bf16 hi, lo;
        split_bf16(v, hi, lo);
        const long long o = (long long)t * p.ldo + n + (long long)p.zofs_n * z;
        p.out_hi[o] = hi;
        p.out_hi[o + p.plane] = lo;
      } else if (EPI == kTcF32) {
        p.out_f32[(long long)t * p.ldo + n] = v;
      } else if (EPI == kTcResidual) {
        if (!need_old) {
          atomicAdd(&p.out_f32[(long long)t * p.ldo + n], v);   // single writer per element: just x += v without a read
          continue;
        }
        const float xnew = pre[c] + v;
        p.out_f32[(long long)t * p.ldo + n] = xnew;
        if (p.g_next) {
          bf16 hi, lo;
          split_bf16(xnew * gnext, hi, lo);
          p.xg_hi[(long long)t * p.ldo + n] = hi;
          p.xg_hi[(long long)t * p.ldo + n + p.xg_plane] = lo;
        }
      } else if (EPI == kTcHeadOut) {
        const int nz = n + p.zofs_n * z;
        v = (p.head_identity && nz < p.d) ? pre[c] : v + pre[c];
        bf16 hi, lo;
        split_bf16(v, hi, lo);
        const long long o = (long long)t * p.ldo + nz;
        p.out_hi[o] = hi;
        p.out_hi[o + p.plane] = lo;
      } else if (EPI == kTcQkv) {
        const int d = p.d;
        if (n < d) p.out_f32[(long long)t * p.ldo + n] = v;
        else if (n < 2 * d) p.kcache[s_slot[stat0 + c] + (n - d)] = __float2bfloat16_rn(v);
        else p.vcache[s_slot[stat0 + c] + (n - 2 * d)] = __float2bfloat16_rn(v);
      }
    }
  }
}

// ---------------------------------------------------------------- bounded-wait self test
// One CTA waits on an mbarrier that nothing ever arrives on, gives up after `limit_cycles`, records the same
// error code the projection kernel would and returns normally: the context stays usable.
static __global__ void wait_probe_kernel(int* error, unsigned long long limit_cycles) {
  __shared__ __align__(8) unsigned long long bar;
  const uint32_t b = smem_u32(&bar);
  if (threadIdx.x == 0) {
    mbar_init(b, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    if (!mbar_wait(b, 0, limit_cycles)) atomicCAS(error, 0, 103);
  }
}

// ---------------------------------------------------------------- epilogue of one (tile, split) unit
// Called by the four epilogue warps (128 threads, named barrier 1).
struct EpiShared {
  float* s_mean; float* s_rstd;
  unsigned long long* s_slot;
  volatile uint32_t* ctl;       // [1] reduces the tile, [3] accumulator arrived
};
struct EpiUnit {
  uint32_t tmem, acc_bar, acc_parity;
  int tile, split, slice, zidx, ntiles, t0, nt, bn, nchunks;
  int acc_groups, acc_live;     // sub-accumulators of this CTA (16 columns each), those with chunks
  bool skip;
};
// Sum of the CTA's sub-accumulators (16 tensor-memory columns each) for this thread's lane: a binary tree over `groups`
// (1, 2, 4 or 8), of which the first `live` hold anything.
__device__ __forceinline__ void sum_groups(uint32_t taddr, int groups, int live, float (&v)[16]) {
  auto leaf = [&](int g, float (&x)[16]) {
    if (g < live) tmem_ld16(taddr + g * 16, x);
    else {
#pragma unroll
      for (int c = 0; c < 16; ++c) x[c] = 0.f;
    }
  };
  auto add = [](float (&x)[16], const float (&y)[16]) {
#pragma unroll
    for (int c = 0; c < 16; ++c) x[c] += y[c];
  };
  leaf(0, v);
  if (groups > 1) { float a[16]; leaf(1, a); add(v, a); }
  if (groups > 2) { float a[16], b[16]; leaf(2, a); leaf(3, b); add(a, b); add(v, a); }
  if (groups > 4) {
    float a[16], b[16], c[16];
    leaf(4, a); leaf(5, b); add(a, b);
    leaf(6, b); leaf(7, c); add(b, c);
    add(a, b);
    add(v, a);
  }
}

template <int EPI>
__device__ __forceinline__ void tc_epilogue(const TcParams& p, const EpiShared& sh, const EpiUnit& u, int warp, int lane) {
  float* s_mean = sh.s_mean;
  float* s_rstd = sh.s_rstd;
  unsigned long long* s_slot = sh.s_slot;
  volatile uint32_t* ctl = sh.ctl;
  const uint32_t tmem = u.tmem;
  const int tile = u.tile, split = u.split, slice = u.slice, t0 = u.t0, nt = u.nt, bn = u.bn, nchunks = u.nchunks;
  const bool skip = u.skip;
  const int q = warp & 3;                          // tensor-memory lane quarter this warp may read
  const int row = q * 32 + lane;
  const int n = tile * kBM + row;                  // feature index within the slice
  const int et = threadIdx.x - 64;                 // 0..127
  if (EPI == kTcQkv && !skip && et < nt) {
    const int t = t0 + et;
    const int b = t / p.rows_per_b, i = t % p.rows_per_b;
    const int pos = p.st.len[b] + i;
    const int page = p.st.page_table[b * p.st.pages_per_row + pos / kPage];
    s_slot[et] = ((unsigned long long)page * kPage + (pos % kPage)) * p.d;
  }
  if (p.ln_x && !skip) {
    // per-token mean and 1/std of the residual stream, computed while the main loop runs: 8 threads per
    // token (at most 16 tokens per tile in this mode), two passes, fixed order
    const int tr = et >> 3, part = et & 7;
    const int trc = min(tr, nt - 1);               // threads beyond the live tokens shadow the last one
    const float4* xr = reinterpret_cast<const float4*>(p.ln_x + (size_t)(t0 + trc) * p.ln_d);
    const int nv = p.ln_d >> 2;
    float sum = 0.f;
#pragma unroll 8
    for (int i = part; i < nv; i += 8) { const float4 a = xr[i]; sum += (a.x + a.y) + (a.z + a.w); }
    sum += __shfl_xor_sync(0xffffffffu, sum, 1);
    sum += __shfl_xor_sync(0xffffffffu, sum, 2);
    sum += __shfl_xor_sync(0xffffffffu, sum, 4);
    const float mean = sum / (float)p.ln_d;
    float sq = 0.f;
#pragma unroll 8
    for (int i = part; i < nv; i += 8) {
      const float4 a = xr[i];
      const float d0 = a.x - mean, d1 = a.y - mean, d2 = a.z - mean, d3 = a.w - mean;
      sq += (d0 * d0 + d1 * d1) + (d2 * d2 + d3 * d3);
    }
    sq += __shfl_xor_sync(0xffffffffu, sq, 1);
    sq += __shfl_xor_sync(0xffffffffu, sq, 2);
    sq += __shfl_xor_sync(0xffffffffu, sq, 4);
    const float rstd = rsqrtf(sq / (float)p.ln_d + p.ln_eps);
    if (part == 0 && tr < nt) { s_mean[tr] = mean; s_rstd[tr] = rstd; }
  }
  // one thread waits for the accumulator; the other 127 learn the outcome through the named barrier
  if (et == 0) {
    bool done = !skip;
    if (nchunks > 0 && !skip) done = mbar_wait(u.acc_bar, u.acc_parity);
    if (!done && !skip) atomicCAS(p.error, 0, 103);
    ctl[3] = done ? 1u : 0u;
  }
  asm volatile("bar.sync 1, 128;" ::: "memory");
  const bool ok = (ctl[3] != 0);
  tc_fence_after();
  const int ntiles = u.ntiles;
  const bool direct = (p.splits == 1);
  float* wsz = p.ws + ((size_t)u.zidx * ntiles + tile) * p.splits * (size_t)bn * kBM;
  if (ok) {
    float v[16];
    sum_groups(tmem + ((uint32_t)(q * 32) << 16), u.acc_groups, u.acc_live, v);
    if (direct) {
      if (n < p.N) {
        const float lo8[8] = {v[0], v[1], v[2], v[3], v[4], v[5], v[6], v[7]};
        const float hi8[8] = {v[8], v[9], v[10], v[11], v[12], v[13], v[14], v[15]};
        tc_store8<EPI>(p, slice, t0, min(8, nt), n, lo8, s_mean, s_rstd, 0, s_slot);
        tc_store8<EPI>(p, slice, t0 + 8, min(8, nt - 8), n, hi8, s_mean, s_rstd, 8, s_slot);
      }
    } else {
      // partial tile -> workspace [split][token][128], coalesced over features
#pragma unroll
      for (int c = 0; c < 16; ++c)
        if (c < nt) wsz[((size_t)split * bn + c) * kBM + row] = v[c];
      asm volatile("bar.sync 1, 128;" ::: "memory");
      if (et == 0) {
        const unsigned prev = atom_add_acq_rel(&p.tile_counters[(size_t)u.zidx * ntiles + tile], 1u);
        ctl[1] = (prev == (unsigned)p.splits - 1) ? 1u : 0u;
      }
      asm volatile("bar.sync 1, 128;" ::: "memory");
      if (ctl[1]) {
        // Splits are added in split order.  The partial tiles sit in L2 and every load is a round trip of about a
        // microsecond, so as many as the registers hold are issued together: G tokens x SB splits = 64 per thread.
        constexpr int G = 8, SB = 8;
        for (int cg = 0; cg < nt; cg += G) {
          float acc[G];
#pragma unroll
          for (int c = 0; c < G; ++c) acc[c] = 0.f;
          for (int s0 = 0; s0 < p.splits; s0 += SB) {
            float v[SB][G];
#pragma unroll
            for (int ss = 0; ss < SB; ++ss)
#pragma unroll
              for (int c = 0; c < G; ++c)
                v[ss][c] = (s0 + ss < p.splits && cg + c < nt)
                               ? __ldcg(&wsz[((size_t)(s0 + ss) * bn + cg + c) * kBM + row]) : 0.f;
            // the `fine` parts of a split first (a binary tree), then the splits in order
            if (p.fine > 1) {
#pragma unroll
              for (int ss = 0; ss < SB; ss += 2)
#pragma unroll
                for (int c = 0; c < G; ++c) v[ss][c] += v[ss + 1][c];
            }
            if (p.fine > 2) {
#pragma unroll
              for (int ss = 0; ss < SB; ss += 4)
#pragma unroll
                for (int c = 0; c < G; ++c) v[ss][c] += v[ss + 2][c];
            }
            if (p.fine > 4) {
#pragma unroll
              for (int c = 0; c < G; ++c) v[0][c] += v[4][c];
            }
#pragma unroll
            for (int ss = 0; ss < SB; ++ss) {
              if (ss % p.fine == 0) {
#pragma unroll
                for (int c = 0; c < G; ++c) acc[c] += v[ss][c];
              }
            }
          }
          if (n < p.N) tc_store8<EPI>(p, slice, t0 + cg, min(8, nt - cg), n, acc, s_mean, s_rstd, cg, s_slot);
        }
        if (et == 0) p.tile_counters[(size_t)u.zidx * ntiles + tile] = 0;   // ready for the next launch
      }
    }
  }
}

// ---------------------------------------------------------------- the kernel
// grid = (feature tiles, K splits, z), z = token tile * zslices + slice (slices: block-diagonal heads).
// tmA: weights [N, K]; tmBh / tmBl: activation planes [rows, K]; box = (64, 128) and (64, bn).
template <int EPI>
__global__ void __launch_bounds__(kThreads)
gemm_tc_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmBh,
               const __grid_constant__ CUtensorMap tmBl, TcParams p, int zslices, int a_rows_per_slice,
               int b_cols_per_slice) {
  pdl_launch_dependents();
  extern __shared__ uint8_t smem_raw[];
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;      // swizzled tiles need 1024-byte alignment
  uint8_t* gen_base = smem_raw + (base - smem_u32(smem_raw));
  const int bn = p.bn;
  const uint32_t stage_sz = (uint32_t)stage_bytes(bn);
  const uint32_t bars = base + kStages * stage_sz;                   // full[kStages], empty[kStages], accum
  volatile uint32_t* ctl = reinterpret_cast<volatile uint32_t*>(gen_base + kStages * stage_sz + 128);
  // ctl[0] = tensor-memory base, ctl[1] = "this CTA reduces the tile", ctl[3] = "the accumulator arrived"
  __shared__ float s_mean[kMaxBN], s_rstd[kMaxBN];
  __shared__ unsigned long long s_slot[kMaxBN];   // kTcQkv: cache slot (element offset) of every token of the tile

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int tile = blockIdx.x, split = blockIdx.y;
  const int ttile = blockIdx.z / zslices, slice = blockIdx.z % zslices;
  const int t0 = ttile * bn;
  const int nt = min(bn, p.T - t0);                                  // live tokens in this tile
  const int total_chunks = (p.K + kBK - 1) / kBK;
  // this CTA's part of its split: acc_groups of the groups
  const int acc_groups = p.groups / p.fine, part0 = (split / p.fine) * p.chunks_per_split;
  const int c0 = part0 + (split % p.fine) * acc_groups * p.group_chunks;
  const int c1 = min(min(total_chunks, part0 + p.chunks_per_split), c0 + acc_groups * p.group_chunks);
  const int nchunks = max(0, c1 - c0);
  const uint32_t ncols = acc_groups > 4 ? 128 : (acc_groups > 2 ? 64 : 32);

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(bars + 8 * s, 1);
      mbar_init(bars + 8 * (kStages + s), 1);
    }
    mbar_init(bars + 8 * 2 * kStages, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    ctl[1] = 0;
  }
  if (warp == 1) tmem_alloc(base + kStages * stage_sz + 128, ncols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = ctl[0];
  bool ok = true;

  if (warp == 0 && lane == 0) {
    // ---------------- TMA producer.  Weights do not depend on the preceding kernel: the first stages'
    // weight tiles are requested before waiting for it; activations only after.
    const int a_row = slice * a_rows_per_slice + tile * kBM;
    const int npre = min(nchunks, kStages);
    for (int it = 0; it < npre; ++it) {
      mbar_expect_tx(bars + 8 * it, stage_sz);
      if (p.stream_weights) tma_load_2d_hint(base + it * stage_sz, &tmA, bars + 8 * it, (c0 + it) * kBK, a_row, l2_evict_first());
      else tma_load_2d(base + it * stage_sz, &tmA, bars + 8 * it, (c0 + it) * kBK, a_row);
    }
    pdl_wait();
    const bool skip = p.all_done && *p.all_done;
    for (int it = 0; it < npre; ++it) {
      const uint32_t sa = base + it * stage_sz;
      const int kx = slice * b_cols_per_slice + (c0 + it) * kBK;
      tma_load_2d(sa + kBM * 128, &tmBh, bars + 8 * it, kx, t0);
      tma_load_2d(sa + kBM * 128 + bn * 128, &tmBl, bars + 8 * it, kx, t0);
    }
    int issued = npre;
    for (int it = npre; it < nchunks && !skip; ++it) {
      const int s = it % kStages;
      const uint32_t ph = (it / kStages) & 1;
      if (!mbar_wait(bars + 8 * (kStages + s), ph ^ 1)) { ok = false; break; }
      issued = it + 1;
      const uint32_t full = bars + 8 * s;
      const uint32_t sa = base + s * stage_sz;
      mbar_expect_tx(full, stage_sz);
      const int kx = (c0 + it) * kBK;
      if (p.stream_weights) tma_load_2d_hint(sa, &tmA, full, kx, a_row, l2_evict_first());
      else tma_load_2d(sa, &tmA, full, kx, a_row);
      tma_load_2d(sa + kBM * 128, &tmBh, full, slice * b_cols_per_slice + kx, t0);
      tma_load_2d(sa + kBM * 128 + bn * 128, &tmBl, full, slice * b_cols_per_slice + kx, t0);
    }
    if (!ok) atomicCAS(p.error, 0, 101);
    if (!ok || skip) {
      // nobody will consume what is in flight: give it a bounded chance to land before shared memory goes away
      for (int it = max(0, issued - kStages); it < issued; ++it) mbar_wait(bars + 8 * (it % kStages), (it / kStages) & 1);
    }
  } else if (warp == 1 && lane == 0) {
    // ---------------- MMA issuer
    const uint32_t idesc = instr_desc_bf16(bn);
    pdl_wait();
    const bool skip = p.all_done && *p.all_done;
    uint32_t acc = tmem;
    for (int it = 0, in_group = 0; it < nchunks && !skip; ++it, ++in_group) {
      const int s = it % kStages;
      const uint32_t ph = (it / kStages) & 1;
      if (in_group == p.group_chunks) { in_group = 0; acc += 16; }
      if (!mbar_wait(bars + 8 * s, ph)) { ok = false; break; }
      tc_fence_after();
      const uint32_t sa = base + s * stage_sz;
#pragma unroll
      for (int kk = 0; kk < kBK / 16; ++kk) {
        const uint64_t ad = smem_desc_sw128(sa + kk * 32);
        const uint64_t bh = smem_desc_sw128(sa + kBM * 128 + kk * 32);
        const uint64_t bl = smem_desc_sw128(sa + kBM * 128 + bn * 128 + kk * 32);
        umma_f16(acc, ad, bh, idesc, (in_group > 0 || kk > 0) ? 1u : 0u);
        umma_f16(acc, ad, bl, idesc, 1u);
      }
      umma_commit(bars + 8 * (kStages + s));       // frees the stage once these MMAs have read it
    }
    if (!skip) umma_commit(bars + 8 * 2 * kStages);            // accumulator complete
    if (!ok) atomicCAS(p.error, 0, 102);
  } else if (warp >= 2) {
    // ---------------- epilogue: thread = one feature row, registers = tokens
    pdl_wait();
    const EpiShared sh{s_mean, s_rstd, s_slot, ctl};
    const EpiUnit u{tmem, bars + 8 * 2 * kStages, 0u, tile, split, slice, (int)blockIdx.z, (int)gridDim.x,
                    t0, nt, bn, nchunks, acc_groups, (nchunks + p.group_chunks - 1) / p.group_chunks, p.all_done && *p.all_done};
    tc_epilogue<EPI>(p, sh, u, warp, lane);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, ncols);
  }
}

}  // namespace tc
}  // namespace bpd
