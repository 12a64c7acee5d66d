// A whole decoder pass of a small fp32 model -- embedding, layers, heads, vocabulary top-1, verification -- as one
// launch of one cluster of 8 CTAs (sessions of at most 16 rows per pass whose weights are at most 4 MB).
//
// Such a pass is a chain of some twenty tiny steps (2 layers of width 64: 0.3 MB of weights each) and its time is what
// lies between them: 22 launches of 3.4 us.  Inside a cluster a step costs a hardware barrier (0.4 us) and a round of
// remote shared-memory stores instead: every CTA owns an eighth of the features of every projection, computes them for
// all rows and writes its results into the shared memory of all eight, so that each step finds its whole input at home.
// What a step needs from memory is requested before the barrier that precedes it (a round trip to L2 is longer than most
// steps): the next weights, committed keys and values, encoder rows; layer norms and biases are fetched once, at the start.
//
// The order of a sum depends on the matrix alone: lane s of the KS lanes that share a feature takes columns 4 (s + KS i) ..,
// the lanes are added by a butterfly.
#pragma once
#include "kernels_simt.cuh"

namespace bpd {
namespace tiny {

constexpr int kCtas = 8;
constexpr int kThreads = 256;
constexpr int kMaxRows = 16;
constexpr int kMaxLayers = 8;
constexpr size_t kMaxWeights = 4 << 20;
constexpr int kAhead = 8;                  // 16-byte weight loads per thread requested ahead of a step

struct Layer {
  const float *ln1g, *ln1b, *wqkv, *wo, *ln2g, *ln2b, *cwq, *cwo, *ln3g, *ln3b, *w1, *b1, *w2, *b2;
  float *kcache, *vcache;
  const float* crosskv;
};
struct Params {
  Layer layers[kMaxLayers];
  int L, d, H, ff, V, km, fh, blockdiag, p1_identity, R, rpb, kh, max_src, local_q, local_m;
  float eps, scale;
  const float *embed, *pe; int npos;
  const float *lnfg, *lnfb, *hw1, *hb1, *hw2, *hb2, *out_proj;
  const int* forced; int forced_rows, kforced;
  float* h_f32;                            // decoder outputs for the caller's dump
  VerifyParams verify;
};

// Layer norms and biases of a layer in shared memory.
__host__ __device__ inline int layer_vectors(int d, int ff) { return 7 * d + ff; }
// Floats of dynamic shared memory: two copies of the stream, its normalised form, Q | K | V, attention output, hidden
// units, head hidden units, head outputs, a step's results on their way out, top-1 keys, layer norms and biases.
__host__ __device__ inline size_t smem_floats(int R, int kh, int d, int ff, int hid, int L) {
  const int widest = hid > ff ? hid : ff, n = widest > 3 * d ? widest : 3 * d, out = n > kh * d ? n : kh * d;
  return (size_t)R * (2 * d + d + 3 * d + d + ff + hid) + (size_t)R * kh * d + (size_t)R * ((out + kCtas - 1) / kCtas + 4) + 2 * kCtas * R * kh +
         2 * 8 * 16 + (size_t)L * layer_vectors(d, ff) + 2 * d + hid + kh * d + 16;
}

__device__ __forceinline__ void arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ uint32_t remote(const void* p, int rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
  return r;
}

// How a matrix [N, K] is worked on: this CTA's features, lanes per feature.
struct Split { int n0, n1, ks; };
__device__ __forceinline__ Split split_of(int N, int K, int rank) {
  const int per = (N + kCtas - 1) / kCtas;
  Split s;
  s.n0 = min(N, rank * per); s.n1 = min(N, s.n0 + per);
  s.ks = 1;
  while (s.ks < 32 && per * s.ks * 2 <= kThreads && s.ks * 8 <= K) s.ks *= 2;
  return s;
}
// This CTA's results of a step ([rows][n1 - n0], ld_in apart, in its own shared memory) into every CTA's copy (columns n0 ..
// of rows ld_out apart).
__device__ __forceinline__ void share(const Split& s, int R, const float* in, int ld_in, float* out, int ld_out) {
  const int n = s.n1 - s.n0;
  __syncthreads();
  if ((n & 3) == 0 && (s.n0 & 3) == 0) {
    const int n4 = n >> 2;
    for (int i = threadIdx.x; i < R * n4 * kCtas; i += kThreads) {
      const int c = i % kCtas, e = i / kCtas, r = e / n4, q = (e - r * n4) * 4;
      const float4 v = *reinterpret_cast<const float4*>(in + r * ld_in + q);
      asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(remote(out + r * ld_out + s.n0 + q, c)), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
    }
  } else {
    for (int i = threadIdx.x; i < R * n * kCtas; i += kThreads) {
      const int c = i % kCtas, e = i / kCtas, r = e / n, q = e - r * n;
      asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(remote(out + r * ld_out + s.n0 + q, c)), "f"(in[r * ld_in + q]) : "memory");
    }
  }
}
struct Ahead { float4 w[kAhead]; };
// The first weights of this thread's first feature.  row(n): address of feature n's weights.
template <typename ROW>
__device__ __forceinline__ Ahead fetch(const Split& s, int K, ROW&& row) {
  Ahead a;
  const int f = threadIdx.x / s.ks, lane = threadIdx.x % s.ks, n = s.n0 + f;
#pragma unroll
  for (int i = 0; i < kAhead; ++i) {
    const int k = 4 * (lane + s.ks * i);
    a.w[i] = (n < s.n1 && k < K) ? __ldg(reinterpret_cast<const float4*>(row(n) + k)) : make_float4(0.f, 0.f, 0.f, 0.f);
  }
  return a;
}
// sum_k w[n][k] x[r][k] for this CTA's features and rows r < R; x(n, r): the row's input (shared memory).  out(n, r, v) is
// called by one of the lanes that hold the sum.  RM: rows held at a time.
template <int RM, typename ROW, typename X, typename OUT>
__device__ __forceinline__ void project(const Split& s, int K, int R, const Ahead& a, ROW&& row, X&& x, OUT&& out) {
  const int lane = threadIdx.x % s.ks, step = kThreads / s.ks, f = threadIdx.x / s.ks;
  for (int n0 = s.n0; n0 < s.n1; n0 += step) {               // uniform over the CTA
    const int n = n0 + f;
    const bool live = n < s.n1;
    const int nn = live ? n : s.n0;
    const float* w = row(nn);
    for (int rb = 0; rb < R; rb += RM) {
      float acc[RM];
#pragma unroll
      for (int r = 0; r < RM; ++r) acc[r] = 0.f;
      auto step4 = [&](const float4& w4, int k) {
#pragma unroll
        for (int r = 0; r < RM; ++r) {
          if (rb + r < R) {
            const float4 v = *reinterpret_cast<const float4*>(x(nn, rb + r) + k);
            acc[r] = fmaf(w4.x, v.x, acc[r]); acc[r] = fmaf(w4.y, v.y, acc[r]); acc[r] = fmaf(w4.z, v.z, acc[r]); acc[r] = fmaf(w4.w, v.w, acc[r]);
          }
        }
      };
#pragma unroll
      for (int i = 0; i < kAhead; ++i) {
        const int k = 4 * (lane + s.ks * i);
        if (k < K) step4(n0 == s.n0 ? a.w[i] : __ldg(reinterpret_cast<const float4*>(w + k)), k);
      }
      int k = 4 * (lane + s.ks * kAhead);
      for (; k + 4 * s.ks * 7 < K; k += 4 * s.ks * 8) {      // eight loads in flight
        float4 w4[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) w4[i] = __ldg(reinterpret_cast<const float4*>(w + k + 4 * s.ks * i));
#pragma unroll
        for (int i = 0; i < 8; ++i) step4(w4[i], k + 4 * s.ks * i);
      }
      for (; k < K; k += 4 * s.ks) step4(__ldg(reinterpret_cast<const float4*>(w + k)), k);
      for (int o = s.ks >> 1; o > 0; o >>= 1) {
#pragma unroll
        for (int r = 0; r < RM; ++r) acc[r] += __shfl_xor_sync(0xffffffffu, acc[r], o);
      }
#pragma unroll
      for (int r = 0; r < RM; ++r)
        if (live && rb + r < R && (r % s.ks) == lane) out(n, rb + r, acc[r]);
    }
  }
}

// Layer norm of the stream's rows (a warp per row), every CTA for itself.
__device__ __forceinline__ void normalise(const Params& p, const float* x, float* y, const float* g, const float* b) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, d = p.d;
  for (int r = warp; r < p.R; r += kThreads / 32) {
    float s = 0.f, q = 0.f;
    for (int c = lane; c < d; c += 32) s += x[r * d + c];
    const float mean = warp_sum(s) / (float)d;
    for (int c = lane; c < d; c += 32) { const float t = x[r * d + c] - mean; q = fmaf(t, t, q); }
    const float rstd = rsqrtf(warp_sum(q) / (float)d + p.eps);
    for (int c = lane; c < d; c += 32) y[r * d + c] = (x[r * d + c] - mean) * rstd * g[c] + b[c];
  }
  __syncthreads();
}

// Attention of one (row, head) by a warp: lane = key in chunks of 32 positions, running maximum and sum chunk by chunk.
// key(pos) / value(pos): addresses of the head's DH floats of a position; q: the query (shared memory).  What does not
// depend on this pass (positions below `fixed`) of the first chunk is requested ahead of the barrier before the step.
template <int DH> struct AttnAhead { float4 k[DH / 4]; float v[DH]; };
template <int DH, typename K, typename V>
__device__ __forceinline__ AttnAhead<DH> attn_fetch(int first, int fixed, K&& key, V&& value) {
  constexpr int PARTS = 32 / DH;                            // lanes that share an output element
  const int lane = threadIdx.x & 31, dim = lane % DH, part = lane / DH, c0 = first & ~31;
  AttnAhead<DH> a;
#pragma unroll
  for (int i = 0; i < DH / 4; ++i) a.k[i] = c0 + lane < fixed ? reinterpret_cast<const float4*>(key(c0 + lane))[i] : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
  for (int i = 0; i < DH; ++i) a.v[i] = c0 + part + PARTS * i < fixed ? value(c0 + part + PARTS * i)[dim] : 0.f;
  return a;
}
template <int DH, typename K, typename V>
__device__ __forceinline__ float attend(const Params& p, const float* q, int first, int limit, int fixed, const AttnAhead<DH>& ahead, K&& key, V&& value) {
  constexpr int PARTS = 32 / DH;
  const int lane = threadIdx.x & 31, dim = lane % DH, part = lane / DH;
  float m = -INFINITY, l = 0.f, acc = 0.f;
  for (int c0 = first & ~31; c0 < limit; c0 += 32) {
    const int pos = c0 + lane, n = min(32, limit - c0);
    const bool live = pos >= first && pos < limit, have = c0 == (first & ~31);
    float s = -INFINITY, v[DH];
    if (live) {
      float4 k4[DH / 4];
      if (have && pos < fixed) {
#pragma unroll
        for (int i = 0; i < DH / 4; ++i) k4[i] = ahead.k[i];
      } else {
        const float4* kr = reinterpret_cast<const float4*>(key(pos));
#pragma unroll
        for (int i = 0; i < DH / 4; ++i) k4[i] = kr[i];
      }
      float dot[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int i = 0; i < DH / 4; ++i) {
        const float4 q4 = reinterpret_cast<const float4*>(q)[i];
        dot[0] = fmaf(q4.x, k4[i].x, dot[0]); dot[1] = fmaf(q4.y, k4[i].y, dot[1]); dot[2] = fmaf(q4.z, k4[i].z, dot[2]); dot[3] = fmaf(q4.w, k4[i].w, dot[3]);
      }
      s = ((dot[0] + dot[1]) + (dot[2] + dot[3])) * p.scale;
    }
#pragma unroll
    for (int i = 0; i < DH; ++i) {
      const int j = part + PARTS * i;
      v[i] = (have && c0 + j < fixed) ? ahead.v[i] : (j < n ? value(c0 + j)[dim] : 0.f);
    }
    const float m_new = fmaxf(m, warp_max(s)), corr = expf(m - m_new), w = live ? expf(s - m_new) : 0.f;
    l = l * corr + warp_sum(w);
    acc *= corr;
    float part_sum[2] = {0.f, 0.f};
#pragma unroll
    for (int i = 0; i < DH; ++i) part_sum[i & 1] = fmaf(__shfl_sync(0xffffffffu, w, part + PARTS * i), v[i], part_sum[i & 1]);
    acc += part_sum[0] + part_sum[1];
    m = m_new;
  }
#pragma unroll
  for (int o = DH; o < 32; o <<= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  return acc / l;
}
