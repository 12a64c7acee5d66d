// Attention of up to 16 query rows of one (sequence, head) per step of a CTA, on mma.sync: the encoder, and the decoder
// passes of sessions whose layers run as one kernel per projection.  Head width 64.
//
// The kernels this replaces spent their time on latency: one warp per query row (or a CTA per row), 760 cycles for a
// 64-element score and 800 for a weighted sum of 32 values, 12-28 us per launch at batch 32.  Here the scores of 16
// rows are one product with the keys and the outputs one with the values, and everything that does not depend on the
// preceding launch -- the cached keys and values below the sequence's length, the encoder's rows in cross-attention --
// is in shared memory before the dependency wait.
//
// Precision is that of fp32: queries, softmax weights and fp32 keys / values are taken apart into three bf16 planes
// (24 bits of mantissa: x = h + m + l) and multiplied plane by plane into fp32 accumulators -- three products where the
// other operand is a bf16 cache entry (exact), the six largest of nine where both are fp32 (the rest is below 2^-24).
//
// Keys are taken in chunks that start at multiples of the chunk length from the first visible key's chunk on, weights
// and outputs are rescaled to the running maximum chunk by chunk.  A row's result depends on key positions alone, not on
// the other rows of the launch.
#pragma once
#include "kernels_simt.cuh"

namespace bpd {
namespace attn {

constexpr int kRows = 16;            // query rows per step (MMA M)
constexpr int kThreads = 256;
constexpr int kPitch = 72;           // bf16 elements between rows of 64 queries: 16-byte rows of 8 lanes hit all banks once
constexpr int kPitchK = 72, kPitchV = 68;   // floats between fp32 keys / values: pairs along a key and single values across
                                            // eight keys are read without bank conflicts
constexpr int kChunk = 256;          // keys per chunk at most: bf16 cache
constexpr int kChunkF32 = 96;        // fp32 keys and values

struct Params {
  AttnParams a;
  int kv_static;       // 1: keys and values do not come from the preceding launch (self-attention: those below len do not)
  int chunk;           // keys per chunk, a multiple of 16
  int tiles_per_cta;   // row tiles a CTA takes in turn
  int one_tile;        // 1: only one
};

// Keys and values; bf16 rows of 128 bytes with their 16-byte pieces swizzled by the row, fp32 rows padded.
__host__ __device__ inline size_t kv_bytes(int chunk, bool f32) { return f32 ? (size_t)chunk * (kPitchK + kPitchV) * 4 : (size_t)chunk * 256; }
__host__ __device__ inline size_t weight_bytes(int chunk) { return (size_t)3 * kRows * (chunk + 8) * 2; }
// The weights take the place of the keys where a CTA has one row tile (the keys have been used by then).
inline size_t smem_bytes(int chunk, bool f32, bool one_tile) {
  return kv_bytes(chunk, f32) + (size_t)3 * kRows * kPitch * 2 + (one_tile ? 0 : weight_bytes(chunk)) + (size_t)kRows * (chunk + 4) * 4;
}

__device__ __forceinline__ uint32_t s_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void ldsm4(uint32_t addr, uint32_t (&r)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void ldsm2_trans(uint32_t addr, uint32_t& r0, uint32_t& r1) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0, %1}, [%2];" : "=r"(r0), "=r"(r1) : "r"(addr) : "memory");
}
__device__ __forceinline__ void mma_bf16(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t pack2(bf16 a, bf16 b) {
  return (uint32_t)__bfloat16_as_ushort(a) | ((uint32_t)__bfloat16_as_ushort(b) << 16);
}
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}

// Byte offset of 16-byte piece `piece` of a bf16 row.
__device__ __forceinline__ uint32_t swz(int row, int piece) { return row * 128 + ((piece ^ (row & 7)) << 4); }
// Two floats taken apart into three pairs of bf16.
__device__ __forceinline__ void split3_pair(float x, float y, uint32_t (&out)[3]) {
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(x, y);
    out[q] = *reinterpret_cast<const uint32_t*>(&h);
    x -= __uint_as_float(out[q] << 16);
    y -= __uint_as_float(out[q] & 0xffff0000u);
  }
}

// Accumulator of the product of planes (q, kq): the largest products have one of their own, the others are spread over
// three, so that no chain of dependent MMAs is longer than two per 16 columns.
__host__ __device__ constexpr int product_slot(int q, int kq, bool f32) {
  return q + kq == 0 ? 0 : (!f32 ? q : (q == 0 ? (kq == 1 ? 1 : 3) : (q == 1 ? 2 : 1)));
}
__device__ __forceinline__ float sum4(const float (&c)[4][4], int i) { return c[0][i] + (c[1][i] + (c[2][i] + c[3][i])); }

// Rows [from, to) (positions c0 + row) of a chunk of keys and values on their way into shared memory.
template <typename CT>
__device__ __forceinline__ void stage_rows(const Params& p, uint32_t ks, uint32_t vs, int b, int h, int c0, int from, int to, const int* pt) {
  const AttnParams& a = p.a;
  constexpr int PIECES = sizeof(CT) == 2 ? 8 : 16, PER = 16 / sizeof(CT);
  const CT* K = reinterpret_cast<const CT*>(a.k);
  const CT* V = reinterpret_cast<const CT*>(a.v);
  for (int i = from * PIECES + threadIdx.x; i < to * PIECES; i += kThreads) {
    const int row = i / PIECES, piece = i % PIECES, pos = c0 + row;
    const size_t at = (a.paged ? ((size_t)pt[pos / kPage] * kPage + (pos % kPage)) * a.ldkv : (size_t)b * a.bstride + (size_t)pos * a.ldkv) + h * 64 + piece * PER;
    cp_async16(ks + (sizeof(CT) == 2 ? swz(row, piece) : (row * kPitchK + piece * 4) * 4), K + at);
    cp_async16(vs + (sizeof(CT) == 2 ? swz(row, piece) : (row * kPitchV + piece * 4) * 4), V + at);
  }
}

// grid = (sequences x heads x groups of row tiles).  CT: element type of keys and values.
template <typename CT>
__global__ void __launch_bounds__(kThreads, 3) attention_mma_kernel(const __grid_constant__ Params p) {
  pdl_launch_dependents();
  constexpr bool F32 = sizeof(CT) == 4;
  extern __shared__ __align__(128) uint8_t asm_raw[];
  __shared__ float s_m[kRows], s_l[kRows], s_corr[kRows];
  const AttnParams& a = p.a;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t4 = lane & 3;
  const int chunk = p.chunk, p_pitch = chunk + 8, s_pitch = chunk + 4;
  uint8_t* kb = asm_raw;
  uint8_t* vb = kb + (F32 ? (size_t)chunk * kPitchK * 4 : (size_t)chunk * 128);
  bf16* qs = reinterpret_cast<bf16*>(kb + kv_bytes(chunk, F32));     // [3][16][kPitch]
  float* sc = reinterpret_cast<float*>(qs + 3 * kRows * kPitch);     // [16][s_pitch]
  // [3][16][p_pitch], in the keys' place where they are not needed again
  bf16* ps = p.one_tile ? reinterpret_cast<bf16*>(kb) : reinterpret_cast<bf16*>(sc + kRows * s_pitch);
  const uint32_t ks = s_addr(kb), vs = s_addr(vb);
  const int rpb = a.rows_per_b, tiles = (rpb + kRows - 1) / kRows, groups = (tiles + p.tiles_per_cta - 1) / p.tiles_per_cta;
  const int item = blockIdx.x / groups, tile0 = (blockIdx.x % groups) * p.tiles_per_cta;
  const int b = item / a.H, h = item % a.H;
  const int* pt = a.paged ? a.st.page_table + b * a.st.pages_per_row : nullptr;
  // neither the lengths nor the page table change during a pass
  const int len = a.causal ? a.st.len[b] : 0;
  const int seen = a.causal ? 0 : a.limit_b[b];             // keys every row sees (not causal)
  const int fixed = p.kv_static ? (a.causal ? len : seen) : 0;   // positions below it do not depend on the preceding launch
  bool waited = false;
  int staged_c0 = -1, staged_to = 0;                        // what the key / value buffers hold: chunk, rows

  for (int tile = tile0; tile < min(tiles, tile0 + p.tiles_per_cta); ++tile) {
    const int r0 = tile * kRows, n = min(kRows, rpb - r0);
    const int limit = a.causal ? len + r0 + n : seen;       // of the tile's last row
    const int c_first = attn_first_key(a, len + r0) / chunk * chunk;
    float acc[4][4] = {};
    if (tid < kRows) { s_m[tid] = -INFINITY; s_l[tid] = 0.f; }
    for (int c0 = c_first; c0 < limit; c0 += chunk) {
      const int nk = min(chunk, limit - c0), nk16 = (nk + 15) & ~15;
      const bool reuse = waited && staged_c0 == c0 && staged_to >= nk;
      const int early = waited ? 0 : max(0, min(nk, fixed - c0));
      if (early > 0) stage_rows<CT>(p, ks, vs, b, h, c0, 0, early, pt);
      if (!waited) {
        pdl_wait();
        waited = true;
        if (a.all_done && *a.all_done) {
          asm volatile("cp.async.wait_all;" ::: "memory");
          return;
        }
      }
      if (!reuse) {
        stage_rows<CT>(p, ks, vs, b, h, c0, early, nk, pt);
        // weight 0 times what lies beyond the last key must be 0
        for (int i = nk * 16 + tid; i < nk16 * 16; i += kThreads) {
          if (F32) *reinterpret_cast<float4*>(vb + ((i >> 4) * kPitchV + (i & 15) * 4) * 4) = make_float4(0.f, 0.f, 0.f, 0.f);
          else if ((i & 15) < 8) *reinterpret_cast<uint4*>(vb + (i >> 4) * 128 + (i & 7) * 16) = make_uint4(0u, 0u, 0u, 0u);
        }
        staged_c0 = c0; staged_to = nk;
      }
      if (c0 == c_first) {
        // the tile's queries: 16 threads per row, four elements each
        const int row = tid >> 4, col = (tid & 15) * 4;
        float4 q4 = make_float4(0.f, 0.f, 0.f, 0.f);
        if (row < n) q4 = *reinterpret_cast<const float4*>(reinterpret_cast<const float*>(a.q) + (long long)(b * rpb + r0 + row) * a.ldq + h * 64 + col);
        uint32_t lo2[3], hi2[3];
        split3_pair(q4.x * a.scale, q4.y * a.scale, lo2);
        split3_pair(q4.z * a.scale, q4.w * a.scale, hi2);
#pragma unroll
        for (int q = 0; q < 3; ++q) *reinterpret_cast<uint2*>(qs + (q * kRows + row) * kPitch + col) = make_uint2(lo2[q], hi2[q]);
      }
      asm volatile("cp.async.wait_all;" ::: "memory");
      __syncthreads();
      // scores: a warp takes every eighth group of 8 keys
      for (int n0 = warp * 8; n0 < nk16; n0 += 64) {
        float c[4][4] = {};                                 // see product_slot
#pragma unroll
        for (int k2 = 0; k2 < 2; ++k2) {
          uint32_t bk[4];
          if (!F32) ldsm4(ks + swz(n0 + (lane & 7), k2 * 4 + (lane >> 3)), bk);
#pragma unroll
          for (int kk = 0; kk < 2; ++kk) {
            const int k = k2 * 2 + kk;
            uint32_t b0[3], b1[3];
            if (F32) {
              const float* kr = reinterpret_cast<const float*>(kb) + (n0 + g) * kPitchK + k * 16 + t4 * 2;
              const float2 x = *reinterpret_cast<const float2*>(kr), y = *reinterpret_cast<const float2*>(kr + 8);
              split3_pair(x.x, x.y, b0);
              split3_pair(y.x, y.y, b1);
            } else {
              b0[0] = bk[kk * 2]; b1[0] = bk[kk * 2 + 1];
            }
#pragma unroll
            for (int q = 0; q < 3; ++q) {
              uint32_t aq[4];
              ldsm4(s_addr(qs + (q * kRows + (lane & 15)) * kPitch + k * 16 + (lane >> 4) * 8), aq);
#pragma unroll
              for (int kq = 0; kq < (F32 ? 3 - q : 1); ++kq)
                mma_bf16(c[product_slot(q, kq, F32)], aq, b0[kq], b1[kq]);
            }
          }
        }
        *reinterpret_cast<float2*>(sc + g * s_pitch + n0 + t4 * 2) = make_float2(sum4(c, 0), sum4(c, 1));
        *reinterpret_cast<float2*>(sc + (g + 8) * s_pitch + n0 + t4 * 2) = make_float2(sum4(c, 2), sum4(c, 3));
      }
      __syncthreads();
      // weights: 16 threads per row
      {
        const int row = tid >> 4, t = tid & 15;
        const int row_limit = row < n ? (a.causal ? len + r0 + row + 1 : seen) : 0, row_first = a.causal ? attn_first_key(a, len + r0 + row) : 0;
        const int lo = row_first - c0, hi = row_limit - c0;
        const float m_old = s_m[row];
        float m_new = m_old;
        for (int j = t * 2; j < nk16; j += 32) {
          const float2 v = *reinterpret_cast<const float2*>(sc + row * s_pitch + j);
          if (j >= lo && j < hi) m_new = fmaxf(m_new, v.x);
          if (j + 1 >= lo && j + 1 < hi) m_new = fmaxf(m_new, v.y);
        }
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) m_new = fmaxf(m_new, __shfl_xor_sync(0xffffffffu, m_new, o));
        float sum = 0.f;
        for (int j = t * 2; j < nk16; j += 32) {
          const float2 v = *reinterpret_cast<const float2*>(sc + row * s_pitch + j);
          const float e0 = (j >= lo && j < hi) ? expf(v.x - m_new) : 0.f, e1 = (j + 1 >= lo && j + 1 < hi) ? expf(v.y - m_new) : 0.f;
          sum += e0 + e1;
          uint32_t w[3];
          split3_pair(e0, e1, w);
#pragma unroll
          for (int q = 0; q < 3; ++q) *reinterpret_cast<uint32_t*>(ps + (q * kRows + row) * p_pitch + j) = w[q];
        }
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
        if (t == 0) {
          const float corr = m_new == -INFINITY ? 1.f : expf(m_old - m_new);      // nothing visible yet: nothing to rescale
          s_m[row] = m_new;
          s_l[row] = s_l[row] * corr + sum;
          s_corr[row] = corr;
        }
      }
      __syncthreads();
      // outputs: warp w owns dims 8w .. 8w + 7
      {
        const float f0 = s_corr[g], f1 = s_corr[g + 8];
#pragma unroll
        for (int i = 0; i < 4; ++i) { acc[i][0] *= f0; acc[i][1] *= f0; acc[i][2] *= f1; acc[i][3] *= f1; }
        for (int k0 = 0; k0 < nk16; k0 += 16) {
          uint32_t b0[3], b1[3];
          if (F32) {
            const float* vr = reinterpret_cast<const float*>(vb) + (k0 + t4 * 2) * kPitchV + warp * 8 + g;
            split3_pair(vr[0], vr[kPitchV], b0);
            split3_pair(vr[8 * kPitchV], vr[9 * kPitchV], b1);
          } else {
            ldsm2_trans(vs + swz(k0 + (lane & 15), warp), b0[0], b1[0]);
          }
#pragma unroll
          for (int q = 0; q < 3; ++q) {
            uint32_t ap[4];
            ldsm4(s_addr(ps + (q * kRows + (lane & 15)) * p_pitch + k0 + (lane >> 4) * 8), ap);
#pragma unroll
            for (int kq = 0; kq < (F32 ? 3 - q : 1); ++kq) mma_bf16(acc[product_slot(q, kq, F32)], ap, b0[kq], b1[kq]);
          }
        }
      }
      __syncthreads();                                      // keys, values, weights and corrections have been used
    }
#pragma unroll
    for (int half = 0; half < 2; ++half) {
      const int row = g + 8 * half;
      if (row >= n) continue;
      const float inv = 1.f / s_l[row];
      const float o0 = sum4(acc, 2 * half) * inv, o1 = sum4(acc, 2 * half + 1) * inv;
      const long long at = (long long)(b * rpb + r0 + row) * a.ldo + h * 64 + warp * 8 + t4 * 2;
      if (a.out_plane) {
        const bf16 h0 = __float2bfloat16_rn(o0), h1 = __float2bfloat16_rn(o1);
        bf16* out = reinterpret_cast<bf16*>(a.out) + at;
        *reinterpret_cast<uint32_t*>(out) = pack2(h0, h1);
        *reinterpret_cast<uint32_t*>(out + a.out_plane) =
            pack2(__float2bfloat16_rn(o0 - __bfloat162float(h0)), __float2bfloat16_rn(o1 - __bfloat162float(h1)));
      } else {
        *reinterpret_cast<float2*>(reinterpret_cast<float*>(a.out) + at) = make_float2(o0, o1);
      }
    }
    __syncthreads();                                        // the sums have been read
  }
}

// Whether a launch takes this kernel; `block`: the most query rows per sequence of any launch of the session (the choice
// must not depend on the pass).  With a CTA on half the SMs (74 items) it is the faster one at any length.  Launches of fewer
// CTAs stay with the kernels that give rows CTAs of their own where a CTA would have less than half of its 16 rows to work
// on, or would walk more than 512 keys alone.  us per pass with the row kernels / with this one in every launch:
//   items (sequences x heads)   48        48        48        64        64        72        80        80        96
//   rows of a sequence           4         6         8         5         7         4         4         8         2
//   up to 140 keys             487/500   357/352   405/375   372/353   417/378   374/332   367/351   490/401   350/312
//   48 items of 8 rows over 450 / 600 / 1200 / 2400 keys: 431/393, 444/402, 492/459, 568/560 (this one for the encoder's
//   rows and the row kernels for the cache: 542); 72 of 8 over 600: 575/407; 80 of 4 over 1200: 685/423
// By this table the line belongs at 64 items and, for 6 rows and more, at 48: of these only 48 items of 4 rows lose with this
// kernel.  It has not been moved there yet.
inline bool applies(const AttnParams& a, int max_keys, int block) {
  const int items = (a.rows / a.rows_per_b) * a.H * ((block + kRows - 1) / kRows);
  return a.dh == 64 && (items >= 74 || (block >= kRows / 2 && max_keys <= 512));
}
// max_keys: the most keys a row of the session can see.
template <typename CT>
int launch(const AttnParams& a, int max_keys, bool kv_static, cudaStream_t st, bool pdl);

}  // namespace attn
}  // namespace bpd
