// The attention kernel of many-row passes and the encoder, and its launch.
#include <algorithm>

#include "attention.cuh"
#include "host.hpp"

namespace bpd {
namespace attn {

template <typename CT>
int launch(const AttnParams& a, int max_keys, bool kv_static, cudaStream_t st, bool pdl) {
  constexpr bool f32 = sizeof(CT) == 4;
  Params p;
  p.a = a;
  p.kv_static = kv_static ? 1 : 0;
  // (at least 32 keys: the weights' planes need the room of 24 bf16 keys)
  p.chunk = std::min(std::max(32, (max_keys + 15) / 16 * 16), f32 ? kChunkF32 : kChunk);
  const int items = (a.rows / a.rows_per_b) * a.H, tiles = (a.rows_per_b + kRows - 1) / kRows;
  // with a CTA for every SM from sequences and heads alone, a CTA stages its keys once for all row tiles
  p.tiles_per_cta = items >= 148 ? tiles : 1;
  p.one_tile = p.tiles_per_cta == 1 ? 1 : 0;
  const size_t smem = smem_bytes(p.chunk, f32, p.one_tile != 0);
  int rc = ensure_smem_limit(reinterpret_cast<const void*>(attention_mma_kernel<CT>), smem);
  if (rc) return rc;
  BPD_CUDA(launch_k(attention_mma_kernel<CT>, dim3(items * ((tiles + p.tiles_per_cta - 1) / p.tiles_per_cta)), dim3(kThreads), smem, st, pdl, p));
  return BPD_OK;
}
template int launch<bf16>(const AttnParams&, int, bool, cudaStream_t, bool);
template int launch<float>(const AttnParams&, int, bool, cudaStream_t, bool);

}  // namespace attn
}  // namespace bpd
