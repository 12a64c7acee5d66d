// The instantiations of the cluster layer kernels.
#include "fused_layer.cuh"
#include "host.hpp"

namespace bpd {
namespace fused {

// lean: self-attention 1 = short schedule only, 2 = long schedule only; cross-attention 1 = encoder rows staged, 0 = not
const void* attn_kernel(bool self, int nt, int lean, int minb) {
#define BPD_V(SELF, NT, LN, MB) \
  if (self == SELF && nt == NT && lean == LN && minb == MB) return reinterpret_cast<const void*>(attn_block_kernel<SELF, NT, LN, MB>)
  if (self && lean == 1) minb = 2;
  BPD_V(true, 1, 1, 2); BPD_V(true, 2, 1, 2);
  BPD_V(true, 1, 2, 1); BPD_V(true, 2, 2, 1); BPD_V(true, 1, 2, 2); BPD_V(true, 2, 2, 2);
  BPD_V(false, 1, 1, 2); BPD_V(false, 2, 1, 2); BPD_V(false, 1, 0, 2); BPD_V(false, 2, 0, 2);
#undef BPD_V
  return nullptr;
}
const void* ffn_kernel(int nt, int minb) {
#define BPD_V(NT, MB) if (nt == NT && minb == MB) return reinterpret_cast<const void*>(ffn_block_kernel<NT, MB>)
  BPD_V(1, 2); BPD_V(2, 2); BPD_V(1, 3); BPD_V(2, 3);
#undef BPD_V
  return nullptr;
}

}  // namespace fused
}  // namespace bpd
