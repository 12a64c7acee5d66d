// The instantiations of the persistent layer kernel (a translation unit of their own: they take a minute to compile).
#include "host.hpp"
#include "layer_stack.cuh"

namespace bpd {
namespace stack {

const void* kernel_for(int nt, int ksteps, int minb, int lean) {
#define BPD_V(NT, KS, MB, LN) \
  if (nt == NT && ksteps == KS && minb == MB && lean == LN) return reinterpret_cast<const void*>(layer_stack_kernel<NT, KS, MB, LN>)
  BPD_V(1, 2, 1, 0); BPD_V(2, 2, 1, 0); BPD_V(1, 4, 1, 0); BPD_V(2, 4, 1, 0);
  BPD_V(1, 2, 2, 0); BPD_V(2, 2, 2, 0); BPD_V(1, 4, 2, 0); BPD_V(2, 4, 2, 0);
  BPD_V(1, 2, 1, 1); BPD_V(2, 2, 1, 1); BPD_V(1, 4, 1, 1); BPD_V(2, 4, 1, 1);
  BPD_V(1, 2, 2, 1); BPD_V(2, 2, 2, 1); BPD_V(1, 4, 2, 1); BPD_V(2, 4, 2, 1);
  BPD_V(1, 2, 1, 2); BPD_V(2, 2, 1, 2); BPD_V(1, 4, 1, 2); BPD_V(2, 4, 1, 2);
  BPD_V(1, 2, 1, 3); BPD_V(2, 2, 1, 3); BPD_V(1, 4, 1, 3); BPD_V(2, 4, 1, 3);
  BPD_V(1, 2, 2, 4); BPD_V(2, 2, 2, 4); BPD_V(1, 4, 2, 4); BPD_V(2, 4, 2, 4);
#undef BPD_V
  return nullptr;
}

}  // namespace stack
}  // namespace bpd

#ifdef BPD_STACK_TRACE
// Development builds only: where the persistent layer kernel writes its per-CTA step timestamps (device memory,
// clusters * 8 * 256 unsigned 64-bit words), or null to stop.
extern "C" int bpd_debug_set_stack_trace(void* dev_buffer) {
  unsigned long long* ptr = static_cast<unsigned long long*>(dev_buffer);
  BPD_CUDA(cudaMemcpyToSymbol(bpd::stack::g_stack_trace, &ptr, sizeof(ptr)));
  return BPD_OK;
}
#endif
