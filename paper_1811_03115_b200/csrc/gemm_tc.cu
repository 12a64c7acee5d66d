// The instantiations of the tensor-core projections.
#include <algorithm>

#include "host.hpp"
#include "tc_host.hpp"

namespace bpd {
namespace tc {

BPD_TC_LAUNCH(kTcPlanes);
BPD_TC_LAUNCH(kTcF32);
BPD_TC_LAUNCH(kTcResidual);
BPD_TC_LAUNCH(kTcQkv);
BPD_TC_LAUNCH(kTcHeadOut);
BPD_TC_LAUNCH(kTcArgmax);

}  // namespace tc
}  // namespace bpd

#ifdef BPD_TC_TRACE
// Development builds only: where the projection kernel writes its per-CTA step timestamps (4096 * 16 unsigned 64-bit
// words of device memory), or null to stop.
extern "C" int bpd_debug_set_tc_trace(void* dev_buffer) {
  unsigned long long* ptr = static_cast<unsigned long long*>(dev_buffer);
  BPD_CUDA(cudaMemcpyToSymbol(bpd::tc::g_tc_trace, &ptr, sizeof(ptr)));
  return BPD_OK;
}
#endif
