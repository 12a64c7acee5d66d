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
