// The persistent layer kernel for d_model 256.
#include "host.hpp"
#include "layer_stack.cuh"

namespace bpd {
namespace stack {

BPD_STACK_KERNELS(256, BPD_STACK_V(256, 256, 2, 2, 4))

}  // namespace stack
}  // namespace bpd
