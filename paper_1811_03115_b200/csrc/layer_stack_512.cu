// The persistent layer kernel for d_model 512.
#include "host.hpp"
#include "layer_stack.cuh"

namespace bpd {
namespace stack {

BPD_STACK_KERNELS(512, )

}  // namespace stack
}  // namespace bpd
