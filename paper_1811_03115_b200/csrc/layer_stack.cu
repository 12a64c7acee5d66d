// The persistent layer kernel for d_model 1024, and the choice among all its instantiations (one translation unit per
// d_model: they take two minutes to compile).
#include "host.hpp"
#include "layer_stack.cuh"

namespace bpd {
namespace stack {

BPD_STACK_KERNELS_HALF_SM(1024)
template <> const void* kernel_of<512>(int nt, int hct, int minb, int lean);
template <> const void* kernel_of<256>(int nt, int hct, int minb, int lean);

const void* kernel_for(int nt, int d, int hct, int minb, int lean) {
  return d == 1024 ? kernel_of<1024>(nt, hct, minb, lean) : d == 512 ? kernel_of<512>(nt, hct, minb, lean) : d == 256 ? kernel_of<256>(nt, hct, minb, lean) : nullptr;
}

}  // namespace stack
}  // namespace bpd
