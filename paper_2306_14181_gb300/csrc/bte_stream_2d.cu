// Instances of the register-streaming forward kernel: 2-D.
#include "bte_stream_kernel.cuh"

namespace bte {
namespace stream {
StreamKernel pick_2d(int lim, bool vec, int kr) { return pick_instance<2>(lim, vec, kr); }
}  // namespace stream
}  // namespace bte
