// Instances of the register-streaming forward kernel: 3-D.
#include "bte_stream_kernel.cuh"

namespace bte {
namespace stream {
StreamKernel pick_3d(int lim, bool vec, int kr) { return pick_instance<3>(lim, vec, kr); }
}  // namespace stream
}  // namespace bte
