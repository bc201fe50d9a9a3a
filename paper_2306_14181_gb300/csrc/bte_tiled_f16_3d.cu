// Instances of the tiled forward kernel: F16 codes rounded to nearest, 3-D grids.
#include "bte_tiled_kernel.cuh"

namespace bte {
namespace tiled {
StepKernel pick_f16_3d(int lim, Rows r, bool sr) {
    return sr ? pick_f16sr_3d(lim, r) : pick_instance<kStoreF16, 3, false>(lim, r);
}
}  // namespace tiled
}  // namespace bte
