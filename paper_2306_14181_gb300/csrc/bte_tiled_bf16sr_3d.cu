// Instances of the tiled forward kernel: BF16 codes rounded stochastically, 3-D grids.
#include "bte_tiled_kernel.cuh"

namespace bte {
namespace tiled {
StepKernel pick_bf16sr_3d(int lim, Rows r) { return pick_instance<kStoreBF16, 3, true>(lim, r); }
}  // namespace tiled
}  // namespace bte
