// Resident sweeps: the kernels of the MPR bond.
#include "mpr_resident_kernel.cuh"

namespace mpr {
namespace resident {
Kernel pick_mpr(bool acc, bool energy) { return pick_model<tiled::kModelMPR>(acc, energy); }
}  // namespace resident
}  // namespace mpr
