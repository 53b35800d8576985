// Resident sweeps: the kernels of the GMRF bond.
#include "mpr_resident_kernel.cuh"

namespace mpr {
namespace resident {
Kernel pick_gmrf(bool acc, bool energy) { return pick_model<tiled::kModelGMRF>(acc, energy); }
}  // namespace resident
}  // namespace mpr
