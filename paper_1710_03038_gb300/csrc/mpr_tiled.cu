// Tiled path: the dispatch of the colour pass to its tile shape (the kernel is in mpr_tiled_kernel.cuh,
// one translation unit per tile shape).
#include "mpr_device.cuh"
#include "mpr_internal.h"
#include "mpr_tiled_kernel.cuh"

namespace mpr {

cudaError_t launch_tiled_32x16(const SweepArgs& a, cudaStream_t s, bool setup_only);
cudaError_t launch_tiled_16x16(const SweepArgs& a, cudaStream_t s, bool setup_only);
cudaError_t launch_tiled_32x32(const SweepArgs& a, cudaStream_t s, bool setup_only);
cudaError_t launch_tiled_16x16_lit(const SweepArgs& a, cudaStream_t s, bool setup_only);
cudaError_t launch_tiled_16x16_gmrf(const SweepArgs& a, cudaStream_t s, bool setup_only);

size_t tiled_pass_smem(int tx, int ty, int gt, int n_cap, int chain_group, int flags) {
    using namespace tiled;
    const int P = pairs_for_group(chain_group);
    if (flags & kGMRF) return Cfg<16, 16, 4, kModelGMRF>::smem_for(gt, n_cap, P);
    if (flags & kLiteralOR) return Cfg<16, 16, 4, kModelLIT>::smem_for(gt, n_cap, P);
    if (tx == 32 && ty == 16) return Cfg<32, 16, 8, kModelMPR>::smem_for(gt, n_cap, P);
    if (tx == 32 && ty == 32) return Cfg<32, 32, 8, kModelMPR>::smem_for(gt, n_cap, P);
    return Cfg<16, 16, 4, kModelMPR>::smem_for(gt, n_cap, P);
}

int tiled_pairs(int chain_group) { return tiled::pairs_for_group(chain_group); }

int tiled_blocks_per_sm(int tx, int ty) {
    using namespace tiled;
    if (tx == 32) return 1024 / Cfg<32, 16, 8, kModelMPR>::NT;
    return 1024 / Cfg<16, 16, 4, kModelMPR>::NT;
}

bool tiled_config_supported(int tx, int ty) {
    return (tx == 32 && ty == 16) || (tx == 16 && ty == 16) || (tx == 32 && ty == 32);
}

bool tiled_model_supported(int tx, int ty, int flags) {
    if (flags & (kGMRF | kLiteralOR)) return tx == 16 && ty == 16;
    return tiled_config_supported(tx, ty);
}

cudaError_t launch_tiled_pass(const SweepArgs& a, int tx, int ty, cudaStream_t s,
                              bool setup_only) {
    // chain groups start on a multiple of 4 chains (16-byte aligned rows)
    if (a.chain_group < 1 || a.chain_group > 32 || (a.chain0 & 3) || a.chain0 < 0 ||
        a.chain_end <= a.chain0 || a.chain_end > a.n_chains ||
        (a.chain_group % 4 != 0 && a.chain_group < a.chain_end - a.chain0))
        return cudaErrorInvalidValue;
    if (!tiled_model_supported(tx, ty, a.flags)) return cudaErrorInvalidValue;
    if (a.flags & kGMRF) return launch_tiled_16x16_gmrf(a, s, setup_only);
    if (a.flags & kLiteralOR) return launch_tiled_16x16_lit(a, s, setup_only);
    if (tx == 32 && ty == 16) return launch_tiled_32x16(a, s, setup_only);
    if (tx == 16 && ty == 16) return launch_tiled_16x16(a, s, setup_only);
    if (tx == 32 && ty == 32) return launch_tiled_32x32(a, s, setup_only);
    return cudaErrorInvalidValue;
}

}  // namespace mpr
