// Resident sweeps: sizes and launch (the kernel is in mpr_resident_kernel.cuh, one
// translation unit per model).
#include <algorithm>

#include "mpr_resident_kernel.cuh"

namespace mpr {
namespace resident {

Kernel pick(bool acc, bool energy, bool gmrf) {
    return gmrf ? pick_gmrf(acc, energy) : pick_mpr(acc, energy);
}

}  // namespace resident

size_t resident_smem(const TileDesc& t, int P, bool gmrf) {
    using namespace resident;
    const size_t n = (size_t)t.cnt[0] + t.cnt[1];
    const size_t cells = n + t.halo_cnt[0] + t.halo_cnt[1] + 2;
    return kFixed + 32 * n + sum_bytes(std::max(t.cnt[0], t.cnt[1])) +
           std::max(cells * P * (gmrf ? 8 : 16) + 2 * n, sizeof(double) * kNT);  // (a recorder: one each)
}

int resident_recorders(int group) { return (group + resident::kRecorderChains - 1) / resident::kRecorderChains; }

cudaError_t resident_blocks(size_t smem, bool gmrf, long long* blocks) {
    using namespace resident;
    *blocks = 0;
    int dev = 0, sms = 0, coop = 0, most = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e != cudaSuccess || !coop || smem > (size_t)most) return e;
    int least = 1 << 30;
    for (int v = 0; v < 4; ++v) {
        const void* f = reinterpret_cast<const void*>(pick(v & 1, v & 2, gmrf));
        int per = 0;
        e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
        if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, f, kNT, smem);
        if (e != cudaSuccess) return e;
        least = std::min(least, per);
    }
    *blocks = (long long)least * sms;
    return cudaSuccess;
}

cudaError_t launch_resident(const ResidentArgs& ra, int n_groups, size_t smem, cudaStream_t s) {
    using namespace resident;
    const Kernel f = pick((ra.a.flags & kAccumulate) != 0, (ra.a.flags & kEnergy) != 0,
                          (ra.a.flags & kGMRF) != 0);
    void* args[] = {const_cast<ResidentArgs*>(&ra)};
    const int x = ra.n_tiles + ((ra.a.flags & kEnergy) ? ra.a.n_img * ra.recorders : 0);
    return cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(f), dim3(x, n_groups), dim3(kNT), args,
                                       smem, s);
}

}  // namespace mpr
