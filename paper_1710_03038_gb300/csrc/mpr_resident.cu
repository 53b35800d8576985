// Resident sweeps: sizes and launch (the kernel is in mpr_resident_kernel.cuh, one
// translation unit per model).
#include <algorithm>

#include "mpr_resident_kernel.cuh"

namespace mpr {
namespace resident {

static_assert(kBlocksPerSM * 152 == kResidentBlocks, "room for as many blocks as fit");

Kernel pick(bool acc, bool energy, bool gmrf) {
    return gmrf ? pick_gmrf(acc, energy) : pick_mpr(acc, energy);
}

}  // namespace resident

int resident_recorders(int group) { return (group + resident::kRecorderChains - 1) / resident::kRecorderChains; }

cudaError_t resident_blocks(size_t smem, long long* blocks) {
    *blocks = 0;
    int dev = 0, sms = 0, coop = 0, most = 0, sm_bytes = 0, reserved = 0;
    cudaError_t e = cudaGetDevice(&dev);
    const auto get = [&](int* v, cudaDeviceAttr a) {
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(v, a, dev);
    };
    get(&sms, cudaDevAttrMultiProcessorCount);
    get(&coop, cudaDevAttrCooperativeLaunch);
    get(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin);
    get(&sm_bytes, cudaDevAttrMaxSharedMemoryPerMultiprocessor);
    get(&reserved, cudaDevAttrReservedSharedMemoryPerBlock);
    if (e != cudaSuccess || !coop || smem > (size_t)most) return e;
    // (shared memory is given out in units of 128 bytes)
    const size_t block = (smem + 127) / 128 * 128 + (size_t)reserved;
    *blocks = (long long)std::min((size_t)resident::kBlocksPerSM, (size_t)sm_bytes / block) * sms;
    return cudaSuccess;
}

cudaError_t resident_prepare(bool gmrf) {
    static OncePerDevice limit[2];
    int dev = 0;
    const cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    return limit[gmrf](dev, [&] {
        int most = 0;
        cudaError_t s = cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
        for (int v = 0; v < 4 && s == cudaSuccess; ++v)
            s = cudaFuncSetAttribute(reinterpret_cast<const void*>(resident::pick(v & 1, v & 2, gmrf)),
                                     cudaFuncAttributeMaxDynamicSharedMemorySize, most);
        return s;
    });
}

cudaError_t launch_resident(const ResidentArgs& ra, int n_groups, size_t smem, cudaStream_t s) {
    using namespace resident;
    const Kernel f = pick((ra.a.flags & kAccumulate) != 0, (ra.a.flags & kEnergy) != 0,
                          (ra.a.flags & kGMRF) != 0);
    void* args[] = {const_cast<ResidentArgs*>(&ra)};
    const int x = ra.n_tiles + ((ra.a.flags & kEnergy) ? ra.a.n_img * ra.recorders : 0);
    const cudaError_t e = cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(f), dim3(x, n_groups),
                                                      dim3(kNT), args, smem, s);
    if (e == cudaSuccess) ++launch_total();
    return e;
}

}  // namespace mpr
