// Sample specific energy without any allocation, for callers that cannot
// call cudaMalloc (or any allocator): the per-block partial results live in
// a fixed array in this library's device memory instead of a workspace.
//
// The array is file scope and shared by every call on a device; it holds the
// last call's partials.  Nothing in it has to start at zero (every partial is
// written before it is read), but two calls that overlap on the GPU (in
// different streams, or in a graph) would overwrite each other's partials.
#include <cmath>
#include <cstring>
#include <mutex>
#include <string>

#include "mpr_device.cuh"
#include "mpr_internal.h"

using namespace mpr;

namespace {

constexpr int kNoAllocMaxImages = 64;   // images per call
constexpr int kNoAllocBlocks = 256;     // partials per image and phase
constexpr double kPiD = 3.14159265358979323846;

struct Partial {        // one thread block's share of one image
    uint32_t zlo, zhi;  // order-preserving encodings of the sample extremes
    unsigned long long n_gap;
    double sum;         // -J sum cos(q dphi) over sample-sample bonds
    unsigned long long n_pair;
};

struct ImgStat {
    float zmin, zmax;
    unsigned long long n_gap;
};

// The scratch: two phases of partials plus per-image extremes.
constexpr size_t kScratchBytes =
    sizeof(Partial) * kNoAllocMaxImages * kNoAllocBlocks + sizeof(ImgStat) * kNoAllocMaxImages;
static __device__ __align__(256) unsigned char g_noalloc_scratch[kScratchBytes];

struct Shapes {
    int n;
    int Lx[kNoAllocMaxImages], Ly[kNoAllocMaxImages];
    long long off[kNoAllocMaxImages];
};

__device__ __forceinline__ uint32_t ordered_f(float f) {
    const uint32_t b = __float_as_uint(f);
    return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}
__device__ __forceinline__ float unordered_f(uint32_t u) {
    return __uint_as_float((u & 0x80000000u) ? (u & 0x7FFFFFFFu) : ~u);
}

template <typename T, typename F>
__device__ T block_reduce(T v, F op, T* sh, T identity) {
    for (int o = 16; o > 0; o >>= 1) v = op(v, __shfl_xor_sync(0xffffffffu, v, o));
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    if (l == 0) sh[w] = v;
    __syncthreads();
    if (w == 0) {
        v = l < (int)(blockDim.x >> 5) ? sh[l] : identity;
        for (int o = 16; o > 0; o >>= 1) v = op(v, __shfl_xor_sync(0xffffffffu, v, o));
    }
    __syncthreads();
    return v;  // valid in thread 0
}

// Phase 1: per-block sample extremes and gap counts.
__global__ void noalloc_extremes_kernel(const __grid_constant__ Shapes S, const float* z,
                                        const uint8_t* gap, Partial* part) {
    __shared__ unsigned long long sh[32];
    const int im = blockIdx.y;
    const long long n = (long long)S.Lx[im] * S.Ly[im];
    const float* zi = z + S.off[im];
    const uint8_t* gi = gap + S.off[im];
    uint32_t lo = 0xFFFFFFFFu, hi = 0u;
    unsigned long long cnt = 0;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x) {
        if (gi[i]) { ++cnt; continue; }
        const uint32_t o = ordered_f(zi[i]);
        lo = min(lo, o);
        hi = max(hi, o);
    }
    auto mn = [](unsigned long long a, unsigned long long b) { return a < b ? a : b; };
    auto mx = [](unsigned long long a, unsigned long long b) { return a > b ? a : b; };
    auto ad = [](unsigned long long a, unsigned long long b) { return a + b; };
    const unsigned long long rlo = block_reduce<unsigned long long>(lo, mn, sh, 0xFFFFFFFFull);
    const unsigned long long rhi = block_reduce<unsigned long long>(hi, mx, sh, 0ull);
    const unsigned long long rc = block_reduce<unsigned long long>(cnt, ad, sh, 0ull);
    if (threadIdx.x == 0) {
        Partial& p = part[im * kNoAllocBlocks + blockIdx.x];
        p.zlo = (uint32_t)rlo;
        p.zhi = (uint32_t)rhi;
        p.n_gap = rc;
    }
}

// Phase 2: sample-sample bond sums with the angles of Eq. map computed on the fly
// exactly as the context's initialisation computes them (FP64 map, rounded to FP32
// once; FP32 bond terms -J cos(q (v - w)), their sum in two FP32 words per thread and
// FP64 from there).  A warp takes 31 columns and kRows rows: each lane maps its pixels
// once, the pixel below is the next row's own, the one on the right the next lane's (the
// last lane only maps).  Mapping both neighbours again for every pixel took 48 us for two
// images of 433^2 and 694^2, most of it FP64.  Every block first combines the image's
// extremes (all blocks get the same bits).
constexpr int kRows = 8, kPairThreads = 256;

__global__ void __launch_bounds__(kPairThreads)
noalloc_pairs_kernel(const __grid_constant__ Shapes S, const float* __restrict__ z,
                     const uint8_t* __restrict__ gap, ImgStat* stat, float q, float J, double scale_J,
                     Partial* part) {
    __shared__ unsigned long long shu[32];
    __shared__ double shd[32];
    __shared__ ImgStat st;
    const int im = blockIdx.y;
    uint32_t plo = 0xFFFFFFFFu, phi = 0u;
    unsigned long long pgap = 0;
    for (int b = threadIdx.x; b < kNoAllocBlocks; b += kPairThreads) {
        const Partial& p = part[im * kNoAllocBlocks + b];
        plo = min(plo, p.zlo);
        phi = max(phi, p.zhi);
        pgap += p.n_gap;
    }
    auto mn = [](unsigned long long a, unsigned long long b) { return a < b ? a : b; };
    auto mx = [](unsigned long long a, unsigned long long b) { return a > b ? a : b; };
    auto add_u = [](unsigned long long a, unsigned long long b) { return a + b; };
    auto add_d = [](double a, double b) { return a + b; };
    const unsigned long long rlo = block_reduce<unsigned long long>(plo, mn, shu, 0xFFFFFFFFull);
    const unsigned long long rhi = block_reduce<unsigned long long>(phi, mx, shu, 0ull);
    const unsigned long long rg = block_reduce<unsigned long long>(pgap, add_u, shu, 0ull);
    if (threadIdx.x == 0) {
        st.zmin = rlo == 0xFFFFFFFFull ? __int_as_float(0x7FC00000) : unordered_f((uint32_t)rlo);
        st.zmax = rlo == 0xFFFFFFFFull ? __int_as_float(0x7FC00000) : unordered_f((uint32_t)rhi);
        st.n_gap = rg;
        if (blockIdx.x == 0) stat[im] = st;
    }
    __syncthreads();
    const int Lx = S.Lx[im], Ly = S.Ly[im];
    const double zmin = st.zmin;
    const double scale = 2.0 * kPiD / ((double)st.zmax - zmin);
    const int lane = threadIdx.x & 31, warps = kPairThreads / 32;
    const int nx = (Lx + 30) / 31, tasks = nx * ((Ly + kRows - 1) / kRows);
    double s = 0.0;
    unsigned long long cnt = 0;
    for (int task = blockIdx.x * warps + (threadIdx.x >> 5); st.zmax > st.zmin && task < tasks;
         task += gridDim.x * warps) {
        const int x = task % nx * 31 + lane, y0 = task / nx * kRows;
        const bool in = x < Lx, own = in && lane < 31;
        const long long o = S.off[im] + (long long)y0 * Lx + x;
        const int rows = min(kRows, Ly - y0);
        float hi = 0.0f, lo = 0.0f;
        bool ok = in && !gap[o];
        float v = ok ? (float)(((double)z[o] - zmin) * scale) : 0.0f;
#pragma unroll 4
        for (int k = 0; k < rows; ++k) {
            const long long i = o + (long long)k * Lx;
            const bool ok_below = in && y0 + k + 1 < Ly && !gap[i + Lx];
            const float below = ok_below ? (float)(((double)z[i + Lx] - zmin) * scale) : 0.0f;
            const float right = __shfl_down_sync(0xffffffffu, v, 1);
            const bool ok_right = __shfl_down_sync(0xffffffffu, (int)ok, 1);
            if (own && ok && ok_right) {
                two_sum(hi, lo, -(J * cosf(q * (v - right))));
                ++cnt;
            }
            if (own && ok && ok_below) {
                two_sum(hi, lo, -(J * cosf(q * (v - below))));
                ++cnt;
            }
            v = below;
            ok = ok_below;
        }
        s += two_sum_value(hi, lo);
    }
    const double rs = block_reduce<double>(s, add_d, shd, 0.0);
    const unsigned long long rc = block_reduce<unsigned long long>(cnt, add_u, shu, 0ull);
    if (threadIdx.x == 0) {
        Partial& p = part[im * kNoAllocBlocks + blockIdx.x];
        p.sum = rs * scale_J;
        p.n_pair = rc;
    }
}

// Phase 3: per image, combine the partials in a fixed order (one thread per partial: a
// loop of one thread over them took 22 us).
__global__ void __launch_bounds__(kNoAllocBlocks)
noalloc_final_kernel(const Partial* part, const ImgStat* stat, double* e_s, long long* n_sp, float* zmin,
                     float* zmax) {
    __shared__ unsigned long long shu[32];
    __shared__ double shd[32];
    const int im = blockIdx.x;
    const Partial& p = part[im * kNoAllocBlocks + threadIdx.x];
    auto add_u = [](unsigned long long a, unsigned long long b) { return a + b; };
    auto add_d = [](double a, double b) { return a + b; };
    const double s = block_reduce<double>(p.sum, add_d, shd, 0.0);
    const unsigned long long c = block_reduce<unsigned long long>(p.n_pair, add_u, shu, 0ull);
    if (threadIdx.x != 0) return;
    const bool ok = stat[im].zmax > stat[im].zmin;
    e_s[im] = (ok && c > 0) ? s / (double)c : __longlong_as_double(0x7FF8000000000000LL);
    if (n_sp) n_sp[im] = ok ? (long long)c : 0;
    if (zmin) zmin[im] = stat[im].zmin;
    if (zmax) zmax[im] = stat[im].zmax;
}

// Per-device address of the scratch array, looked up once per device.
std::mutex g_mu;
void* g_scratch_ptr[64] = {nullptr};

}  // namespace

extern "C" mpr_status mpr_sample_energy_noalloc(int n_img, const int* Lx, const int* Ly,
                                                const float* z, const uint8_t* gap, double q,
                                                double J, double* e_s, int64_t* n_sp,
                                                float* z_min, float* z_max, mpr_stream stream) {
    static_assert(kNoAllocMaxImages == MPR_NOALLOC_MAX_IMAGES, "header and scratch disagree");
    if (n_img < 1 || n_img > kNoAllocMaxImages)
        return set_last_error(MPR_ERR_INVALID_ARG,
                              "mpr_sample_energy_noalloc: n_img = " + std::to_string(n_img) +
                                  " is outside [1, " + std::to_string(kNoAllocMaxImages) +
                                  "], the capacity of its fixed scratch array");
    if (!Lx || !Ly || !z || !gap || !e_s)
        return set_last_error(MPR_ERR_INVALID_ARG, "mpr_sample_energy_noalloc: NULL argument");
    if (!(q > 0.0) || !(J > 0.0))
        return set_last_error(MPR_ERR_INVALID_ARG, "mpr_sample_energy_noalloc: q and J must be positive");
    Shapes S;
    std::memset(&S, 0, sizeof(S));
    S.n = n_img;
    long long off = 0;
    for (int i = 0; i < n_img; ++i) {
        if (Lx[i] < 2 || Ly[i] < 2 || Lx[i] > 65535 || Ly[i] > 65535)
            return set_last_error(MPR_ERR_INVALID_ARG,
                                  "mpr_sample_energy_noalloc: image sides must lie in [2, 65535]");
        S.Lx[i] = Lx[i];
        S.Ly[i] = Ly[i];
        S.off[i] = off;
        off += (long long)Lx[i] * Ly[i];
    }
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64)
        return set_last_error(MPR_ERR_CUDA, "mpr_sample_energy_noalloc: no current device");
    void* base = nullptr;
    {
        std::lock_guard<std::mutex> lk(g_mu);
        if (!g_scratch_ptr[dev]) {
            void* p = nullptr;
            const cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
            if (e != cudaSuccess || !p)
                return set_last_error(MPR_ERR_CUDA, std::string("mpr_sample_energy_noalloc: "
                                                                "cudaGetSymbolAddress: ") +
                                                        cudaGetErrorString(e));
            g_scratch_ptr[dev] = p;
        }
        base = g_scratch_ptr[dev];
    }
    Partial* part = static_cast<Partial*>(base);
    ImgStat* stat = reinterpret_cast<ImgStat*>(part + kNoAllocMaxImages * kNoAllocBlocks);
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    dim3 grid(kNoAllocBlocks, n_img);
    const ScaledJ j(J);
    noalloc_extremes_kernel<<<grid, 256, 0, s>>>(S, z, gap, part);
    noalloc_pairs_kernel<<<grid, kPairThreads, 0, s>>>(S, z, gap, stat, (float)q, j.m, j.scale, part);
    noalloc_final_kernel<<<n_img, kNoAllocBlocks, 0, s>>>(part, stat, e_s, reinterpret_cast<long long*>(n_sp),
                                              z_min, z_max);
    const cudaError_t e = launched(3);
    if (e != cudaSuccess)
        return set_last_error(MPR_ERR_CUDA, std::string("mpr_sample_energy_noalloc: ") +
                                                cudaGetErrorString(e));
    return MPR_OK;
}
