// Context-free kernels: lattice energy and its gradient for dense angle
// grids (the forward and backward of the energy as a differentiable
// function), and direct access to the random stream's Philox blocks.
#include <curand_philox4x32_x.h>

#include <algorithm>
#include <vector>

#include "mpr_device.cuh"
#include "mpr_internal.h"

using namespace mpr;

namespace {

struct GridTable {
    int Lx, Ly;
    long long off;
};

// Shapes travel in the kernel parameters (no device allocation): up to
// kMaxGrids grids per launch, more are launched in chunks.
constexpr int kMaxGrids = 256;
struct Grids {
    GridTable g[kMaxGrids];
};

// One thread walks kRows rows of one column (blockIdx.x: columns and row chunks of a
// grid, blockIdx.y: the grid), so that no pixel index is divided, the pixel below is
// the next row's own pixel, and a bond's sine serves both of its ends (sin is odd, bit
// for bit): the bond above comes from the row before, the one on the left from the
// lane before.  Bond terms in FP32; their sums in two FP32 words (two_sum:
// about 48 bits), FP64 from the end of the column on: an FP64 addition per pixel alone would
// take as long as everything else (12 grids of 509 x 383: energy 102 us, gradient 115
// us before, with a 64-bit division and an FP64 addition per pixel).
constexpr int kRows = 16, kCols = 128;

struct Column {
    const float* p;
    int x, y0, y1, Lx, Ly;
    bool in;
};

__device__ __forceinline__ Column column_of(const GridTable& g, const float* phi) {
    const unsigned nx = ((unsigned)g.Lx + kCols - 1u) / kCols;
    Column c;
    c.x = (int)min((unsigned)(blockIdx.x % nx) * kCols + threadIdx.x, (unsigned)g.Lx);
    c.y0 = (int)min((long long)(blockIdx.x / nx) * kRows, (long long)g.Ly);  // (past its last chunk: nothing)
    c.y1 = (int)min((long long)c.y0 + kRows, (long long)g.Ly);
    c.Lx = g.Lx;
    c.Ly = g.Ly;
    c.in = c.x < g.Lx && c.y0 < g.Ly;
    c.p = phi + g.off + c.x;
    return c;
}

// Sum over the block, added to *out.
__device__ __forceinline__ void add_block(double v, double* out) {
    __shared__ double part[kCols / 32];
    v = warp_sum(v);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
#pragma unroll
        for (int k = 1; k < kCols / 32; ++k) v += part[k];
        if (v != 0.0) atomicAdd(out, v);
    }
}

// By site: a thread per pixel, FP64 sums.  The shorter way for small batches and for grids
// that leave a block's columns or rows idle (by_columns).
__global__ void lattice_energy_site_kernel(const __grid_constant__ Grids G, int k0,
                                           const float* __restrict__ phi, float q, float J, double* H) {
    const GridTable g = G.g[blockIdx.y];
    const long long n = (long long)g.Lx * g.Ly;
    const float* p = phi + g.off;
    double s = 0.0;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x) {
        const int x = (int)(i % g.Lx), y = (int)(i / g.Lx);
        const float v = p[i];
        float e = 0.0f;
        if (x + 1 < g.Lx) e -= J * cosf(q * (v - p[i + 1]));
        if (y + 1 < g.Ly) e -= J * cosf(q * (v - p[i + g.Lx]));
        s += (double)e;
    }
    s = warp_sum(s);
    if ((threadIdx.x & 31) == 0 && s != 0.0) atomicAdd(H + k0 + blockIdx.y, s);
}

template <bool GRAD, bool GJ>
__global__ void lattice_grad_site_kernel(const __grid_constant__ Grids G, int k0,
                                         const float* __restrict__ phi, float q, float J, const double* up,
                                         float* __restrict__ grad, double* gJ) {
    const GridTable g = G.g[blockIdx.y];
    const long long n = (long long)g.Lx * g.Ly;
    const float* p = phi + g.off;
    const double uk = up[k0 + blockIdx.y];
    const float w = (float)uk * J * q;
    double sJ = 0.0;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x) {
        const int x = (int)(i % g.Lx), y = (int)(i / g.Lx);
        const float v = p[i];
        if (GRAD) {
            float s = 0.0f;
            if (y > 0) s += sinf(q * (v - p[i - g.Lx]));
            if (y + 1 < g.Ly) s += sinf(q * (v - p[i + g.Lx]));
            if (x > 0) s += sinf(q * (v - p[i - 1]));
            if (x + 1 < g.Lx) s += sinf(q * (v - p[i + 1]));
            grad[g.off + i] = w * s;
        }
        if (GJ) {
            float e = 0.0f;
            if (x + 1 < g.Lx) e -= cosf(q * (v - p[i + 1]));
            if (y + 1 < g.Ly) e -= cosf(q * (v - p[i + g.Lx]));
            sJ += (double)e;
        }
    }
    if (GJ) {
        sJ = warp_sum(sJ) * uk;
        if ((threadIdx.x & 31) == 0 && sJ != 0.0) atomicAdd(gJ, sJ);
    }
}

// H_k = -J sum_<ij> cos(q (phi_i - phi_j)) over the right and down bonds of grid k.
__global__ void __launch_bounds__(kCols)
lattice_energy_kernel(const __grid_constant__ Grids G, int k0, const float* __restrict__ phi, float q,
                      float J, double scale, double* H) {
    const Column c = column_of(G.g[blockIdx.y], phi);
    float hi = 0.0f, lo = 0.0f;
    if (c.in) {
        float v = c.p[(long long)c.y0 * c.Lx];
#pragma unroll 4
        for (int y = c.y0; y < c.y1; ++y) {
            const float* row = c.p + (long long)y * c.Lx;
            float e = 0.0f, below = 0.0f;
            if (c.x + 1 < c.Lx) e -= J * cosf(q * (v - row[1]));
            if (y + 1 < c.Ly) {
                below = row[c.Lx];
                e -= J * cosf(q * (v - below));
            }
            two_sum(hi, lo, e);
            v = below;
        }
    }
    add_block(two_sum_value(hi, lo) * scale, H + k0 + blockIdx.y);
}

// Gradients of L = sum_k g_k H_k: GRAD the torque of every site, dL/dphi_i = g_k J q
// sum_j sin(q (phi_i - phi_j)) (the local field that the sweep uses); GJ dL/dJ =
// -sum_k g_k sum over the right and down bonds of cos(q dphi).
template <bool GRAD, bool GJ>
__global__ void __launch_bounds__(kCols)
lattice_grad_kernel(const __grid_constant__ Grids G, int k0, const float* __restrict__ phi, float q,
                    float J, const double* up, float* __restrict__ grad, double* gJ) {
    const GridTable g = G.g[blockIdx.y];
    const Column c = column_of(g, phi);
    const double uk = up[k0 + blockIdx.y];
    const float w = (float)uk * J * q;
    float hi = 0.0f, lo = 0.0f;
    const long long top = (long long)c.y0 * c.Lx;
    float v = c.in ? c.p[top] : 0.0f;
    // sine of the bond to the pixel above, as that pixel sees it
    float s_above = GRAD && c.in && c.y0 > 0 ? sinf(q * (c.p[top - c.Lx] - v)) : 0.0f;
    const int rows = min(kRows, c.Ly - c.y0);  // (the same for the whole block)
#pragma unroll 2
    for (int k = 0; k < rows; ++k) {
        const int y = c.y0 + k;
        const long long i = (long long)y * c.Lx;
        const bool has_right = c.in && c.x + 1 < c.Lx, has_below = c.in && y + 1 < c.Ly;
        const float d_right = has_right ? q * (v - c.p[i + 1]) : 0.0f;
        const float below = has_below ? c.p[i + c.Lx] : 0.0f;
        const float d_below = has_below ? q * (v - below) : 0.0f;
        if (GRAD) {
            const float s_right = sinf(d_right), s_below = sinf(d_below);
            float s_left = __shfl_up_sync(0xffffffffu, s_right, 1);
            if ((threadIdx.x & 31) == 0 && c.in && c.x > 0) s_left = sinf(q * (c.p[i - 1] - v));
            float s = 0.0f;
            if (y > 0) s -= s_above;
            if (has_below) s += s_below;
            if (c.x > 0) s -= s_left;
            if (has_right) s += s_right;
            if (c.in) grad[g.off + i + c.x] = w * s;
            s_above = s_below;
        }
        if (GJ) {
            float e = 0.0f;
            if (has_right) e -= cosf(d_right);
            if (has_below) e -= cosf(d_below);
            two_sum(hi, lo, e);
        }
        v = below;
    }
    if (GJ) add_block(two_sum_value(hi, lo) * uk, gJ);
}

__global__ void philox_kernel(int n, const uint32_t* ctr, uint2 key, uint32_t* out, int reference) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const uint4 c = make_uint4(ctr[4 * i], ctr[4 * i + 1], ctr[4 * i + 2], ctr[4 * i + 3]);
    const uint4 w = reference ? curand_Philox4x32_10(c, key) : philox4x32_10(c, key);
    out[4 * i] = w.x;
    out[4 * i + 1] = w.y;
    out[4 * i + 2] = w.z;
    out[4 * i + 3] = w.w;
}

__global__ void math_probe_kernel(int fn, int n, const float* a, const float* b, float* out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    float v = 0.0f;
    switch (fn) {
        case 0: v = atan2_pair(f2(a[i]), f2(b[i])).x; break;
        case 1: v = atan2f(a[i], b[i]); break;
        case 2: v = sin_taylor2(f2(a[i])).x; break;
        default: v = sinf(a[i]); break;
    }
    out[i] = v;
}

// A launch's grids: blocks to a grid by columns and by site, pixels of all of them.
struct Chunk {
    int blocks, site_blocks;
    double sites, fill;  // fill: share of the columns' threads and rows that have a pixel
};

// By columns or by site.  us, columns / site (energy, both gradients): 12 x 128^2 11.5 / 14.4,
// 14.9 / 17.0; 40 x 64^2 11.8 / 10.4, 14.9 / 15.0; 1 x 256^2 13.2 / 9.7, 16.8 / 10.6; 12 x 509 x
// 383 14.9 / 105, 24.7 / 117.  Thin grids leave most of a block idle: 10^6 x 2 162 / 25, 543 / 31;
// 10^5 x 32 28.9 / 28.9, 65 / 46; 30000 x 64 15.0 / 24.6, 30.4 / 30.3.  The torque alone sums
// nothing and is the shorter by site up to larger batches: 4 x 512^2 12.9 / 11.9, 12 x 509 x 383
// 17.0 / 20.9, 1 x 2048^2 27 / 36.
bool by_columns(const Chunk& c, bool sums) { return c.fill >= 0.45 && c.sites >= (sums ? 1.8e5 : 2e6); }

template <typename F>
mpr_status for_chunks(int n, const int* Lx, const int* Ly, F launch) {
    if (n < 1 || !Lx || !Ly) return MPR_ERR_INVALID_ARG;
    long long off = 0;
    for (int k0 = 0; k0 < n; k0 += kMaxGrids) {
        Grids G;
        const int m = std::min(kMaxGrids, n - k0);
        long long blocks = 1, most = 1;
        const long long first = off;
        for (int j = 0; j < m; ++j) {
            const int i = k0 + j;
            if (Lx[i] < 1 || Ly[i] < 1) return MPR_ERR_INVALID_ARG;
            G.g[j] = GridTable{Lx[i], Ly[i], off};
            off += (long long)Lx[i] * Ly[i];
            most = std::max(most, (long long)Lx[i] * Ly[i]);
            blocks = std::max(blocks, ((kCols - 1LL + Lx[i]) / kCols) * ((kRows - 1LL + Ly[i]) / kRows));
        }
        Chunk c;
        c.sites = (double)(off - first);
        c.fill = blocks > 0x7FFFFFFFLL ? 0.0 : c.sites / ((double)blocks * m * kCols * kRows);
        c.blocks = (int)std::min(blocks, 0x7FFFFFFFLL);
        c.site_blocks = (int)std::min((most + 255) / 256, 1024LL);
        if (launch(G, k0, m, c) != cudaSuccess) return MPR_ERR_CUDA;
    }
    return MPR_OK;
}

template <bool GRAD, bool GJ>
mpr_status gradients(int n, const int* Lx, const int* Ly, const float* phi, double q, double J, const double* g,
                     float* grad, double* gJ, cudaStream_t s) {
    return for_chunks(n, Lx, Ly, [&](const Grids& G, int k0, int m, const Chunk& c) {
        if (by_columns(c, GJ))
            lattice_grad_kernel<GRAD, GJ><<<dim3(c.blocks, m), kCols, 0, s>>>(G, k0, phi, (float)q, (float)J, g,
                                                                             grad, gJ);
        else
            lattice_grad_site_kernel<GRAD, GJ><<<dim3(c.site_blocks, m), 256, 0, s>>>(G, k0, phi, (float)q,
                                                                                     (float)J, g, grad, gJ);
        return launched();
    });
}

}  // namespace

extern "C" {

mpr_status mpr_lattice_energy(int n, const int* Lx, const int* Ly, const float* phi, double q,
                              double J, double* H_out, mpr_stream stream) {
    if (!phi || !H_out) return MPR_ERR_INVALID_ARG;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    if (cudaMemsetAsync(H_out, 0, sizeof(double) * (n > 0 ? n : 0), s) != cudaSuccess)
        return MPR_ERR_CUDA;
    const ScaledJ j(J);
    return for_chunks(n, Lx, Ly, [&](const Grids& G, int k0, int m, const Chunk& c) {
        if (by_columns(c, true))
            lattice_energy_kernel<<<dim3(c.blocks, m), kCols, 0, s>>>(G, k0, phi, (float)q, j.m, j.scale, H_out);
        else
            lattice_energy_site_kernel<<<dim3(c.site_blocks, m), 256, 0, s>>>(G, k0, phi, (float)q, (float)J,
                                                                              H_out);
        return launched();
    });
}

mpr_status mpr_lattice_torque(int n, const int* Lx, const int* Ly, const float* phi, double q,
                              double J, const double* g, float* grad, mpr_stream stream) {
    if (!phi || !g || !grad) return MPR_ERR_INVALID_ARG;
    return gradients<true, false>(n, Lx, Ly, phi, q, J, g, grad, nullptr, reinterpret_cast<cudaStream_t>(stream));
}

mpr_status mpr_lattice_grad(int n, const int* Lx, const int* Ly, const float* phi, double q,
                            double J, const double* g, float* grad_phi, double* grad_J,
                            mpr_stream stream) {
    if (!phi || !g || (!grad_phi && !grad_J)) return MPR_ERR_INVALID_ARG;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    if (grad_J && cudaMemsetAsync(grad_J, 0, sizeof(double), s) != cudaSuccess) return MPR_ERR_CUDA;
    if (!grad_J) return gradients<true, false>(n, Lx, Ly, phi, q, J, g, grad_phi, nullptr, s);
    if (!grad_phi) return gradients<false, true>(n, Lx, Ly, phi, q, J, g, nullptr, grad_J, s);
    return gradients<true, true>(n, Lx, Ly, phi, q, J, g, grad_phi, grad_J, s);
}

mpr_status mpr_philox(int n, const uint32_t* ctr, const uint32_t* key, uint32_t* out, int reference,
                      mpr_stream stream) {
    if (n < 0 || !ctr || !key || !out) return MPR_ERR_INVALID_ARG;
    if (n == 0) return MPR_OK;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    philox_kernel<<<(n + 255) / 256, 256, 0, s>>>(n, ctr, make_uint2(key[0], key[1]), out, reference);
    return launched() == cudaSuccess ? MPR_OK : MPR_ERR_CUDA;
}

mpr_status mpr_math_probe(int fn, int n, const float* a, const float* b, float* out,
                          mpr_stream stream) {
    if (fn < 0 || fn > 3 || n < 0 || !a || !out || (fn < 2 && !b)) return MPR_ERR_INVALID_ARG;
    if (n == 0) return MPR_OK;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    math_probe_kernel<<<(n + 255) / 256, 256, 0, s>>>(fn, n, a, b, out);
    return launched() == cudaSuccess ? MPR_OK : MPR_ERR_CUDA;
}

}  // extern "C"
