// Dense views of the tiled path: prediction, states in and out, energies of the
// chains.  The state is slot-major with the chains interleaved, so a thread per pixel
// and chain reads 4 bytes of a 128-byte row at a time; these kernels take one tile
// per block instead, move whole rows, and turn them in shared memory.
#include <algorithm>

#include "mpr_device.cuh"
#include "mpr_internal.h"

namespace mpr {

namespace {

// Conditional mean and standard deviation over realisations (Alg. 2 step 6), a block
// per tile: the samples by pixel, the gaps by slot, so that every lane of the FP64
// work is busy.  Bound by the FP64 units (2 lanes per clock and SM): one thread per
// pixel with FP64 divisions and square root took 1562 us at 4096^2 with 40 % gaps;
// the divisions are multiplications by 1 / n and 1 / 2 pi here, and the root is one
// FP64 Newton step from the FP32 estimate (relative error below 1e-13).
__global__ void __launch_bounds__(128)
predict_tile_kernel(const ImgDev* img, const TileDesc* tiles, int tx_log, int npix,
                    const uint32_t* __restrict__ slot_pos, const double* __restrict__ acc1,
                    const double* __restrict__ acc2, const float* __restrict__ zin,
                    const uint8_t* __restrict__ gap, double inv_n, const Control* ctl,
                    float* __restrict__ zhat, float* __restrict__ zstd) {
    const TileDesc T = tiles[blockIdx.x];
    const ImgDev& I = img[T.img];
    const int Lx = I.Lx, Ly = I.Ly;
    const long long site0 = I.site_off + (long long)T.y0 * Lx + T.x0;
    for (int i = threadIdx.x; i < npix; i += 128) {
        const int x = i & ((1 << tx_log) - 1), y = i >> tx_log;
        if (T.x0 + x >= Lx || T.y0 + y >= Ly) continue;
        const long long s = site0 + (long long)y * Lx + x;
        if (gap[s]) continue;
        zhat[s] = zin[s];
        if (zstd) zstd[s] = 0.0f;
    }
    constexpr double kInvTwoPiD = 0.15915494309189533577;
    const bool cut_short = ctl->status != 0;
    if (cut_short) inv_n = __longlong_as_double(0x7FF8000000000000LL);
    const double per_rad = ((double)I.zmax - (double)I.zmin) * kInvTwoPiD;  // field units per rad
    const double scale = per_rad * inv_n, zmin = I.zmin;
    for (int j = threadIdx.x; j < T.cnt[0] + T.cnt[1]; j += 128) {
        const long long k = T.slot_off + (j < T.cnt[0] ? T.off[0] + j : T.off[1] + j - T.cnt[0]);
        const uint32_t p = slot_pos[k];
        const long long s = I.site_off + (long long)(p >> 16) * Lx + (p & 0xFFFFu);
        const double a = acc1[k];
        zhat[s] = (float)fma(a, scale, zmin);
        if (zstd) {
            const double m = a * inv_n;
            const double v = fma(-m, m, acc2[k] * inv_n);
            const float vf = (float)v;
            float sd = cut_short ? __int_as_float(0x7FC00000) : 0.0f;
            if (vf > 1e30f || (vf <= 1e-30f && v > 0.0)) {  // (beyond the estimate's range)
                sd = (float)(sqrt(v) * per_rad);
            } else if (vf > 1e-30f) {
                const double r = (double)rsqrtf(vf), y = v * r;
                sd = (float)(fma(fma(-y, y, v), 0.5 * r, y) * per_rad);
            }
            zstd[s] = sd;
        }
    }
}

// States of 32 chains of a tile <-> dense planes (SET: the gap sites only), through
// shared memory: rows of 32 chains on one side, rows of the tile on the other.  Bound by
// the plane rows (64 bytes each); shared memory is sized by the batch's fullest tile, so
// that eight blocks share an SM.
template <bool SET>
__global__ void __launch_bounds__(256)
state_tile_kernel(const ImgDev* img, const TileDesc* tiles, int tx_log, int npix,
                  int n_max, const uint32_t* __restrict__ slot_pos, const float* __restrict__ samp,
                  float* __restrict__ state, int n_chains, const Control* ctl, float* __restrict__ dense) {
    extern __shared__ float rows[];  // [sites of the tile, at most n_max][33], then the tile's map
    uint16_t* map = reinterpret_cast<uint16_t*>(rows + n_max * 33);  // pixel -> site, 0xFFFF: a sample
    const TileDesc T = tiles[blockIdx.x];
    const ImgDev& I = img[T.img];
    const int Lx = I.Lx, Ly = I.Ly, n = T.cnt[0] + T.cnt[1];
    const int r0 = blockIdx.y * 32, nr = min(32, n_chains - r0);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int i = threadIdx.x; i < npix; i += 256) map[i] = 0xFFFFu;
    __syncthreads();
    const auto slot_of = [&](int j) { return j < T.cnt[0] ? T.off[0] + j : T.off[1] + j - T.cnt[0]; };
    for (int j = threadIdx.x; j < n; j += 256) {
        const uint32_t p = slot_pos[T.slot_off + slot_of(j)];
        map[(((int)(p >> 16) - T.y0) << tx_log) + (int)(p & 0xFFFFu) - T.x0] = (uint16_t)j;
    }
    float* st = state + T.state_off + r0 + lane;
    if (!SET && lane < nr) {
        const bool cut_short = ctl->status != 0;
#pragma unroll 8
        for (int j = warp; j < n; j += 8)
            rows[j * 33 + lane] = cut_short ? __int_as_float(0x7FC00000) : st[(long long)slot_of(j) * T.cp];
    }
    __syncthreads();
    const long long plane = (long long)Lx * Ly;
    float* d0 = dense + I.site_off * n_chains + r0 * plane;
    // out, four pixels of a row at a time, where every plane's rows start on 16 bytes and the
    // tile is whole in x (2048^2 x 32: 256 -> 160 us)
    const bool quads = !SET && T.x0 + (1 << tx_log) <= Lx && Lx % 4 == 0 && I.site_off % 4 == 0 &&
                       (reinterpret_cast<uintptr_t>(dense) & 15) == 0;
    for (int i = 4 * (threadIdx.x & 63); quads && i < npix; i += 256) {
        const int x = T.x0 + (i & ((1 << tx_log) - 1)), y = T.y0 + (i >> tx_log);
        if (y >= Ly) continue;
        const long long site = (long long)y * Lx + x;
        const ushort4 m = *reinterpret_cast<const ushort4*>(map + i);
        const float4 sample = *reinterpret_cast<const float4*>(samp + I.site_off + site);
        const auto row = [&](unsigned j) { return rows + (j == 0xFFFFu ? 0u : j * 33u); };
        const float *a = row(m.x), *b = row(m.y), *c = row(m.z), *d = row(m.w);
#pragma unroll 4
        for (int r = threadIdx.x >> 6; r < nr; r += 4) {
            float4 v = sample;
            if (m.x != 0xFFFFu) v.x = a[r];
            if (m.y != 0xFFFFu) v.y = b[r];
            if (m.z != 0xFFFFu) v.z = c[r];
            if (m.w != 0xFFFFu) v.w = d[r];
            *reinterpret_cast<float4*>(d0 + r * plane + site) = v;
        }
    }
    for (int i = threadIdx.x; !quads && i < npix; i += 256) {
        const int x = T.x0 + (i & ((1 << tx_log) - 1)), y = T.y0 + (i >> tx_log);
        if (x >= Lx || y >= Ly) continue;
        const long long site = (long long)y * Lx + x;
        const int m = map[i];
        float* d = d0 + site;
        if (SET) {
            if (m == 0xFFFF) continue;
            float* row = rows + m * 33;
#pragma unroll 8
            for (int r = 0; r < nr; ++r, d += plane) row[r] = *d;
        } else if (m == 0xFFFF) {
            const float v = samp[I.site_off + site];
            for (int r = 0; r < nr; ++r, d += plane) *d = v;
        } else {
            const float* row = rows + m * 33;
#pragma unroll 8
            for (int r = 0; r < nr; ++r, d += plane) *d = row[r];
        }
    }
    if (SET) {
        __syncthreads();
        if (lane < nr)
            for (int j = warp; j < n; j += 8) st[(long long)slot_of(j) * T.cp] = rows[j * 33 + lane];
    }
}

// H of the chains r_base to r_end of an image (blockIdx.z), C to a block (blockIdx.y): a lane
// is a pixel and a chain, C chains (a power of two) beside one another and 32 / C pixels,
// so that batches of few chains leave few lanes idle.  A block walks strips of STRIP rows
// of a tile.  The strip's angles and those right of and below it lie in shared memory, a
// row of C chains per pixel.  FP32 bond terms; their sum in two FP32 words (two_sum), FP64
// from the strip on: an FP64 addition per pixel and chain ran at 1/32 of the rate.  Bound
// by the two cosines per pixel and chain; small batches by the chain of a warp's pixels.
// 1000 x 777, us a call with 2, 4, 10, 16 and 24 chains: a thread per pixel and chain 35, 46,
// 85, 126, 176; a lane per chain whatever their number 107, 107, 115, 115, 116; this 32, 39,
// 75, 75, 112.
template <int STRIP, int NW, int C>
__global__ void __launch_bounds__(NW * 32)
energy_tile_kernel(const ImgDev* img, const TileDesc* tiles, int tx_log, int ty, const float* state,
                   const float* samp, const int* slot_map, int n_chains, int r_base, int r_end, float q,
                   float J, double scale, int gmrf, double* out) {
    extern __shared__ float ang[];  // [(STRIP + 1) x (tx + 1)][C]
    __shared__ double part[NW][C];
    constexpr int kPixels = 32 / C;  // pixels of a warp side by side
    const ImgDev& I = img[blockIdx.z];
    const int Lx = I.Lx, Ly = I.Ly, tx = 1 << tx_log, ew = tx + 1, strips = ty / STRIP;
    const int r0 = r_base + blockIdx.y * C, nr = min(C, r_end - r0);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int ch = lane & (C - 1), px = lane / C;
    const int r = min(ch, nr - 1);  // lanes without a chain repeat the last one
    double sum = 0.0;
    for (int t = blockIdx.x; t < I.ntiles * strips; t += gridDim.x) {
        const TileDesc& T = tiles[I.tile0 + t / strips];
        const int x00 = T.x0, y00 = T.y0 + t % strips * STRIP;
        // with the neighbours that exist (rows below the image: nothing to do)
        const int w = min(ew, Lx - x00), h = min(STRIP + 1, Ly - y00);
        const float* st = state + I.state_off + r0 + r;
        __syncthreads();
        for (int y = warp; y < h; y += NW) {
            const long long s0 = I.site_off + (long long)(y00 + y) * Lx + x00;
            if (C == 32) {
                // a row's slots and samples by lane, then its cells' rows of chains, all in flight
                for (int x0 = 0; x0 < w; x0 += 32) {
                    const bool in = x0 + lane < w;
                    const int slot = in ? slot_map[s0 + x0 + lane] : -1;
                    const float sample = in ? samp[s0 + x0 + lane] : 0.0f;
#pragma unroll 8
                    for (int x = 0; x < min(32, w - x0); ++x) {
                        const int s = __shfl_sync(0xffffffffu, slot, x);
                        const float v = __shfl_sync(0xffffffffu, sample, x);
                        ang[(y * ew + x0 + x) * C + lane] = s >= 0 ? st[(long long)s * I.sstride] : v;
                    }
                }
            } else {
#pragma unroll 4
                for (int x = px; x < w; x += kPixels) {
                    const int s = slot_map[s0 + x];
                    ang[(y * ew + x) * C + ch] = s >= 0 ? st[(long long)s * I.sstride] : samp[s0 + x];
                }
            }
        }
        __syncthreads();
        const int hn = min(STRIP, Ly - y00);
        float hi = 0.0f, lo = 0.0f;
        // the bonds to the right of and below pixel x of row y
        const auto bonds = [&](const float* a, int x, int y, float v, float right) {
            float e = 0.0f;
            if (x + 1 < w) {
                const float d = v - right;
                e += gmrf ? J * gmrf_bond(d) : -J * cosf(q * d);
            }
            if (y + 1 < h) {
                const float d = v - a[ew * C];
                e += gmrf ? J * gmrf_bond(d) : -J * cosf(q * d);
            }
            two_sum(hi, lo, e);
        };
        if (C == 32) {
            const int x_hi = min(tx, Lx - x00);
            for (int y = warp; y < hn; y += NW) {
                const float* a = ang + y * ew * C + lane;
                float v = *a;
#pragma unroll 4
                for (int x = 0; x < x_hi; ++x, a += C) {
                    const float right = x + 1 < w ? a[C] : 0.0f;
                    bonds(a, x, y, v, right);
                    v = right;
                }
            }
        } else {
            for (int i = warp * kPixels + px; i < hn * tx; i += NW * kPixels) {
                const int x = i & (tx - 1), y = i >> tx_log;
                if (x00 + x >= Lx) continue;
                const float* a = ang + (y * ew + x) * C + ch;
                bonds(a, x, y, *a, x + 1 < w ? a[C] : 0.0f);
            }
        }
        sum += two_sum_value(hi, lo);
    }
#pragma unroll
    for (int o = C; o < 32; o <<= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if (lane < C) part[warp][lane] = sum;
    __syncthreads();
    if (warp == 0 && lane < nr) {
        double s = 0.0;
#pragma unroll
        for (int k = 0; k < NW; ++k) s += part[k][lane];
        atomicAdd(out + (long long)blockIdx.z * n_chains + r0 + lane, s * scale);
    }
}

int log2_of(int v) {
    int l = 0;
    while ((1 << l) < v) ++l;
    return l;
}

}  // namespace

cudaError_t launch_predict_tiles(const ImgDev* img, const TileDesc* tiles, int n_tiles, int tx, int ty,
                                 const uint32_t* slot_pos, const double* acc1, const double* acc2,
                                 const float* z, const uint8_t* gap, double n_samples,
                                 const Control* ctl, float* zhat, float* zstd, cudaStream_t s) {
    predict_tile_kernel<<<n_tiles, 128, 0, s>>>(img, tiles, log2_of(tx), tx * ty, slot_pos, acc1, acc2, z,
                                                gap, 1.0 / n_samples, ctl, zhat, zstd);
    return launched();
}

cudaError_t launch_state_tiles(const ImgDev* img, const TileDesc* tiles, int n_tiles, int tx, int ty,
                               int n_max, const uint32_t* slot_pos, const float* samp, float* state,
                               int n_chains, const Control* ctl, float* dense, bool set, cudaStream_t s) {
    n_max = (n_max + 3) & ~3;  // (the map after the rows starts on 16 bytes)
    const size_t smem = (size_t)n_max * 33 * sizeof(float) + (size_t)tx * ty * sizeof(uint16_t);
    const auto kernel = set ? state_tile_kernel<true> : state_tile_kernel<false>;
    if (smem > 48 * 1024) {  // (32 x 16 and 32 x 32 tiles)
        const cudaError_t e =
            cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    kernel<<<dim3(n_tiles, (n_chains + 31) / 32), 256, smem, s>>>(img, tiles, log2_of(tx), tx * ty, n_max,
                                                                  slot_pos, samp, state, n_chains, ctl, dense);
    return launched();
}

cudaError_t launch_energy_tiles(const ImgDev* img, const TileDesc* tiles, int n_img, int max_tiles, int tx,
                                int ty, const float* state, const float* samp, const int* slot_map,
                                int n_chains, float q, double J, int gmrf, double* out, cudaStream_t s) {
    const ScaledJ j(J);
    const auto launch = [&](auto kernel, int strip, int C, int r_base, int chains) {
        const int groups = (chains + C - 1) / C;
        const size_t smem = (size_t)(tx + 1) * (strip + 1) * C * sizeof(float);
        if (smem > 48 * 1024) {  // (32 x 32 tiles)
            const cudaError_t e =
                cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            if (e != cudaSuccess) return e;
        }
        const long long most = 152LL * 8 / std::max(1, groups * n_img) + 1;
        const int blocks = (int)std::max(1LL, std::min((long long)max_tiles * (ty / strip), most));
        kernel<<<dim3(blocks, groups, n_img), 256, smem, s>>>(img, tiles, log2_of(tx), ty, state, samp, slot_map,
                                                              n_chains, r_base, r_base + chains, q, j.m, j.scale, gmrf, out);
        return launched();
    };
    const auto chains_to_lanes = [](int n) { return n <= 1 ? 1 : n <= 2 ? 2 : n <= 4 ? 4 : n <= 8 ? 8 : n <= 16 ? 16 : 32; };
    // below a tile per SM strips of two rows are the shorter chain (us, strips / tiles: 128^2 x 16
    // 14.5 / 18.8, x 4 12.2 / 14.5; 256^2 x 4 20.6 / 15.4, x 16 20.9 / 20.4), by at most 16
    // chains (64^2 x 20 14.4 by 32, 11.6 by 16)
    if ((long long)max_tiles * ((n_chains + 31) / 32) * n_img < 152) {
        switch (chains_to_lanes(n_chains)) {
            case 1: return launch(energy_tile_kernel<2, 8, 1>, 2, 1, 0, n_chains);
            case 2: return launch(energy_tile_kernel<2, 8, 2>, 2, 2, 0, n_chains);
            case 4: return launch(energy_tile_kernel<2, 8, 4>, 2, 4, 0, n_chains);
            case 8: return launch(energy_tile_kernel<2, 8, 8>, 2, 8, 0, n_chains);
            default: return launch(energy_tile_kernel<2, 8, 16>, 2, 16, 0, n_chains);
        }
    }
    // whole groups of 32 chains, then the chains left over by as many lanes as they need
    const int rest = n_chains % 32, whole = rest > 16 ? n_chains : n_chains - rest;
    if (whole) {
        const cudaError_t e = launch(energy_tile_kernel<16, 8, 32>, 16, 32, 0, whole);
        if (e != cudaSuccess || whole == n_chains) return e;
    }
    switch (chains_to_lanes(rest)) {
        case 1: return launch(energy_tile_kernel<16, 8, 1>, 16, 1, whole, rest);
        case 2: return launch(energy_tile_kernel<16, 8, 2>, 16, 2, whole, rest);
        case 4: return launch(energy_tile_kernel<16, 8, 4>, 16, 4, whole, rest);
        case 8: return launch(energy_tile_kernel<16, 8, 8>, 16, 8, whole, rest);
        default: return launch(energy_tile_kernel<16, 8, 16>, 16, 16, whole, rest);
    }
}

}  // namespace mpr
