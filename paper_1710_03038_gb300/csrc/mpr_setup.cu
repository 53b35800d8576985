// Initialisation of a batch: extremes and gap counts, tile records, slot space, ring
// lists and per-slot constants, hot start, sample energy.  Every table is built on the
// device; the host reads back one small record per image (sizes of the slot space) and
// one per batch (largest tiles).
#include <algorithm>
#include <cstring>

#include "mpr_device.cuh"
#include "mpr_internal.h"
#include "mpr_resident.h"

namespace mpr {

namespace {

constexpr double kPiD = 3.14159265358979323846;

__device__ __forceinline__ uint32_t ordered(float f) {
    const uint32_t b = __float_as_uint(f);
    return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}

// Extremes over sample sites and gap counts, per image (blockIdx.y).  Bound by the
// reads (5 bytes per pixel); four pixels per load where the image starts on a multiple
// of four, one set of atomics per block (per warp: 28 us at 2048^2, most of it the
// atomics).
__global__ void __launch_bounds__(256)
minmax_kernel(const ImgDev* img, const float* __restrict__ z, const uint8_t* __restrict__ gap,
              ImgScan* scan) {
    __shared__ uint32_t s_lo[8], s_hi[8];
    __shared__ unsigned s_cnt[8];
    const ImgDev& I = img[blockIdx.y];
    const long long n = (long long)I.Lx * I.Ly, step = (long long)gridDim.x * 256;
    const float* zi = z + I.site_off;
    const uint8_t* gi = gap + I.site_off;
    uint32_t lo = 0xFFFFFFFFu, hi = 0u;
    unsigned cnt = 0;
    const auto one = [&](bool g, float v) {
        const uint32_t o = ordered(v);
        lo = min(lo, g ? 0xFFFFFFFFu : o);
        hi = max(hi, g ? 0u : o);
        cnt += g;
    };
    long long i = blockIdx.x * 256LL + threadIdx.x;
    if (((reinterpret_cast<uintptr_t>(zi) & 15) | (reinterpret_cast<uintptr_t>(gi) & 3)) == 0) {
        for (long long k = i; k < n / 4; k += step) {
            const float4 v = reinterpret_cast<const float4*>(zi)[k];
            const uchar4 g = reinterpret_cast<const uchar4*>(gi)[k];
            one(g.x, v.x);
            one(g.y, v.y);
            one(g.z, v.z);
            one(g.w, v.w);
        }
        i += n / 4 * 4;
    }
    for (; i < n; i += step) one(gi[i], zi[i]);
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    cnt = __reduce_add_sync(0xffffffffu, cnt);
    const int w = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0) {
        s_lo[w] = lo;
        s_hi[w] = hi;
        s_cnt[w] = cnt;
    }
    __syncthreads();
    if (threadIdx.x != 0) return;
    unsigned long long c = 0;
    for (int k = 0; k < 8; ++k) {
        lo = min(lo, s_lo[k]);
        hi = max(hi, s_hi[k]);
        c += s_cnt[k];
    }
    ImgScan& S = scan[blockIdx.y];
    atomicMin(&S.lo, lo);
    atomicMax(&S.hi, hi);
    if (c) atomicAdd(&S.n_gap, c);
}

// Image of a tile: the last whose first tile is not beyond it.
__device__ __forceinline__ int image_of(const ImgDev* img, int n_img, int tile) {
    int a = 0, b = n_img - 1;
    while (a < b) {
        const int m = (a + b + 1) >> 1;
        if (img[m].tile0 <= tile) a = m;
        else b = m - 1;
    }
    return a;
}

// Tile record (image, origin) and its gap sites per colour.
__global__ void __launch_bounds__(256)
tile_count_kernel(const ImgDev* img, int n_img, TileDesc* tiles, const uint8_t* __restrict__ gap,
                  int tx_log, int npix, int ty, int* counts) {
    __shared__ int s_cnt[2];
    __shared__ int s_img;
    const int t = blockIdx.x;
    if (threadIdx.x == 0) s_img = image_of(img, n_img, t);
    if (threadIdx.x < 2) s_cnt[threadIdx.x] = 0;
    __syncthreads();
    const ImgDev& I = img[s_img];
    const int tx = 1 << tx_log, row = (I.Lx + tx - 1) >> tx_log, k = t - I.tile0;
    const int x0 = (k % row) << tx_log, y0 = k / row * ty;
    int c0 = 0, c1 = 0;
    for (int i = threadIdx.x; i < npix; i += 256) {
        const int X = x0 + (i & (tx - 1)), Y = y0 + (i >> tx_log);
        const bool g = X < I.Lx && Y < I.Ly && gap[I.site_off + (long long)Y * I.Lx + X];
        const unsigned m = __ballot_sync(0xffffffffu, g), m1 = __ballot_sync(0xffffffffu, g && ((X + Y) & 1));
        c0 += __popc(m & ~m1);
        c1 += __popc(m1);
    }
    if ((threadIdx.x & 31) == 0) {
        if (c0) atomicAdd(&s_cnt[0], c0);
        if (c1) atomicAdd(&s_cnt[1], c1);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        tiles[t].img = s_img;
        tiles[t].x0 = x0;
        tiles[t].y0 = y0;
        counts[2 * t] = s_cnt[0];
        counts[2 * t + 1] = s_cnt[1];
    }
}

// Slot segments of every tile of an image (one block per image): an exclusive scan of
// the counts, each padded to 4 slots.
__global__ void __launch_bounds__(1024)
tile_scan_kernel(const ImgDev* img, TileDesc* tiles, const int* counts, ImgScan* scan) {
    constexpr int kPer = 8;  // tiles per thread and round
    __shared__ long long s_sum[32];
    __shared__ long long s_base;
    const ImgDev& I = img[blockIdx.x];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) s_base = 0;
    for (int r0 = 0; r0 < I.ntiles; r0 += 1024 * kPer) {
        const int t0 = r0 + threadIdx.x * kPer;
        long long sum = 0;
        for (int k = 0; k < kPer && t0 + k < I.ntiles; ++k) {
            const int2 c = reinterpret_cast<const int2*>(counts)[I.tile0 + t0 + k];
            sum += ((c.x + 3) & ~3) + ((c.y + 3) & ~3);
        }
        long long inc = sum;
        for (int o = 1; o < 32; o <<= 1) {
            const long long v = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += v;
        }
        __syncthreads();  // (the round before has read s_sum and set s_base)
        if (lane == 31) s_sum[warp] = inc;
        __syncthreads();
        long long off = s_base + inc - sum;
        for (int w = 0; w < warp; ++w) off += s_sum[w];
        for (int k = 0; k < kPer && t0 + k < I.ntiles; ++k) {
            const int2 c = reinterpret_cast<const int2*>(counts)[I.tile0 + t0 + k];
            TileDesc& T = tiles[I.tile0 + t0 + k];
            T.cnt[0] = c.x;
            T.cnt[1] = c.y;
            T.off[0] = (int)off;
            off += (c.x + 3) & ~3;
            T.off[1] = (int)off;
            off += (c.y + 3) & ~3;
        }
        __syncthreads();
        if (threadIdx.x == 1023) s_base = off;  // (past the last tile: the total)
        __syncthreads();
    }
    if (threadIdx.x == 0) scan[blockIdx.x].slots = (unsigned long long)s_base;
}

// Slots of a tile's gap sites (row-major inside the tile, per colour) and the rest of
// its record; the padding slots of both segments.
__global__ void __launch_bounds__(256)
tile_fill_kernel(const ImgDev* img, TileDesc* tiles, const uint8_t* __restrict__ gap, int tx_log, int npix,
                 uint32_t* __restrict__ slot_pos, int* __restrict__ slot_map) {
    __shared__ int s_cnt[8][2];
    const int t = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const TileDesc T = tiles[t];
    const ImgDev& I = img[T.img];
    uint32_t* pos = slot_pos + I.slot_off;
    int base0 = T.off[0], base1 = T.off[1];
    for (int i0 = 0; i0 < npix; i0 += 256) {
        const int i = i0 + threadIdx.x, X = T.x0 + (i & ((1 << tx_log) - 1)), Y = T.y0 + (i >> tx_log);
        const bool in = X < I.Lx && Y < I.Ly;
        const long long site = I.site_off + (long long)Y * I.Lx + X;
        const bool g = in && gap[site], black = (X + Y) & 1;
        const unsigned m = __ballot_sync(0xffffffffu, g), m1 = __ballot_sync(0xffffffffu, g && black);
        if (lane == 0) {
            s_cnt[warp][0] = __popc(m & ~m1);
            s_cnt[warp][1] = __popc(m1);
        }
        __syncthreads();
        int k0 = base0, k1 = base1;
        for (int w = 0; w < 8; ++w) {
            if (w < warp) {
                k0 += s_cnt[w][0];
                k1 += s_cnt[w][1];
            }
            base0 += s_cnt[w][0];
            base1 += s_cnt[w][1];
        }
        const unsigned below = (1u << lane) - 1u;
        const int k = black ? k1 + __popc(m1 & below) : k0 + __popc(m & ~m1 & below);
        if (g) pos[k] = ((uint32_t)Y << 16) | (uint32_t)X;
        if (in) slot_map[site] = g ? k : -1;
        __syncthreads();
    }
    if (threadIdx.x < 8) {
        const int c = threadIdx.x >> 2, k = T.cnt[c] + (threadIdx.x & 3);
        if (k < ((T.cnt[c] + 3) & ~3)) pos[T.off[c] + k] = 0xFFFFFFFFu;
    }
    if (threadIdx.x == 0) {
        tiles[t].cp = (int)I.sstride;
        tiles[t].state_off = I.state_off;
        tiles[t].slot_off = I.slot_off;
    }
}

template <typename T>
__device__ __forceinline__ void raise_to(T* at, T v) {
    if (*reinterpret_cast<volatile T*>(at) < v) atomicMax(at, v);
}

// Ring lists (for the pass of colour c, the gap cells of the other colour in the
// 1-cell ring around the tile, corners excluded, as (slot, cell)), then the per-slot
// constants of both colours: for every gap site of colour c, the table entries of its
// four neighbours in the pass of colour c (interior other-colour cells 1 + j, ring
// cells 1 + n_oth + k, 0 where the neighbour is a sample or outside) and its sample
// field, summed over its sample neighbours in the order up, down, left, right: (cos q
// phi, sin q phi), with literal != 0 also (cos phi, sin phi), or for the GMRF model
// (sum of the sample angles, number of existing neighbours).  A cell is read by the
// passes of one colour only, so one map of the tile's cells serves both.  Raises the
// batch's largest tiles in stats.
__global__ void __launch_bounds__(128)
tile_link_kernel(const ImgDev* img, TileDesc* tiles, int tx_log, int ty, const uint32_t* __restrict__ slot_pos,
                 const int* __restrict__ slot_map, int2* __restrict__ halo, int cap,
                 const float* __restrict__ samp_all, float q, int gmrf, int literal,
                 uint2* __restrict__ slot_ref, float4* __restrict__ slot_cs, int res_P, TileStats* stats) {
    extern __shared__ uint16_t cellmap[];  // [(ty + 2) * (tx + 2)]
    __shared__ int n_ring[2];
    const int t = blockIdx.x, tx = 1 << tx_log, ew = tx + 2;
    const TileDesc T = tiles[t];
    const ImgDev& I = img[T.img];
    const int Lx = I.Lx, Ly = I.Ly;
    if (threadIdx.x < 2) n_ring[threadIdx.x] = 0;
    for (int i = threadIdx.x; i < ew * (ty + 2); i += 128) cellmap[i] = 0;
    __syncthreads();
    const uint32_t* spos = slot_pos + I.slot_off;
    const int n0 = T.cnt[0], n = T.cnt[0] + T.cnt[1];
    for (int j = threadIdx.x; j < n; j += 128) {
        const int own = j < n0 ? j : j - n0;
        const uint32_t p = spos[j < n0 ? T.off[0] + own : T.off[1] + own];
        cellmap[((int)(p >> 16) - T.y0 + 1) * ew + (int)(p & 0xFFFFu) - T.x0 + 1] = (uint16_t)(1 + own);
    }
    for (int i = threadIdx.x; i < 2 * (tx + ty); i += 128) {
        int xx, yy;
        if (i < tx) { xx = i + 1; yy = 0; }
        else if (i < 2 * tx) { xx = i - tx + 1; yy = ty + 1; }
        else if (i < 2 * tx + ty) { xx = 0; yy = i - 2 * tx + 1; }
        else { xx = tx + 1; yy = i - 2 * tx - ty + 1; }
        const int X = T.x0 + xx - 1, Y = T.y0 + yy - 1;
        if (X < 0 || X >= Lx || Y < 0 || Y >= Ly) continue;
        const int slot = slot_map[I.site_off + (long long)Y * Lx + X];
        if (slot < 0) continue;
        const int pass = ((xx + yy) & 1) ^ 1;  // the colour whose update reads this cell
        const int k = atomicAdd(&n_ring[pass], 1);
        halo[((long long)t * 2 + pass) * cap + k] = make_int2(slot, yy * ew + xx);
        cellmap[yy * ew + xx] = (uint16_t)(1 + T.cnt[pass ^ 1] + k);
    }
    __syncthreads();
    const float* samp = samp_all + I.site_off;
    for (int j = threadIdx.x; j < n; j += 128) {
        const int k = j < n0 ? T.off[0] + j : T.off[1] + j - n0;
        const uint32_t p = spos[k];
        const int X = (int)(p & 0xFFFFu), Y = (int)(p >> 16);
        const int cell = (Y - T.y0 + 1) * ew + (X - T.x0 + 1);
        float4 f = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        uint32_t ref[4];
#pragma unroll
        for (int m = 0; m < 4; ++m) {  // up, down, left, right
            const int dx = m < 2 ? 0 : 2 * m - 5;
            const int dy = m < 2 ? 2 * m - 1 : 0;
            const int nx = X + dx, ny = Y + dy;
            ref[m] = 0u;
            if (nx < 0 || nx >= Lx || ny < 0 || ny >= Ly) continue;
            if (gmrf) f.y += 1.0f;
            const float v = samp[(long long)ny * Lx + nx];
            if (v >= 0.0f) {
                if (gmrf) {
                    f.x += v;
                } else {
                    float sn, cs;
                    __sincosf(q * v, &sn, &cs);
                    f.x += cs;
                    f.y += sn;
                    if (literal) {
                        __sincosf(v, &sn, &cs);
                        f.z += cs;
                        f.w += sn;
                    }
                }
            } else {
                ref[m] = cellmap[cell + dy * ew + dx];
            }
        }
        slot_ref[I.slot_off + k] = make_uint2(ref[0] | (ref[1] << 16), ref[2] | (ref[3] << 16));
        slot_cs[I.slot_off + k] = f;
    }
    if (threadIdx.x < 2) {
        const int c = threadIdx.x, h = n_ring[c];
        tiles[t].halo_cnt[c] = h;
        raise_to(&stats->gt[c], T.cnt[c ^ 1] + h + 1);
        raise_to(&stats->n_cap[c], T.cnt[c]);
    }
    if (threadIdx.x == 2)
        raise_to(&stats->res_smem,
                 (unsigned)resident_smem(T.cnt[0], T.cnt[1], n_ring[0], n_ring[1], res_P, gmrf != 0));
}

// Tiles with more than e table entries or o own sites, per colour: h[colour][0][e],
// h[colour][1][o] count the tiles of each size.
__global__ void tile_hist_kernel(const TileDesc* tiles, int n, int* h) {
    __shared__ int s[4 * kTileSizes];
    for (int i = threadIdx.x; i < 4 * kTileSizes; i += blockDim.x) s[i] = 0;
    __syncthreads();
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < n; t += gridDim.x * blockDim.x)
        for (int c = 0; c < 2; ++c) {
            atomicAdd(&s[2 * c * kTileSizes + tiles[t].cnt[c ^ 1] + tiles[t].halo_cnt[c] + 1], 1);
            atomicAdd(&s[(2 * c + 1) * kTileSizes + tiles[t].cnt[c]], 1);
        }
    __syncthreads();
    for (int i = threadIdx.x; i < 4 * kTileSizes; i += blockDim.x)
        if (s[i]) atomicAdd(h + i, s[i]);
}

// Tile list of a colour (blockIdx.x): the light tiles (at most e_max table entries and
// own_max own sites) in order from the front, the others in order from the back's
// start; their number to n_light.  One block: a scan over the tiles.
__global__ void __launch_bounds__(1024)
tile_split_kernel(const TileDesc* tiles, int n, int2 max0, int2 max1, int* list, int* n_light) {
    __shared__ int s_sum[32];
    __shared__ int s_base;
    const int c = blockIdx.x, e_max = c ? max1.x : max0.x, own_max = c ? max1.y : max0.y;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const auto light = [&](int t) {
        return tiles[t].cnt[c ^ 1] + tiles[t].halo_cnt[c] + 1 <= e_max && tiles[t].cnt[c] <= own_max;
    };
    // two rounds over the tiles: the light ones' number, then the places
    for (int round = 0; round < 2; ++round) {
        if (threadIdx.x == 0) s_base = 0;
        const int total = round ? n_light[c] : 0;
        for (int r0 = 0; r0 < n; r0 += 1024) {
            const int t = r0 + threadIdx.x;
            const bool l = t < n && light(t);
            const unsigned m = __ballot_sync(0xffffffffu, l);
            __syncthreads();
            if (lane == 0) s_sum[warp] = __popc(m);
            __syncthreads();
            int before = s_base, all = 0;
            for (int w = 0; w < 32; ++w) {
                if (w < warp) before += s_sum[w];
                all += s_sum[w];
            }
            before += __popc(m & ((1u << lane) - 1u));
            if (round && t < n) list[(long long)c * n + (l ? before : total + t - before)] = t;
            __syncthreads();
            if (threadIdx.x == 0) s_base += all;
            __syncthreads();
        }
        if (round == 0 && threadIdx.x == 0) n_light[c] = s_base;
        __syncthreads();
    }
}

// Eq. map into the per-image sample plane (FP64 arithmetic, rounded once);
// gap sites hold -1.
__global__ void map_kernel(const ImgDev* img, const float* z, const uint8_t* gap, float* samp,
                           int unconditional) {
    const ImgDev& I = img[blockIdx.y];
    const long long n = (long long)I.Lx * I.Ly;
    const double zmin = I.zmin, scale = 2.0 * kPiD / ((double)I.zmax - (double)I.zmin);
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x) {
        const long long s = I.site_off + i;
        samp[s] = (unconditional || gap[s]) ? -1.0f : (float)(((double)z[s] - zmin) * scale);
    }
}

// Start of the tiled state: hot (slot -> 2 pi u with the site's first uniform
// at sweep 0xFFFFFFFF) or cold (every gap angle pi); padding slots and the padding chains up
// to the next multiple of 4 hold 0, what wider rows have beyond them stays undefined.  One thread per (slot, four chains): two Philox blocks (words 0 and 2 of the
// pair's) and one 16-byte store; bound by the stores (2048^2 x 32: 215 MB).  A thread per
// pair with a 64-bit division took 75 us of it.
__global__ void __launch_bounds__(256)
hot_start_kernel(const ImgDev* img, const uint32_t* __restrict__ slot_pos, float* __restrict__ state,
                 long long slots, int img_i, int n_chains, uint2 key, uint32_t img_tag, int cold) {
    const ImgDev& I = img[img_i];
    const uint32_t nq = (uint32_t)((n_chains + 3) / 4);  // chains in fours per slot
    const long long row = I.sstride / 4;
    float4* st = reinterpret_cast<float4*>(state + I.state_off);
    const long long total = slots * nq;
    for (long long t = blockIdx.x * 256LL + threadIdx.x; t < total; t += gridDim.x * 256LL) {
        const long long k = total <= 0xFFFFFFFFLL ? (long long)((uint32_t)t / nq) : t / nq;
        const int c0 = 4 * (int)(t - k * nq);
        const uint32_t p = slot_pos[I.slot_off + k];
        float4 v = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        if (p != 0xFFFFFFFFu) {
            if (cold) {
                v = make_float4(kPi, kPi, kPi, kPi);
            } else {
                const int X = (int)(p & 0xFFFFu), Y = (int)(p >> 16);
                const uint4 a = philox4x32_10(site_counter(X, Y, (X + Y) & 1, 0xFFFFFFFFu, (uint32_t)c0,
                                                           (uint32_t)img_i | img_tag), key);
                const uint4 b = philox4x32_10(site_counter(X, Y, (X + Y) & 1, 0xFFFFFFFFu, (uint32_t)c0 + 2u,
                                                           (uint32_t)img_i | img_tag), key);
                v = make_float4(kTwoPi * u24(a.x), kTwoPi * u24(a.z), kTwoPi * u24(b.x), kTwoPi * u24(b.z));
            }
            if (c0 + 1 >= n_chains) v.y = 0.0f;
            if (c0 + 2 >= n_chains) v.z = 0.0f;
            if (c0 + 3 >= n_chains) v.w = 0.0f;
        }
        st[k * row + c0 / 4] = v;
    }
}

// Sample specific energy sums (Eq. mpr-sse): one bond's energy in FP32, the same
// expression as the allocation-free entry point's, summed in two FP32 words per lane and
// FP64 from there.  A warp takes 31 columns and 8 rows: the pixel below is the next
// row's own, the one on the right the next lane's.
__device__ __forceinline__ float bond_energy(float d, float q, float J, int gmrf) {
    return gmrf ? J * (d * d * (float)(0.5 / (kPiD * kPiD)) - 1.0f) : -J * cosf(q * d);
}

__global__ void __launch_bounds__(256)
sample_energy_kernel(const ImgDev* img, const float* __restrict__ samp, float q, float J, double scale,
                     int gmrf, double* sums, unsigned long long* npairs) {
    constexpr int kRows = 8;
    __shared__ double s_sum[8];
    __shared__ unsigned s_cnt[8];
    const ImgDev& I = img[blockIdx.y];
    const int Lx = I.Lx, Ly = I.Ly, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nx = (Lx + 30) / 31;
    const long long tasks = (long long)nx * ((Ly + kRows - 1) / kRows);
    double s = 0.0;
    unsigned cnt = 0;
    for (long long task = blockIdx.x * 8LL + warp; task < tasks; task += gridDim.x * 8LL) {
        const int x = (int)(task % nx) * 31 + lane, y0 = (int)(task / nx) * kRows;
        const bool in = x < Lx, own = in && lane < 31;
        const float* p = samp + I.site_off + (long long)y0 * Lx + x;
        const int rows = min(kRows, Ly - y0);
        float hi = 0.0f, lo = 0.0f;
        float v = in ? *p : -1.0f;
#pragma unroll 4
        for (int k = 0; k < rows; ++k, p += Lx) {
            const float below = in && y0 + k + 1 < Ly ? p[Lx] : -1.0f;
            const float right = __shfl_down_sync(0xffffffffu, v, 1);
            if (own && v >= 0.0f && right >= 0.0f) {
                two_sum(hi, lo, bond_energy(v - right, q, J, gmrf));
                ++cnt;
            }
            if (own && v >= 0.0f && below >= 0.0f) {
                two_sum(hi, lo, bond_energy(v - below, q, J, gmrf));
                ++cnt;
            }
            v = below;
        }
        s += two_sum_value(hi, lo);
    }
    s = warp_sum(s);
    cnt = warp_sum(cnt);
    if (lane == 0) {
        s_sum[warp] = s;
        s_cnt[warp] = cnt;
    }
    __syncthreads();
    if (threadIdx.x != 0) return;
    unsigned long long c = cnt;
    for (int k = 1; k < 8; ++k) {
        s += s_sum[k];
        c += s_cnt[k];
    }
    if (s != 0.0) atomicAdd(sums + blockIdx.y, s * scale);
    if (c) atomicAdd(npairs + blockIdx.y, c);
}

__global__ void sample_energy_finish_kernel(ImgDev* img, const double* sums, const unsigned long long* npairs,
                                            int n_img) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n_img) return;
    img[i].n_sp = (long long)npairs[i];
    img[i].E_ss = sums[i];
    img[i].e_s = npairs[i] > 0 ? sums[i] / (double)npairs[i] : __longlong_as_double(0x7FF8000000000000LL);
}

// A small host record in the kernel's parameters: a copy from pageable host memory
// would wait for the stream first.
constexpr int kBlobWords = 896;
struct Blob {
    uint32_t w[kBlobWords];
};
__global__ void put_kernel(const __grid_constant__ Blob b, uint32_t* dst, int words) {
    for (int i = threadIdx.x; i < words; i += blockDim.x) dst[i] = b.w[i];
}

int log2_of(int v) {
    int l = 0;
    while ((1 << l) < v) ++l;
    return l;
}

int blocks_for(long long n, long long per, int most) {
    return (int)std::max(1LL, std::min((n + per - 1) / per, (long long)most));
}

}  // namespace

cudaError_t launch_put(void* dst, const void* src, size_t bytes, cudaStream_t s) {
    for (size_t o = 0; o < bytes; o += sizeof(Blob)) {
        Blob b;
        const size_t n = std::min(sizeof(Blob), bytes - o);
        std::memcpy(b.w, static_cast<const char*>(src) + o, n);
        put_kernel<<<1, 256, 0, s>>>(b, reinterpret_cast<uint32_t*>(static_cast<char*>(dst) + o), (int)(n / 4));
        const cudaError_t e = launched();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t launch_minmax(const ImgDev* img, int n_img, long long max_sites, const float* z,
                          const uint8_t* gap, ImgScan* scan, cudaStream_t s) {
    minmax_kernel<<<dim3(blocks_for(max_sites, 4096, 608), n_img), 256, 0, s>>>(img, z, gap, scan);
    return launched();
}

cudaError_t launch_tile_count(const ImgDev* img, int n_img, TileDesc* tiles, int n_tiles, const uint8_t* gap,
                              int tx, int ty, int* counts, ImgScan* scan, cudaStream_t s) {
    tile_count_kernel<<<n_tiles, 256, 0, s>>>(img, n_img, tiles, gap, log2_of(tx), tx * ty, ty, counts);
    cudaError_t e = launched();
    if (e != cudaSuccess) return e;
    tile_scan_kernel<<<n_img, 1024, 0, s>>>(img, tiles, counts, scan);
    return launched();
}

cudaError_t launch_map(const ImgDev* img, int n_img, long long max_sites, const float* z, const uint8_t* gap,
                       float* samp, bool unconditional, cudaStream_t s) {
    map_kernel<<<dim3(blocks_for(max_sites, 256, 2048), n_img), 256, 0, s>>>(img, z, gap, samp,
                                                                              unconditional ? 1 : 0);
    return launched();
}

cudaError_t launch_tile_tables(const ImgDev* img, TileDesc* tiles, int n_tiles, const uint8_t* gap, int tx,
                               int ty, uint32_t* slot_pos, int* slot_map, int2* halo, int halo_cap,
                               const float* samp, float q, int gmrf, int literal, uint2* slot_ref,
                               float4* slot_cs, int res_P, TileStats* stats, cudaStream_t s) {
    tile_fill_kernel<<<n_tiles, 256, 0, s>>>(img, tiles, gap, log2_of(tx), tx * ty, slot_pos, slot_map);
    cudaError_t e = launched();
    if (e != cudaSuccess) return e;
    tile_link_kernel<<<n_tiles, 128, sizeof(uint16_t) * (tx + 2) * (ty + 2), s>>>(
        img, tiles, log2_of(tx), ty, slot_pos, slot_map, halo, halo_cap, samp, q, gmrf, literal, slot_ref,
        slot_cs, res_P, stats);
    return launched();
}

cudaError_t launch_tile_hist(const TileDesc* tiles, int n_tiles, int* hist, cudaStream_t s) {
    tile_hist_kernel<<<blocks_for(n_tiles, 256, 152), 256, 0, s>>>(tiles, n_tiles, hist);
    return launched();
}

cudaError_t launch_tile_split(const TileDesc* tiles, int n_tiles, const int e_max[2], const int own_max[2],
                              int* list, int* n_light, cudaStream_t s) {
    tile_split_kernel<<<2, 1024, 0, s>>>(tiles, n_tiles, make_int2(e_max[0], own_max[0]),
                                         make_int2(e_max[1], own_max[1]), list, n_light);
    return launched();
}

cudaError_t launch_hot_start(const ImgDev* img, const uint32_t* slot_pos, float* state, long long slots,
                             int img_i, int n_chains, uint2 key, uint32_t img_tag, bool cold, cudaStream_t s) {
    const long long n = slots * ((n_chains + 3) / 4);
    if (n == 0) return cudaSuccess;
    hot_start_kernel<<<blocks_for(n, 1024, 152 * 32), 256, 0, s>>>(img, slot_pos, state, slots, img_i, n_chains,
                                                                   key, img_tag, cold ? 1 : 0);
    return launched();
}

cudaError_t launch_sample_energy(ImgDev* img, int n_img, long long max_sites, const float* samp, float q,
                                 double J, int gmrf, double* sums, unsigned long long* npairs, cudaStream_t s) {
    const ScaledJ j(J);
    sample_energy_kernel<<<dim3(blocks_for(max_sites, 31 * 64, 152 * 8), n_img), 256, 0, s>>>(
        img, samp, q, j.m, j.scale, gmrf, sums, npairs);
    cudaError_t e = launched();
    if (e != cudaSuccess) return e;
    sample_energy_finish_kernel<<<(n_img + 127) / 128, 128, 0, s>>>(img, sums, npairs, n_img);
    return launched();
}

}  // namespace mpr
