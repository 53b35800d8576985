// Resident sweeps: a run of n sweeps as one cooperative launch, for batches whose
// tiles all fit the GPU at once.
//
// What bounds small batches is not the updates but the chain of dependent launches:
// three per sweep (two colour passes, the bookkeeping), each a few microseconds for
// a fraction of a microsecond of work, and each colour pass rebuilds its tile's
// constants and tables.  Here one thread block keeps one 16 x 16 tile of one chain
// group for the whole run: neighbour rows, sample fields and random-stream words of
// both colours stay in shared memory, and so do the two tables of cells.  A pass
// writes its new cells straight into the table that the other colour's pass reads.
// Equilibration / sampling sweeps, us, launches per colour -> resident: 64^2 x 7
// chains at 30 % gaps 10.8 / 7.2 -> 4.1 / 4.3; 256^2 x 16 at 50 % 13.8 / 11.9 -> 8.4 /
// 7.1; 350^2 x 4 12.1 / 10.8 -> 6.6 / 5.5.  Which runs come here: resident_runs.  What is
// left of a 64^2 pass (2 us) is latency: about 1 us of dependent instructions of one warp
// step, the rest the trip of the packets through L2.
//
// Exchange.  Only the ring cells come from other blocks.  A block publishes its
// boundary sites as packets of two 64-bit words (angle, epoch), one per chain of the
// pair, and a reader polls the words it needs until they carry the epoch of the pass
// that it waits for: one trip through L2, no barrier and no fence (with a barrier of the
// group's blocks per colour a 64^2 sweep took 6.3 us, with packets 4.3).  Per chain and
// parity of the sweep, words count the tiles that have finished a sweep (upper 24 bits)
// and their accepted proposals (lower 40): an equilibration sweep starts once the last
// one's counts are complete (they decide a), a sampling sweep once those of the sweep
// before the last are.  A chain has one such word per 64 tiles, because the arrivals at
// one word are served one after another (961 tiles x 32 chains on one word each: 24.6 us
// an equilibration sweep, more than the launches).  Black packets are read in the next
// sweep, so a tile that may start sweep k may still owe the reads of sweep k - 1: three
// packet buffers, by sweep, keep every packet until all its readers have finished a
// later pass.  Recorded energies go the same way, one packet per tile and chain, to
// blocks that only sum and record them.  The chains of a
// group are independent of all others: nothing waits across images or groups.
//
// The arithmetic, its order inside a block and the split into blocks are those of
// the launch per colour, so both give the same bits.
//
// Waiting.  The launch is cooperative (every block is resident), a block waits only
// for blocks of its own launch, every wait has an iteration limit (ResidentArgs::polls),
// and one that gives up sets the status word and ends its block.  The states and sums are
// then those of a run cut short: whatever reads them out gives NaN (mpr_check).
#pragma once

#include "mpr_device.cuh"
#include "mpr_resident.h"
#include "mpr_tiled_kernel.cuh"

namespace mpr {
namespace resident {

using namespace tiled;

constexpr int kNW = 4, kNT = kNW * 32;  // warps and threads of a block, as the 16 x 16 pass
constexpr int kRing = 32;               // ring cells of one colour (16 + 16)
constexpr unsigned kNoEdge = 0xFFu;
constexpr int kRecorderChains = 4;
// 72 registers a thread: at 64 the variants that record energies spill
constexpr int kBlocksPerSM = 7;

// Shared memory: fixed part, then per own site of both colours the neighbour rows and
// the constants (32 bytes), sampling runs' fixed-point sums (one colour's sites of the
// pass, 8 bytes each; both colours' of the run, 16 bytes each), the two tables, and per
// own site its places among the tile's packets (2 bytes).
struct Fixed {
    float4 red[kNW * 16];
    float a[32], alpha[32];
    uint32_t cnt[32], prev[2][32];  // accepted proposals up to a sweep, up to two sweeps before
    float a_new, alpha_new;         // what a chain below the target takes after the last sweep
    // what a pass of a colour needs, by colour: read where it is used, which keeps some
    // twenty registers free for the update
    int n[2], off[2], halo[2], first[2];  // own sites, their slots, ring cells, first record
    unsigned tab[2];                      // table, byte offset in the block's shared memory
    unsigned long long* my_words;         // the words of chain 0 at which this tile counts
    ulonglong2* my_energies;              // this tile's energy packets
    ulonglong2* my_packets;               // and its first boundary packet (pair 0 of the group)
    long long word_step, energy_buf, packet_buf;
    int ring[2][kRing];  // ring cells: packet index (tile, place) of the cell's site
    int slot[kRing];     // ring cells of the first red pass: their slots
};
constexpr size_t kFixed = kResidentFixed;
static_assert(sizeof(Fixed) <= kFixed && kFixed % 16 == 0, "fixed part of the shared memory");

// A tile's packets: top row 0-15, bottom row 16-31, left column 32-47, right column
// 48-63 (a corner site has two).
__device__ __forceinline__ unsigned edge_places(int lx, int ly) {
    const unsigned row = ly == 0 ? (unsigned)lx : ly == 15 ? 16u + lx : kNoEdge;
    const unsigned col = lx == 0 ? 32u + ly : lx == 15 ? 48u + ly : kNoEdge;
    // the first place in the low byte, so that an inner site shows in one comparison
    return row != kNoEdge ? row | (col << 8) : col | (kNoEdge << 8);
}

__device__ __forceinline__ void publish(ulonglong2* pk, float2 v, uint32_t epoch) {
    const unsigned long long e = (unsigned long long)epoch << 32;
    asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(pk),
                 "l"(e | __float_as_uint(v.x)), "l"(e | __float_as_uint(v.y)) : "memory");
}

__device__ __forceinline__ bool try_receive(const ulonglong2* pk, uint32_t epoch, float2& v) {
    unsigned long long x, y;
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(x), "=l"(y) : "l"(pk) : "memory");
    v = make_float2(__uint_as_float((uint32_t)x), __uint_as_float((uint32_t)y));
    return (uint32_t)(x >> 32) == epoch && (uint32_t)(y >> 32) == epoch;
}

// The packet's angles once both words carry the epoch; false when it never comes.
__device__ __forceinline__ bool receive(const ulonglong2* pk, uint32_t epoch, float2& v, int polls) {
    for (int k = 0; k < polls; ++k)
        if (try_receive(pk, epoch, v)) return true;
    return false;
}

// A chain's word once `tiles` arrivals (modulo 2^24) are in.
__device__ __forceinline__ bool arrived(const unsigned long long* word, uint32_t tiles,
                                        unsigned long long& v, int polls) {
    for (int k = 0; k < polls; ++k) {
        asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(word) : "memory");
        // at most one sweep's arrivals beyond the awaited ones are in
        if ((((uint32_t)(v >> 40) - tiles) & 0xFFFFFFu) < 0x800000u) return true;
    }
    return false;
}

// Tiles of an image that count at word s of a chain (recorded runs: and the recorder).
__device__ __forceinline__ uint32_t arrivals_at(const ResidentArgs& ra, int tiles_img, int s, bool energy) {
    return (uint32_t)((tiles_img - s + (1 << ra.spread_log) - 1) >> ra.spread_log) + (energy && s == 0 ? 1u : 0u);
}

// Sums the energies of every sweep of up to four chains of one image (961 tiles x 32
// chains for one block: 40 us a sweep).
__device__ __forceinline__ bool run_recorder(const ResidentArgs& ra, unsigned char* smem, int img, int r0,
                                             int ng) {
    const SweepArgs& a = ra.a;
    const ImgDev& I = a.img[img];
    double* part = reinterpret_cast<double*>(smem + kFixed);
    constexpr int C = kRecorderChains, t_step = kNT / C;
    const int tid = threadIdx.x, ch = tid & (C - 1);
    const long long chain0 = (long long)img * a.n_chains + r0;
    const uint32_t epoch0 = *ra.epoch;
    const ulonglong2* pk = ra.energies + (long long)I.tile0 * a.n_chains + r0 + ch;
    const long long pk_buf = (long long)ra.n_tiles * a.n_chains;
    double sum = 0.0, sum2 = 0.0, e = 0.0;  // of chain tid
    for (int k = 0; k < ra.n; ++k) {
        if (tid < ng)  // (the sweep before is recorded)
            atomicAdd(ra.words + (((long long)(k & 1) * a.n_img * a.n_chains) << ra.spread_log) + chain0 + tid, 1ull << 40);
        const uint32_t epoch = epoch0 + 2u * (uint32_t)k + 2u;
        double E = 0.0;
        bool there = true;
        // eight packets in flight
        for (int t0 = tid / C; ch < ng && there && t0 < I.ntiles; t0 += 8 * t_step) {
            float2 v[8];
            unsigned wait = 0;
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                v[i] = f2(0.0f);
                const int t = t0 + i * t_step;
                if (t < I.ntiles &&
                    !try_receive(pk + (k % 3) * pk_buf + (long long)t * a.n_chains, epoch, v[i]))
                    wait |= 1u << i;
            }
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                if (wait >> i & 1u)
                    there = there && receive(pk + (k % 3) * pk_buf + (long long)(t0 + i * t_step) * a.n_chains,
                                             epoch, v[i], ra.polls);
                E += __hiloint2double(__float_as_int(v[i].y), __float_as_int(v[i].x));
            }
        }
        part[tid] = E;
        if (__syncthreads_or(!there)) return false;
        if (tid < ng) {
            E = 0.0;
            for (int t = 0; t < t_step; ++t) E += part[t * C + tid];
            e = (E + I.E_ss) / I.n_bonds;
            sum += e;
            sum2 += e * e;
        }
        __syncthreads();
    }
    if (tid < ng) {
        a.ch.e_last[chain0 + tid] = e;
        if (ra.stats) {
            a.ch.e_sum[chain0 + tid] += sum;
            a.ch.e_sum2[chain0 + tid] += sum2;
        }
    }
    return true;
}

// One tile and chain group (WHOLE: of 2P chains) for the whole run.
template <int P, bool ACC, bool ENERGY, int MODEL, bool WHOLE>
__device__ __forceinline__ bool run_tile(const ResidentArgs& ra, unsigned char* smem, int tile, int r0,
                                         int ng) {
    constexpr int SPW = 32 / P;
    constexpr int NTP = kNT / P;
    constexpr int CB = Cell<MODEL>::bytes;
    constexpr uint32_t kRow = (uint32_t)CB * P;
    const SweepArgs& a = ra.a;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int p = lane & (P - 1), s = lane / P, e_lo = tid / P;
    const bool has0 = WHOLE || 2 * p < ng, has1 = WHOLE || 2 * p + 1 < ng;
    Fixed* fx = reinterpret_cast<Fixed*>(smem);
    uint4* rows = reinterpret_cast<uint4*>(smem + kFixed);
    const int np = (a.n_chains + 1) >> 1;  // packets from one place to the next

    // -- constants of both colours, ring cells, zero cells ---------------------------
    {
        const TileDesc T = a.tiles[tile];
        const ImgDev& I = a.img[T.img];
        const int n0 = T.cnt[0], n1 = T.cnt[1], nmax = max(n0, n1);
        uint4* cons = rows + n0 + n1;
        const unsigned acc0 = (unsigned)(kFixed + 32 * (n0 + n1));
        const unsigned tab0 = acc0 + (ACC ? resident_sum_bytes(nmax) : 0u);
        const unsigned tab1 = tab0 + (unsigned)(1 + n1 + T.halo_cnt[0]) * kRow;
        const unsigned edge0 = tab1 + (unsigned)(1 + n0 + T.halo_cnt[1]) * kRow;
        uint16_t* edge = reinterpret_cast<uint16_t*>(smem + edge0);
        const float* st = a.state + T.state_off + r0 + 2 * p;
        if (tid == 0) {
            fx->n[0] = n0;
            fx->n[1] = n1;
            fx->off[0] = T.off[0];
            fx->off[1] = T.off[1];
            fx->halo[0] = T.halo_cnt[0];
            fx->halo[1] = T.halo_cnt[1];
            fx->first[0] = 0;
            fx->first[1] = n0;
            fx->tab[0] = tab0;
            fx->tab[1] = tab1;
            fx->word_step = (long long)a.n_img * a.n_chains;
            fx->my_words = ra.words + ((tile - I.tile0) & ((1 << ra.spread_log) - 1)) * fx->word_step +
                           (long long)T.img * a.n_chains + r0;
            fx->energy_buf = (long long)ra.n_tiles * a.n_chains;
            fx->my_energies = ra.energies + (long long)tile * a.n_chains + r0;
            fx->packet_buf = (long long)ra.n_tiles * 64 * np;
            fx->my_packets = ra.packets + (long long)tile * 64 * np + (r0 >> 1);
        }
        for (int j = tid; j < n0 + n1; j += kNT) {
            const int c = j >= n0;
            const long long slot = T.slot_off + (c ? T.off[1] + (j - n0) : T.off[0] + j);
            const uint2 r = a.slot_ref[slot];
            const float4 f = a.slot_cs[slot];
            rows[j] = make_uint4((r.x & 0xFFFFu) * kRow, (r.x >> 16) * kRow, (r.y & 0xFFFFu) * kRow,
                                 (r.y >> 16) * kRow);
            const uint32_t pos = a.slot_pos[slot];
            const uint2 pw = philox_site_words((pos & 0xFFFF0000u) | ((pos & 0xFFFFu) >> 1),
                                               (uint32_t)T.img | a.img_tag | ((uint32_t)c << 31), a.rk);
            cons[j] = make_uint4(__float_as_uint(f.x), __float_as_uint(f.y), pw.x, pw.y);
            edge[j] = (uint16_t)edge_places((int)(pos & 0xFFFFu) - T.x0, (int)(pos >> 16) - T.y0);
        }
        if (tid < 2 * kRing) {
            const int c = tid / kRing, k = tid % kRing;
            if (k < (c ? T.halo_cnt[1] : T.halo_cnt[0])) {
                const int2 h = a.halo[((long long)tile * 2 + c) * a.halo_cap + k];  // slot, cell
                const int xx = h.y % 18, yy = h.y / 18, row = (I.Lx + 15) / 16;
                const int t = yy == 0 ? -row : yy == 17 ? row : xx == 0 ? -1 : 1;
                const int place = yy == 0 ? 16 + xx - 1 : yy == 17 ? xx - 1 : xx == 0 ? 48 + yy - 1 : 32 + yy - 1;
                fx->ring[c][k] = t * 64 + place;  // from this tile's first packet
                if (c == 0) fx->slot[k] = h.x;
            }
        }
        if (tid < 2 * P) {
            unsigned char* z = smem + (tid < P ? tab0 : tab1) + (tid & (P - 1)) * CB;
            if (CB == 8) *reinterpret_cast<float2*>(z) = f2(0.0f);
            else *reinterpret_cast<float4*>(z) = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        }
        if (ACC)
            for (unsigned j = tid; j < resident_sum_bytes(nmax) / 4; j += kNT)
                reinterpret_cast<uint32_t*>(smem + acc0)[j] = 0u;
        const long long chain0 = (long long)T.img * a.n_chains + r0;
        if (tid < 32) {
            fx->cnt[tid] = fx->prev[0][tid] = fx->prev[1][tid] = 0u;
            fx->a[tid] = tid < ng ? a.ch.a[chain0 + tid] : 1.0f;
            fx->alpha[tid] = tid >= ng ? 0.0f
                             : (a.flags & kAlphaOne) ? proposal_width(1.0f) : a.ch.alpha[chain0 + tid];
        }
        if (has0)  // black cells as they stand; the red ones follow from the first red pass
            for (int e = e_lo; e < n1; e += NTP)
                store_cell<MODEL>(smem + tab0 + (size_t)((1 + e) * P + p) * CB, a.q,
                                  *reinterpret_cast<const float2*>(st + (long long)(T.off[1] + e) * T.cp));
    }
    if (tid == kNT - 1 && ra.equil) {
        fx->a_new = (float)(1.0 + (double)(a.ctl->equil_index + 1u) / ra.k_a);
        fx->alpha_new = proposal_width(fx->a_new);
    }
    __syncthreads();

    const TileDesc& T = a.tiles[tile];
    const ImgDev& I = a.img[T.img];
    const long long slot_off = T.slot_off;
    const int cp = T.cp;
    float* st = a.state + T.state_off + r0 + 2 * p;  // the lane's pair at slot 0
    const UpdateConst uk{a.q, a.inv_q, a.two_pi_q, a.J};
    const float c_acc = 1.4426950408889634f * I.invT;
    const uint32_t sweep0 = a.ctl->sweep, epoch0 = *ra.epoch;
    const uint32_t c2 = (uint32_t)(r0 >> 1) + (uint32_t)p;
    // counts below A_targ n_gap: whole numbers below its ceiling
    const uint32_t low_cnt = (uint32_t)ceil(ra.A_targ * (double)I.n_gap);
    const int tiles_img = I.ntiles;
    float2 vn = f2(0.0f);  // own angles of the next warp step
    if (has0 && warp * SPW + s < fx->n[0])
        vn = *reinterpret_cast<const float2*>(st + (long long)(fx->off[0] + warp * SPW + s) * cp);

    // the word of chain ch at spread sp after sweep k: false when it never completes
    const auto finished = [&](int k, int ch, int sp, unsigned long long& v) {
        return arrived(ra.words + (((k & 1) << ra.spread_log) + sp) * fx->word_step +
                           (long long)T.img * a.n_chains + r0 + ch,
                       (uint32_t)((k >> 1) + 1) * arrivals_at(ra, tiles_img, sp, ENERGY), v, ra.polls);
    };
    // adds up the accepted proposals of every chain up to sweep k
    const auto count = [&](int k) {
        for (int w = tid; w < (2 * P) << ra.spread_log; w += kNT) {
            const int ch = w & (2 * P - 1);
            if (!WHOLE && ch >= ng) continue;
            unsigned long long v;
            if (!finished(k, ch, w / (2 * P), v)) return false;
            atomicAdd(&fx->cnt[ch], (uint32_t)v);  // (differences are taken modulo 2^32)
        }
        return true;
    };

    bool stop = false;  // the same in every thread
    int buf = 0, buf_before = 2;  // packet buffers of sweeps k and k - 1
    float2 alpha_s = f2(0.0f);
    for (int k = 0; k < ra.n; ++k) {
        const PhiloxPair pair_words = philox_pair_words(sweep0 + (uint32_t)k, c2, a.rk);
        unsigned cnt0 = 0, cnt1 = 0;
        float2 esum = f2(0.0f);
#pragma unroll 1
        for (int c = 0; c < 2; ++c) {
            const bool settle = c == 0 && k > 0 && ra.equil;
            // -- wait: the counts that this sweep needs, then the ring cells ------------
            bool there = true;
            if (settle) {
                there = count(k - 1);
            } else if (c == 0 && k > 1) {
                // one chain's words for the tiles (and the first recorder), one for each other recorder
                const int rec = tid - (1 << ra.spread_log) + 1;
                unsigned long long v;
                if (rec <= 0) there = finished(k - 2, 0, tid, v);
                else if (ENERGY && rec * kRecorderChains < ng) there = finished(k - 2, rec * kRecorderChains, 0, v);
            }
            if (has0) {
                // the last sweep's black sites for the red pass, this sweep's red ones for the black
                const ulonglong2* from = fx->my_packets + (c ? buf : buf_before) * fx->packet_buf + p;
                const uint32_t epoch = epoch0 + 2u * (uint32_t)k + (uint32_t)c;
                unsigned char* ring = smem + fx->tab[c] + (size_t)((1 + fx->n[c ^ 1]) * P + p) * CB;
                const int n_halo = fx->halo[c];
                for (int e = e_lo; e < n_halo; e += NTP) {
                    float2 v;
                    if (c == 0 && k == 0) {
                        v = *reinterpret_cast<const float2*>(st + (long long)fx->slot[e] * cp);
                    } else if (!receive(from + (long long)fx->ring[c][e] * np, epoch, v, ra.polls)) {
                        there = false;
                        break;
                    }
                    store_cell<MODEL>(ring + (size_t)e * kRow, a.q, v);
                }
            }
            stop = __syncthreads_or(!there);
            if (stop) break;
            if (c == 0) {
                alpha_s = make_float2(fx->alpha[2 * p], fx->alpha[2 * p + 1]);
                if (settle) {
                    const uint32_t* before = fx->prev[(k - 1) & 1];
                    if (fx->cnt[2 * p] - before[2 * p] < low_cnt) alpha_s.x = fx->alpha_new;
                    if (fx->cnt[2 * p + 1] - before[2 * p + 1] < low_cnt) alpha_s.y = fx->alpha_new;
                }
            } else if (k > 0 && ra.equil && tid < ng) {
                // (every thread has its new alpha)
                if (fx->cnt[tid] - fx->prev[(k - 1) & 1][tid] < low_cnt) {
                    fx->a[tid] = fx->a_new;
                    fx->alpha[tid] = fx->alpha_new;
                }
                fx->prev[(k - 1) & 1][tid] = fx->cnt[tid];
                fx->cnt[tid] = 0u;
            }
            const int n_own = fx->n[c], off_own = fx->off[c];
            const unsigned char* tabp = smem + fx->tab[c] + p * CB;  // this lane's column
            const uint4* own_rows = rows + fx->first[c];
            const uint4* own_k = own_rows + fx->n[0] + fx->n[1];
            const bool energy = ENERGY && c == 1;
            if (energy && has0) {
                const uint4* cons = rows + fx->n[0] + fx->n[1];  // the red sites first
                for (int e = e_lo; e < fx->n[0]; e += NTP) {
                    const unsigned char* t = tabp + (size_t)(1 + e) * kRow;
                    const float4 cell = MODEL == kModelGMRF ? float4{} : tab_f4(t);
                    const float2 v = MODEL == kModelGMRF ? tab_f2(t) : f2(0.0f);
                    esum = add_sample_bonds<MODEL>(a, I, cell, v, __uint_as_float(cons[e].x),
                                                   __uint_as_float(cons[e].y), slot_off + fx->off[0] + e, esum);
                }
            }
            const int n_steps = (n_own + SPW - 1) / SPW;
            unsigned char* next = smem + fx->tab[c ^ 1] + (size_t)(P + p) * CB;  // its cells of the other table
            const uint16_t* own_edge = reinterpret_cast<const uint16_t*>(
                smem + fx->tab[1] + (size_t)(1 + fx->n[0] + fx->halo[1]) * kRow) + fx->first[c];
            uint32_t* accs = reinterpret_cast<uint32_t*>(smem + kFixed + 32 * (fx->n[0] + fx->n[1]));
            const int nmax = max(fx->n[0], fx->n[1]);
            float* sto = st + (long long)off_own * cp;
            ulonglong2* to = fx->my_packets + buf * fx->packet_buf + p;
            const uint32_t epoch = epoch0 + 2u * (uint32_t)k + (uint32_t)c + 1u;
            for (int g = warp; g < n_steps; g += kNW) {
                const float2 vc = vn;
                {
                    const int jn = (g + kNW) * SPW + s;
                    vn = f2(0.0f);
                    if (has0 && jn < n_own) vn = *reinterpret_cast<const float2*>(sto + jn * cp);
                }
                const int j = g * SPW + s;
                const bool in = j < n_own, act = in && has0, act1 = act && has1;
                const int jj = in ? j : 0;
                const uint4 rw = own_rows[jj];
                const uint4 kk = own_k[jj];
                const PairRand u = pair_uniforms_flipped(philox_finish(kk.z, kk.w, pair_words, a.rk));
                const PairOut o = update_site<MODEL, ENERGY>(a, I, tabp, rw, kk, float4{}, vc, u, uk, alpha_s,
                                                             c_acc, slot_off + off_own + jj);
                if (act) {
                    const unsigned places = own_edge[j];
                    if ((places & 0xFFu) != kNoEdge) {
                        publish(to + (long long)((places & 0xFFu) * np), o.phi, epoch);
                        if ((places >> 8) != kNoEdge) publish(to + (long long)((places >> 8) * np), o.phi, epoch);
                    }
                    *reinterpret_cast<float2*>(sto + j * cp) = o.phi;
                    store_cell<MODEL>(next + (size_t)j * kRow, a.q, o.phi);
                }
                if (ACC) {
                    const float x0 = act ? o.phi.x : 0.0f, x1 = act1 ? o.phi.y : 0.0f;
                    const float sa = x0 + x1, sb = fmaf(x0, x0, x1 * x1);
                    if (P >= 16) {
                        const bool lower = p < 8;
                        const float v = (lower ? sa : sb) + __shfl_xor_sync(0xffffffffu, lower ? sb : sa, 8);
                        if (in)
                            atomicAdd(&accs[(lower ? 0 : nmax) + j],
                                      __float2uint_rn(v * (lower ? 16777216.0f : 2097152.0f)));
                    } else if (in) {
                        atomicAdd(&accs[j], __float2uint_rn(sa * 16777216.0f));
                        atomicAdd(&accs[nmax + j], __float2uint_rn(sb * 2097152.0f));
                    }
                }
                cnt0 += (act && o.acc0) ? 1u : 0u;
                cnt1 += (act1 && o.acc1) ? 1u : 0u;
                if (energy) esum = add2(esum, make_float2(act ? o.e.x : 0.0f, act1 ? o.e.y : 0.0f));
            }
            // the next pass's first own angles (this thread's own stores)
            vn = f2(0.0f);
            if (has0 && warp * SPW + s < fx->n[c ^ 1])
                vn = *reinterpret_cast<const float2*>(st + (long long)(fx->off[c ^ 1] + warp * SPW + s) * cp);
            if (c == 1) {
                float e0 = esum.x, e1 = esum.y;
#pragma unroll
                for (int o = P; o < 32; o <<= 1) {
                    cnt0 += __shfl_xor_sync(0xffffffffu, cnt0, o);
                    cnt1 += __shfl_xor_sync(0xffffffffu, cnt1, o);
                    if (ENERGY) {
                        e0 += __shfl_xor_sync(0xffffffffu, e0, o);
                        e1 += __shfl_xor_sync(0xffffffffu, e1, o);
                    }
                }
                if (lane < P)
                    fx->red[warp * P + lane] = make_float4(e0, e1, __uint_as_float(cnt0), __uint_as_float(cnt1));
            }
            __syncthreads();  // cells, sums and totals of this pass are in shared memory
            if (ACC && tid < n_own) {
                // the site's sums of the run, in 64 bits
                unsigned long long* run = reinterpret_cast<unsigned long long*>(accs + 2 * nmax) + 2 * (fx->first[c] + tid);
                run[0] += accs[tid];
                run[1] += accs[nmax + tid];
                accs[tid] = accs[nmax + tid] = 0u;
            }
            if (c == 1 && tid == kNT - 1 && ra.equil) {  // for the sweep after next's chains, while they wait
                fx->a_new = (float)(1.0 + (double)(a.ctl->equil_index + (uint32_t)k + 1u) / ra.k_a);
                fx->alpha_new = proposal_width(fx->a_new);
            }
            if (c == 1 && tid < ng) {  // thread ch: the tile's totals of chain ch
                double E = 0.0;
                unsigned m = 0;
#pragma unroll
                for (int w = 0; w < kNW; ++w) {
                    const float4 r = fx->red[w * P + (tid >> 1)];
                    if (ENERGY) E += (double)((tid & 1) ? r.y : r.x);
                    m += __float_as_uint((tid & 1) ? r.w : r.z);
                }
                // sampling sweeps run ahead of one another: only the last one's counts
                if (!ra.equil && k + 1 < ra.n) m = 0;
                atomicAdd(fx->my_words + (((k & 1) * fx->word_step) << ra.spread_log) + tid, (1ull << 40) | m);
                if (ENERGY)
                    publish(fx->my_energies + buf * fx->energy_buf + tid,
                            make_float2(__int_as_float(__double2loint(E)), __int_as_float(__double2hiint(E))),
                            epoch);
            }
        }
        if (stop) break;
        buf_before = buf;
        buf = buf == 2 ? 0 : buf + 1;
    }
    if (stop) return false;
    if (tile == I.tile0) {  // the image's first tile keeps the chains' records
        if (__syncthreads_or(!count(ra.n - 1))) return false;
        const long long ch = (long long)T.img * a.n_chains + r0 + tid;
        if (tid < ng) {
            const uint32_t cnt = fx->cnt[tid] - fx->prev[(ra.n - 1) & 1][tid];
            a.ch.acc_last[ch] = cnt;
            if (ra.equil) {
                const float v = cnt < low_cnt ? fx->a_new : fx->a[tid];
                a.ch.a[ch] = v;
                a.ch.alpha[ch] = proposal_width(v);
            }
            if (!ENERGY) a.ch.e_last[ch] = __longlong_as_double(0x7FF8000000000000LL);
        }
    }
    if (ACC) {
        // one add per site and run: the sums of a run are exact in 64 bits.  Thread t takes
        // the red and the black site t, as in the passes, so that it reads what it wrote itself
        // (a walk over the records in order would cross threads, with no barrier since the last
        // pass's sums)
        const bool accum2 = (a.flags & kAccumulate2) != 0;
        const unsigned long long* run = reinterpret_cast<const unsigned long long*>(
            smem + kFixed + 32 * (fx->n[0] + fx->n[1]) + 8 * max(fx->n[0], fx->n[1]));
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            if (tid >= fx->n[c]) continue;
            const long long slot = slot_off + fx->off[c] + tid;
            const unsigned long long* sums = run + 2 * (fx->first[c] + tid);
            atomicAdd(a.acc1 + slot, (double)sums[0] * 0x1p-24);
            if (accum2) atomicAdd(a.acc2 + slot, (double)sums[1] * 0x1p-21);
        }
    }
    return true;
}

template <int P, bool ACC, bool ENERGY, int MODEL>
__device__ __forceinline__ bool run_group(const ResidentArgs& ra, unsigned char* smem, int tile, int r0, int ng) {
    return ng == 2 * P ? run_tile<P, ACC, ENERGY, MODEL, true>(ra, smem, tile, r0, ng)
                       : run_tile<P, ACC, ENERGY, MODEL, false>(ra, smem, tile, r0, ng);
}

template <bool ACC, bool ENERGY, int MODEL>
__global__ void __launch_bounds__(kNT, kBlocksPerSM) resident_kernel(const __grid_constant__ ResidentArgs ra) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int tile = blockIdx.x, grp = blockIdx.y;
    const int r0 = grp * ra.group;  // the remaining chains follow the whole groups
    const int ng = min(ra.group, ra.a.n_chains - r0);
    // the pairs per site of the launch per colour: the remaining chains have their own
    const int P = grp < ra.n_whole ? ra.P : ra.P_rest;
    bool ok;
    if (ENERGY && tile >= ra.n_tiles) {
        const int img = (tile - ra.n_tiles) / ra.recorders, rec = (tile - ra.n_tiles) % ra.recorders;
        const int left = min(kRecorderChains, ng - rec * kRecorderChains);
        ok = left <= 0 || run_recorder(ra, smem, img, r0 + rec * kRecorderChains, left);
    } else {
        switch (P) {
            case 1: ok = run_group<1, ACC, ENERGY, MODEL>(ra, smem, tile, r0, ng); break;
            case 2: ok = run_group<2, ACC, ENERGY, MODEL>(ra, smem, tile, r0, ng); break;
            case 4: ok = run_group<4, ACC, ENERGY, MODEL>(ra, smem, tile, r0, ng); break;
            case 8: ok = run_group<8, ACC, ENERGY, MODEL>(ra, smem, tile, r0, ng); break;
            default: ok = run_group<16, ACC, ENERGY, MODEL>(ra, smem, tile, r0, ng); break;
        }
    }
    Control* ctl = ra.a.ctl;
    if (!ok && threadIdx.x == 0) atomicOr(&ctl->status, 2u);
    // the last block to finish clears the words and advances the counters
    const bool mine = threadIdx.x == 0;
    __syncthreads();
    unsigned last = 0;
    if (mine) {
        __threadfence();
        last = atomicAdd(&ctl->ticket, 1u) == gridDim.x * gridDim.y - 1;
    }
    if (__syncthreads_or((int)last)) {
        const int nw = (2 * ra.a.n_img * ra.a.n_chains) << ra.spread_log;
        for (int i = threadIdx.x; i < nw; i += kNT) ra.words[i] = 0ull;
        if (mine) {
            ctl->ticket = 0;
            ctl->sweep += (uint32_t)ra.n;
            *ra.epoch += 2u * (uint32_t)ra.n;
            if (ra.equil) ctl->equil_index += (uint32_t)ra.n;
        }
    }
}

template <int MODEL>
Kernel pick_model(bool acc, bool energy) {
    static const Kernel k[4] = {resident_kernel<false, false, MODEL>, resident_kernel<true, false, MODEL>,
                                resident_kernel<false, true, MODEL>, resident_kernel<true, true, MODEL>};
    return k[(acc ? 1 : 0) + (energy ? 2 : 0)];
}

}  // namespace resident
}  // namespace mpr
