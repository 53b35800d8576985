// Resident sweeps (mpr_resident.cu): arguments and launchers.
#pragma once

#include "mpr_internal.h"

namespace mpr {

struct ResidentArgs {
    SweepArgs a;         // as for the colour passes (flags without the per-colour kEnergy rule: set
                         // when the sweeps record energies)
    int n;               // sweeps of the run
    int equil, stats;    // adapt a; add the energies to the chains' sums
    double A_targ, k_a;
    int group, n_whole;  // chains per group, groups of that size; the remaining chains follow
    int P, P_rest;       // chain pairs per site of a whole group and of the remaining chains
    int n_tiles;
    int recorders;       // blocks per image and group that record energies (recorded runs only)
    int spread_log;      // 2^spread_log words per chain and parity: about one per 64 tiles of an image
    // [parity of the sweep][spread][chain]: tiles done << 40 | accepted proposals (zero
    // between launches)
    unsigned long long* words;
    ulonglong2* packets;   // [3][tile][64 places][chain pairs]: (angle, epoch) words of both chains
    ulonglong2* energies;  // [3][tile][chain]: (half of a double, epoch) words
    uint32_t* epoch;       // epoch of the last launch's last pass
    int polls;             // reads of a wait before it gives up
};

// The most blocks that the device holds at once: 152 SMs of seven.
constexpr int kResidentBlocks = 152 * 7;
// (about a second)
constexpr int kDefaultPolls = 1 << 21;

// Shared memory of a block: the fixed part, the own sites' records and sums, the two
// tables and the sites' packet places, for a tile of n0 red and n1 black sites with h0
// and h1 ring cells and P chain pairs per site.
constexpr int kResidentFixed = 2304;
__host__ __device__ inline unsigned resident_sum_bytes(int n_max) {
    return (40u * (unsigned)n_max + 15u) / 16u * 16u;
}
__host__ __device__ inline unsigned resident_smem(int n0, int n1, int h0, int h1, int P, bool gmrf) {
    const unsigned n = (unsigned)(n0 + n1);
    const unsigned tables = (n + (unsigned)(h0 + h1) + 2u) * (unsigned)P * (gmrf ? 8u : 16u) + 2u * n;
    // (a block that records energies: a double per thread)
    return (unsigned)kResidentFixed + 32u * n + resident_sum_bytes(n0 > n1 ? n0 : n1) +
           (tables > 1024u ? tables : 1024u);
}
// n sweeps as resident launches of at most kMost each (a chain's word holds 2^40 accepted
// proposals: 2^20 sweeps of 2048 tiles).  *done: the sweeps launched.  A launch that is
// refused because the blocks cannot run at once is no error: a context may use fewer SMs
// than the device has, by which residency was decided, and the sweeps left over can go as
// launches per colour (*done < n).
constexpr int kMostSweeps = 1 << 20;
template <typename Launch>
cudaError_t resident_chunks(int n, Launch launch, int* done) {
    for (*done = 0; *done < n;) {
        const int m = n - *done < kMostSweeps ? n - *done : kMostSweeps;
        const cudaError_t e = launch(m);
        if (e == cudaErrorCooperativeLaunchTooLarge || e == cudaErrorNotSupported) return cudaSuccess;
        if (e != cudaSuccess) return e;
        *done += m;
    }
    return cudaSuccess;
}

// Blocks that record the energies of a group of that many chains.
int resident_recorders(int group);
// Blocks of that size that the device holds at once (0: no cooperative launches, or
// one block does not fit).
cudaError_t resident_blocks(size_t smem, long long* blocks);
// Sets the kernels' shared-memory limit (not during a capture).
cudaError_t resident_prepare(bool gmrf);
cudaError_t launch_resident(const ResidentArgs& ra, int n_groups, size_t smem, cudaStream_t s);

namespace resident {
using Kernel = void (*)(ResidentArgs);
Kernel pick_mpr(bool acc, bool energy);
Kernel pick_gmrf(bool acc, bool energy);
}  // namespace resident

}  // namespace mpr
