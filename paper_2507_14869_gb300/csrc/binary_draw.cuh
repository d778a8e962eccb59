// The two-label draw: a comparison of the uniform with a threshold of the
// site's configuration (resident.cu builds the table), shared by the two-label
// sweeps and the tile-resident kernel.
#pragma once

#include "pcad_internal.h"

namespace pcad {
namespace bind {

// Table entries: configuration index e = 2 (b + n1) + x_i with the base
// b = (g (NB + 1) + nm) (NB + 1).
template <int NB>
constexpr int btab_entries()
{
    return 4 * (NB + 1) * (NB + 1);
}

constexpr int kThrBytes = 6656;   // a ThrTab of either neighbourhood

// Thresholds of every configuration in shared memory: thr[] (one 32-bit read
// and a compare per draw), the full entries for the rare draws near a
// threshold, and the largest uncertain band.
template <int NB>
struct ThrTab {
    int thr[NB == 4 ? btab_entries<4>() : 2 * 168];   // NB 4: [2 b + x]; 8: [168 x + b]
    uint4 full[btab_entries<NB>()];
    uint32_t band;
};

static_assert(sizeof(ThrTab<4>) <= kThrBytes && sizeof(ThrTab<8>) <= kThrBytes, "table space");

template <int NB>
__device__ __forceinline__ int thr_index(int e)
{
    return NB == 4 ? e : (e >> 1) + 168 * (e & 1);
}

// (ends with a block barrier)
template <int NB>
__device__ __forceinline__ void load_thresholds(ThrTab<NB> &tab, const uint4 *src, int tid, int n)
{
    if (tid == 0)
        tab.band = 0u;
    __syncthreads();
    for (int i = tid; i < btab_entries<NB>(); i += n) {
        const uint4 e = src[i];
        tab.full[i] = e;
        tab.thr[thr_index<NB>(i)] = (int)e.x;
        atomicMax(&tab.band, e.z);
    }
    __syncthreads();
}

// New labels of one quad from its Philox words u: S holds base + count per
// byte, M the current labels (0 or 1 per byte).  Returns the labels as bytes;
// adds the draws of the bytes of `act` that the FP64 re-draw decides to nre:
// those with u in [A, B), a band around the threshold, looked at only when
// some draw of the quad lies within the largest band of its threshold.
template <int NB>
__device__ __forceinline__ uint32_t quad_draw(const ThrTab<NB> &tab, uint32_t S, uint32_t M,
                                              const uint32_t (&u)[4], uint32_t act, uint32_t &nre)
{
    const uint32_t K = NB == 4 ? 2u * S + M : S;   // NB 4: at most 99 per byte, no carry
    uint32_t out = 0u;
    int near = 0x7FFFFFFF;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        int i = (int)((K >> (8 * j)) & 0xFFu);
        if (NB == 8)
            i += 168 * (int)((M >> (8 * j)) & 1u);
        const int d = (int)(u[j] >> 8) - tab.thr[i];
        out |= d >= 0 ? 1u << (8 * j) : 0u;
        near = min(near, abs(d));
    }
    if ((uint32_t)near <= tab.band) {
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if ((act >> (8 * j)) & 1u) {
                const uint4 e = tab.full[((S >> (8 * j)) & 0xFFu) * 2u + ((M >> (8 * j)) & 1u)];
                nre += ((u[j] >> 8) - e.y) < e.z ? 1u : 0u;
            }
    }
    return out;
}

}  // namespace bind
}  // namespace pcad
