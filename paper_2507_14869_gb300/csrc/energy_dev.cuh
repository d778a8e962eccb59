// The last step of an energy reduction, shared by the energy kernel and the
// sweeps that reduce the energy of the state they read: H from the integer
// sums and, when tracking, the trace and the running minimum.
#pragma once

#include "pcad_internal.h"

namespace pcad {

struct EnergyLast {
    unsigned int n;               // entries recorded
    int which;                    // the minimum's plane
    double best;
    unsigned long long done;      // completed sweeps of the state
};

__device__ __forceinline__ EnergyLast energy_last(const EnergyTrack &tr, const uint32_t *tdev,
                                                  uint32_t sweep_off)
{
    EnergyLast l;
    l.n = *tr.n;
    l.which = *tr.which;
    l.best = *tr.best;
    l.done = (unsigned long long)(*tdev + sweep_off) + 1ull;
    return l;
}

// One thread, after the last block's ticket: every block's sums are in (and
// every block has read tr.which).  Zeroes the sums for the next reduction.
__device__ __forceinline__ void energy_finish(const EnergyCoef &k, unsigned long long *sums,
                                              double *out, const EnergyTrack &tr,
                                              const EnergyLast &last)
{
    __threadfence();
    const double fp = (double)atomicExch(&sums[0], 0ull), fd = (double)atomicExch(&sums[1], 0ull);
    sums[2] = 0;
    double e = __dmul_rn(k.pair_c, fp);
    if (k.gauss)
        e = __dadd_rn(e, __ddiv_rn(fd, k.two_s2));
    else if (!k.none)
        e = __dadd_rn(e, __dadd_rn(__dmul_rn(k.lf_same, __dsub_rn((double)k.n_sites, fd)),
                                   __dmul_rn(k.lf_diff, fd)));
    if (out) {   // H and the two sums (exact in FP64: both are < 2^53)
        out[0] = e;
        out[1] = fp;
        out[2] = fd;
    }
    if (tr.trace) {
        if (last.n < (unsigned int)tr.cap) {
            tr.trace[last.n] = e;
            *tr.n = last.n + 1;
        }
        if (e < last.best) {
            *tr.best = e;
            *tr.best_sweep = last.done;
            *tr.which = last.which ^ 1;
        }
    }
}

}  // namespace pcad
