// Posterior energy of a labelling and minimum-energy tracking.
//
//   H(x) = sum over unordered neighbour pairs <ij> of V(x_i, x_j) + sum_i U(g_i, x_i)
//
// is the energy of the posterior Gibbs measure pi_post ~ exp(-H) (Section 4,
// Eq. mrf_gauss_noise_posterior_distribution) with the per-edge pair weight
// of the single-site conditional (Eq. gibbs_sampler_elementary_step).  Each
// term is a model coefficient times an integer count:
//   pair sum: Potts -> pairs with equal labels (V = -c_P each),
//             truncated linear -> sum of min(|x_i - x_j|, T) (V = c_T each);
//   data sum: Gaussian -> sum of (g_i - x_i)^2 (U = that / (2 sigma^2)),
//             flip -> sites with x_i != g_i (U = -ln p there, -ln(1 - p) elsewhere);
//             none (prior only) -> 0.
// The sums are reduced exactly in integers; H is combined from them in FP64 by
// one thread.  Pairs are counted once: right and down neighbours
// (and the two lower diagonals for the 8-neighbourhood), free boundary.
#include "energy_dev.cuh"

namespace pcad {

namespace {

constexpr int kEThreads = 256;

// One pair term over the 4 sites of a word: equal labels (Potts) or
// min(|a - b|, T), for the bytes of `mask`.
__device__ __forceinline__ uint32_t pair_term(const EnergyCoef &k, uint32_t a, uint32_t b,
                                              uint32_t T4, uint32_t mask)
{
    if (k.potts)
        return (uint32_t)__popc(__vcmpeq4(a, b) & mask & 0x01010101u);
    return __dp4a(__vminu4(__vabsdiffu4(a, b), T4) & mask, 0x01010101u, 0u);
}

// The sums, H from them and, when tracking, the trace, the running minimum and
// its state, in one launch: with a launch each for the sums, H and the copy of
// a new minimum, energy tracking of a 301 x 453 image spent 6.5 us per sweep
// beside a 12 us sweep, nearly all of it launch latency (4.9 us here).  The blocks copy the
// labels to the one of two planes that does not hold the minimum; the last
// block to finish (a ticket) combines H and, for a new minimum, makes that
// plane the minimum's.  A thread takes 4 sites (one word) per step.
__global__ void __launch_bounds__(kEThreads)
    energy_kernel(const uint8_t *__restrict__ x, const uint8_t *__restrict__ g, int H, int W,
                  int pitch, EnergyCoef k, unsigned long long *sums, double *out, EnergyTrack tr,
                  const uint32_t *tdev, uint32_t sweep_off)
{
    const int Wq = (W + 3) >> 2;
    const long n = (long)H * Wq;
    const uint32_t T4 = (uint32_t)min(k.T, 255) * 0x01010101u;
    uint8_t *const spare = tr.trace ? (*tr.which ? tr.xb[0] : tr.xb[1]) : nullptr;
    EnergyLast last{};   // early: nothing writes it before the last block does
    if (tr.trace && threadIdx.x == 0)
        last = energy_last(tr, tdev, sweep_off);
    // 64 bits: a thread may see any share of a large image
    unsigned long long pair = 0, data = 0;
    for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (long)gridDim.x * blockDim.x) {
        const int r = (int)(i / Wq), q = (int)(i - (long)r * Wq);
        const uint8_t *px = x + (size_t)r * pitch + 4 * q;
        const uint32_t M = *reinterpret_cast<const uint32_t *>(px);
        const uint32_t G = *reinterpret_cast<const uint32_t *>(g + (size_t)r * pitch + 4 * q);
        const int nv = W - 4 * q;                              // sites from this word on
        const uint32_t in = nv >= 4 ? 0xFFFFFFFFu : (1u << (8 * nv)) - 1u;
        // sites with a right neighbour, and their neighbours' word
        const uint32_t inr = nv >= 5 ? 0xFFFFFFFFu : (nv == 1 ? 0u : (1u << (8 * (nv - 1))) - 1u);
        const uint32_t R = (M >> 8) | (nv > 4 ? (uint32_t)px[4] << 24 : 0u);
        uint32_t p = pair_term(k, M, R, T4, inr);
        if (r + 1 < H) {
            const uint32_t D = *reinterpret_cast<const uint32_t *>(px + pitch);
            p += pair_term(k, M, D, T4, in);
            if (k.nbhd == 8) {
                const uint32_t DR = (D >> 8) | (nv > 4 ? (uint32_t)px[pitch + 4] << 24 : 0u);
                const uint32_t DL = (D << 8) | (q > 0 ? (uint32_t)px[pitch - 1] : 0u);
                p += pair_term(k, M, DR, T4, inr);
                p += pair_term(k, M, DL, T4, q > 0 ? in : in & 0xFFFFFF00u);
            }
        }
        pair += p;
        if (!k.none) {
            const uint32_t d = __vabsdiffu4(G, M) & in;
            data += k.gauss ? __dp4a(d, d, 0u) : (uint32_t)__popc(__vcmpne4(G, M) & in & 0x01010101u);
        }
        if (spare)
            *reinterpret_cast<uint32_t *>(spare + (size_t)r * pitch + 4 * q) = M;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        pair += __shfl_down_sync(0xFFFFFFFFu, pair, o);
        data += __shfl_down_sync(0xFFFFFFFFu, data, o);
    }
    __shared__ unsigned long long sp[kEThreads / 32], sd[kEThreads / 32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (lane == 0) {
        sp[warp] = pair;
        sd[warp] = data;
    }
    __syncthreads();
    if (threadIdx.x != 0)
        return;
    unsigned long long P = 0, D = 0;
    for (int w = 0; w < kEThreads / 32; ++w) {
        P += sp[w];
        D += sd[w];
    }
    atomicAdd(&sums[0], P);
    atomicAdd(&sums[1], D);
    __threadfence();
    if (atomicAdd(&sums[2], 1ull) != (unsigned long long)gridDim.x - 1ull)
        return;
    energy_finish(k, sums, out, tr, last);
}

int reduce_grid(long n)
{
    const long blocks = (n + kEThreads - 1) / kEThreads;
    return (int)(blocks < 1024 ? (blocks < 1 ? 1 : blocks) : 1024);
}

}  // namespace

EnergyCoef energy_coef(const pcad_model &m, long n_sites)
{
    EnergyCoef k{};
    k.potts = m.pair == PCAD_PAIR_POTTS;
    k.T = m.pair == PCAD_PAIR_POTTS ? 1 : m.pair_T;
    k.gauss = m.noise == PCAD_NOISE_GAUSS;
    k.none = m.noise == PCAD_NOISE_NONE;
    k.nbhd = m.nbhd;
    k.pair_c = (k.potts ? -1.0 : 1.0) * (double)m.pair_coef;
    k.two_s2 = 2.0 * (double)m.sigma * (double)m.sigma;
    if (m.noise == PCAD_NOISE_FLIP) {
        const double p = (double)m.flip_p;
        k.lf_same = -std::log1p(-p);
        k.lf_diff = -std::log(p);
    }
    k.n_sites = (unsigned long long)n_sites;
    return k;
}

cudaError_t launch_energy(const uint8_t *x, const uint8_t *g, int H, int W, int pitch,
                          const EnergyCoef &k, unsigned long long *sums, double *out,
                          const EnergyTrack &tr, const uint32_t *tdev, uint32_t sweep_off,
                          cudaStream_t s)
{
    const long n = (long)H * ((W + 3) / 4);
    energy_kernel<<<reduce_grid(n), kEThreads, 0, s>>>(x, g, H, W, pitch, k, sums, out, tr, tdev,
                                                       sweep_off);
    return cudaGetLastError();
}

}  // namespace pcad
