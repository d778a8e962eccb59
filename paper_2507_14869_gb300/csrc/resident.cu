// Whole chains of small two-label images in one launch, in shared memory
// (lazy PCA, Section 5.2; checkerboard Gibbs, Section 5.1), and sweeps of
// larger two-label images.
//
// A 64 x 64 binary chain does 4096 site-updates per sweep: one launch per
// sweep costs more than the sweep.  Here one CTA of 1024 threads (a chain of
// a batch, the smallest images) or a cluster of 8 (resident_cluster_kernel)
// holds the whole state in shared memory and runs every sweep of a run in one
// launch, with one block barrier per sweep (PCA) or colour phase (Gibbs).
//
// The draw.  With two labels the conditional law of site i depends on the
// site only through its configuration (x_i, g_i, n1, nm): n1 neighbours at
// label 1, nm neighbours outside the image (the rest at label 0).  The prior
// sums P(0) = n1 + nm T and P(1) = n0 + nm T are small integers, exact in
// FP32 in any order.  For one configuration the FP32 draw of the other
// kernels picks label 1 exactly when fl(fl(u 2^-24) Z) >= C0, a monotone
// test in the 24-bit uniform numerator u; its certified margin leaves one
// contiguous band [A, B) of u uncertain, where the FP64 re-draw decides,
// again by a monotone test (label 1 iff u >= D).  The whole draw therefore
// is "label 1 iff u >= max(A, min(D, B))", and the FP64 re-draw count is
// the number of draws with u in [A, B).  A set-up kernel finds A, B and D
// for every configuration by bisection over u, calling the very FP32 draw
// and FP64 re-draw functions the other kernels use, so the labels and the
// re-draw count are theirs draw for draw.
//
// The sweep.  Labels live in shared memory as bytes in padded rows (four
// zero bytes left and right of each row, a zero row above and below), so a
// thread reads the 4-site word of its quad and the words around it and
// counts the label-1 neighbours of its four sites with byte-wise integer
// adds (no carries: a count is at most 8).  A per-site base byte holds
// (g_i, nm) in the table's index.  One Philox call gives the quad's four
// uniforms of the sweep.  Posterior-mean counts accumulate in packed 16-bit
// registers and reach global memory at the end of the launch.
#include "binary_draw.cuh"

namespace pcad {

namespace {

using namespace bind;

constexpr int kResThreads = 1024;
constexpr int kResMaxQuadsPerThread = 4;
constexpr int kResMaxSmem = 200 * 1024;

constexpr int kBtabStride = 4 * 9 * 9;   // entries per table in a batch's table array

__device__ unsigned long long g_btab_redraws;   // re-draw counter of the bisection (unused)

// One warp per configuration: A (first u with label 1 or an uncertain FP32
// draw), B (first u with a certain label 1), D (first u whose FP64 draw is
// label 1).  Entry {max(A, min(D, B)), A, B - A, 0}; impossible
// configurations (n1 + nm > NB) get zeros.
// Row blockIdx.y of the grid takes job blockIdx.y.  A table takes about 15 us, nearly
// all of it the latency of 72 bisection steps in order, so a batch's tables go in one
// launch: a batch of 16 two-label chains is created in 1.13 ms against 1.65.
template <int N>
struct BtabJobs {
    BtabJob job[N];
};

template <int NB, int N>
__global__ void __launch_bounds__(256) btab_kernel(const __grid_constant__ BtabJobs<N> jobs)
{
    const DevModel &m = jobs.job[N > 1 ? blockIdx.y : 0].m;
    uint4 *const out = jobs.job[N > 1 ? blockIdx.y : 0].out;
    constexpr int NE = btab_entries<NB>();
    const int e = (int)(blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5));
    const int lane = (int)(threadIdx.x & 31u);
    if (e >= NE)
        return;   // whole warps
    const int xi = e & 1, v = e >> 1;
    const int n1 = v % (NB + 1), nm = (v / (NB + 1)) % (NB + 1), g = v / ((NB + 1) * (NB + 1));
    if (n1 + nm > NB) {
        if (lane == 0)
            out[e] = make_uint4(0u, 0u, 0u, 0u);
        return;
    }
    SiteIn<NB> in{};
    in.g = g;
    in.xi = xi;
#pragma unroll
    for (int j = 0; j < NB; ++j)
        in.xni[j] = j < n1 ? 1 : (j < n1 + nm ? kMissingLabelI : 0);
    uint32_t bound[2];
#pragma unroll 1
    for (int which = 0; which < 2; ++which) {
        uint32_t lo = 0u, hi = 1u << 24;
        while (lo < hi) {
            const uint32_t mid = (lo + hi) >> 1;
            in.ub = mid;
            bool certain = true;
            const int s = draw_binary<NB>(m, in, certain);
            const bool hit = which == 0 ? (s == 1 || !certain) : (s == 1 && certain);
            if (hit)
                hi = mid;
            else
                lo = mid + 1u;
        }
        bound[which] = lo;
    }
    uint32_t lo = 0u, hi = 1u << 24;
    while (lo < hi) {   // warp-uniform: every lane holds the same bounds
        const uint32_t mid = (lo + hi) >> 1;
        in.ub = mid;
        int s = warp_redraw_fp64<NB>(m, lane == 0, in, 0, &g_btab_redraws);
        s = __shfl_sync(0xFFFFFFFFu, s, 0);
        if (s == 1)
            hi = mid;
        else
            lo = mid + 1u;
    }
    const uint32_t A = bound[0], B = bound[1], D = lo;
    if (lane == 0)
        out[e] = make_uint4(max(A, min(D, B)), A, B - A, 0u);
}

// Padded label plane: H + 2 rows of Wq + 8 bytes (Wq = W rounded up to 4).
inline int res_plane_bytes(int H, int W)
{
    return (H + 2) * (((W + 3) & ~3) + 8);
}

// Shared memory of a launch: table, one (Gibbs) or two (PCA) planes, base bytes.
inline int res_smem_bytes(int nb, bool gibbs, int H, int W)
{
    (void)nb;
    return kThrBytes + (gibbs ? 1 : 2) * res_plane_bytes(H, W) + H * ((W + 3) & ~3);
}

// Label-1 neighbour counts of the 4 sites of the word at index o (one per
// byte), from the padded plane X with pw words per row; M gets the word.
template <int NB>
__device__ __forceinline__ uint32_t quad_counts(const uint32_t *X, int o, int pw, uint32_t &M)
{
    M = X[o];
    const uint32_t U = X[o - pw], D = X[o + pw];
    uint32_t S = U + D + ((M << 8) | (X[o - 1] >> 24)) + ((M >> 8) | (X[o + 1] << 24));
    if (NB == 8)
        S += ((U << 8) | (X[o - pw - 1] >> 24)) + ((U >> 8) | (X[o - pw + 1] << 24)) +
             ((D << 8) | (X[o + pw - 1] >> 24)) + ((D >> 8) | (X[o + pw + 1] << 24));
    return S;
}

__device__ __forceinline__ void quad_words(const SweepArgs &a, uint32_t tag, uint32_t t, int r,
                                           int c4, uint32_t (&u)[4])
{
    philox4x32_10((uint32_t)c4, (uint32_t)(r + a.row_off), t, (tag << 24) | (a.chain & 0xFFFFFFu),
                  (uint32_t)(a.seed & 0xFFFFFFFFull), (uint32_t)(a.seed >> 32), u[0], u[1], u[2],
                  u[3]);
}

// Gibbs colour phase ph of a quad in row r: the bytes whose site has colour
// ph ((r + c) mod 2 for 4 neighbours, (r mod 2, c mod 2) for 8).
template <int NB>
__device__ __forceinline__ uint32_t phase_mask(int r, int ph)
{
    if (NB == 4)
        return ((r ^ ph) & 1) == 0 ? 0x00FF00FFu : 0xFF00FF00u;
    if ((r & 1) != (ph >> 1))
        return 0u;
    return (ph & 1) ? 0xFF00FF00u : 0x00FF00FFu;
}

// One CTA runs nsweeps sweeps of one chain from plane xg_in with the
// threshold table btab; the final labels go to xg_out (pitch a.pitch), the
// posterior-mean counts are added to a.acc and the re-draw count to
// a.fp64_draws.  Thread i takes the quads i, i + 1024, ... (QPT at most), a
// quad being 4 adjacent sites of a row.
template <int NB, bool GIBBS, int QPT>
__device__ __forceinline__ void resident_run(const SweepArgs &a, const uint4 *btab,
                                             const uint8_t *xg_in, uint8_t *xg_out, int nsweeps)
{
    extern __shared__ __align__(16) uint8_t sm[];
    const int tid = (int)threadIdx.x;
    const int H = a.H, W = a.W;
    const int Wq = (W + 3) & ~3, P = Wq + 8, pw = P >> 2;
    const int plane = (H + 2) * P;
    const int nplanes = GIBBS ? 1 : 2;
    ThrTab<NB> &tab = *reinterpret_cast<ThrTab<NB> *>(sm);
    uint8_t *const pl0 = sm + kThrBytes;
    uint8_t *const pl1 = pl0 + (GIBBS ? 0 : plane);
    uint8_t *const bs = pl0 + nplanes * plane;
    {
        uint32_t *z = reinterpret_cast<uint32_t *>(pl0);
        const int nz = (nplanes * plane + H * Wq) >> 2;
        for (int i = tid; i < nz; i += kResThreads)
            z[i] = 0u;   // borders, row padding and the base bytes of padding sites stay 0
    }
    load_thresholds<NB>(tab, btab, tid, kResThreads);
    for (int i = tid; i < H * W; i += kResThreads) {
        const int r = i / W, c = i - (i / W) * W;
        const int gv = a.g[(size_t)r * a.pitch + c];
        pl0[(r + 1) * P + 4 + c] = xg_in[(size_t)r * a.pitch + c];
        int nm = (r == 0) + (r == H - 1) + (c == 0) + (c == W - 1);
        if (NB == 8)
            nm += (r == 0 || c == 0) + (r == 0 || c == W - 1) + (r == H - 1 || c == 0) +
                  (r == H - 1 || c == W - 1);
        bs[r * Wq + c] = (uint8_t)((gv * (NB + 1) + nm) * (NB + 1));
    }
    __syncthreads();

    const int qrow = Wq >> 2, nq = H * qrow;
    int qo[QPT], qr[QPT], qc[QPT];
    uint32_t qb[QPT], qm[QPT], clo[QPT], chi[QPT];
#pragma unroll
    for (int i = 0; i < QPT; ++i) {
        const int q = tid + i * kResThreads;
        qo[i] = -1;
        qr[i] = qc[i] = 0;
        qb[i] = qm[i] = clo[i] = chi[i] = 0u;
        if (q < nq) {
            qr[i] = q / qrow;
            qc[i] = q - qr[i] * qrow;
            qo[i] = (qr[i] + 1) * pw + 1 + qc[i];
            qb[i] = reinterpret_cast<const uint32_t *>(bs)[q];
            const int nv = min(4, W - 4 * qc[i]);
            qm[i] = nv >= 4 ? 0xFFFFFFFFu : (1u << (8 * nv)) - 1u;
        }
    }
    const uint32_t t0 = sweep_index(a);
    const uint32_t tag = GIBBS ? kTagGibbs : kTagPCA;
    uint32_t nre = 0u;
    int cur = 0, nacc = 0;
    // add the counts of the 16-bit lanes to the accumulator and clear them
    auto flush = [&]() {
#pragma unroll
        for (int i = 0; i < QPT; ++i) {
            if (qo[i] < 0)
                continue;
            const uint32_t cnt[4] = {clo[i] & 0xFFFFu, chi[i] & 0xFFFFu, clo[i] >> 16,
                                     chi[i] >> 16};
            float *accq = a.acc + (size_t)qr[i] * W + 4 * qc[i];
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (((qm[i] >> (8 * j)) & 1u) && cnt[j] != 0u)
                    accq[j] += (float)cnt[j];
            clo[i] = chi[i] = 0u;
        }
    };
    for (int k = 0; k < nsweeps; ++k) {
        const uint32_t t = t0 + (uint32_t)k;
        const bool acc_now = accumulate_after(a, t);
        uint32_t *X = reinterpret_cast<uint32_t *>(cur ? pl1 : pl0);
        if (!GIBBS) {
            uint32_t *Y = reinterpret_cast<uint32_t *>(cur ? pl0 : pl1);
#pragma unroll
            for (int i = 0; i < QPT; ++i) {
                if (qo[i] < 0)
                    continue;
                uint32_t u[4];
                quad_words(a, tag, t, qr[i], qc[i], u);
                uint32_t M;
                const uint32_t S = quad_counts<NB>(X, qo[i], pw, M) + qb[i];
                const uint32_t nw = quad_draw<NB>(tab, S, M, u, qm[i], nre) & qm[i];
                Y[qo[i]] = nw;
                if (acc_now) {
                    clo[i] += nw & 0x00FF00FFu;
                    chi[i] += (nw >> 8) & 0x00FF00FFu;
                }
            }
            __syncthreads();
            cur ^= 1;
        } else {
            constexpr int kColours = NB == 4 ? 2 : 4;
            uint32_t u[QPT][4];
#pragma unroll
            for (int i = 0; i < QPT; ++i)
                if (qo[i] >= 0)
                    quad_words(a, tag, t, qr[i], qc[i], u[i]);
#pragma unroll 1
            for (int ph = 0; ph < kColours; ++ph) {
#pragma unroll
                for (int i = 0; i < QPT; ++i) {
                    const uint32_t act = qo[i] < 0 ? 0u : phase_mask<NB>(qr[i], ph) & qm[i];
                    if (act == 0u)
                        continue;
                    uint32_t M;
                    const uint32_t S = quad_counts<NB>(X, qo[i], pw, M) + qb[i];
                    const uint32_t nw = quad_draw<NB>(tab, S, M, u[i], act, nre);
                    X[qo[i]] = (M & ~act) | (nw & act);
                }
                __syncthreads();
            }
            if (acc_now) {
#pragma unroll
                for (int i = 0; i < QPT; ++i) {
                    if (qo[i] < 0)
                        continue;
                    const uint32_t w = X[qo[i]];
                    clo[i] += w & 0x00FF00FFu;
                    chi[i] += (w >> 8) & 0x00FF00FFu;
                }
            }
        }
        if (acc_now && ++nacc == 0xFFFF) {   // a 16-bit lane is full
            flush();
            nacc = 0;
        }
    }
    flush();
    const uint8_t *fin = cur ? pl1 : pl0;
    for (int i = tid; i < H * W; i += kResThreads) {
        const int r = i / W, c = i - (i / W) * W;
        xg_out[(size_t)r * a.pitch + c] = fin[(r + 1) * P + 4 + c];
    }
    const uint32_t warp_re = __reduce_add_sync(0xFFFFFFFFu, nre);
    if ((tid & 31) == 0 && warp_re != 0u)
        atomicAdd(a.fp64_draws, (unsigned long long)warp_re);
}

template <int NB, bool GIBBS, int QPT>
__global__ void __launch_bounds__(kResThreads, 1)
    resident_kernel(const SweepArgs a, const uint8_t *xg_in, uint8_t *xg_out, int nsweeps)
{
    resident_run<NB, GIBBS, QPT>(a, a.m.btab, xg_in, xg_out, nsweeps);
}

// ------------------------------------------------------- one chain, 8 CTAs
// One chain alone leaves 151 SMs idle, and its sweep is bound by the issue
// slots of the one it has: 0.87 us for 64 x 64 (Gibbs 1.31), against 0.50
// (0.85) here, bound by the latency of a pass and of the exchange.  A cluster of 8 CTAs takes the
// chain in bands of rows with a halo of h rows: h sweeps (Gibbs: h colour
// phases) run on shrinking extensions of the band, then each CTA pushes its
// border rows into its neighbours' receive buffers through distributed shared
// memory and the cluster's barrier makes them visible (two buffers in turn: a
// buffer is written again only after the barrier that follows its reading).
// Draws are keyed by (sweep, site), so both owners of an extended row draw the
// same labels.  A thread keeps its quads, their base bytes, their counts and
// the next sweep's uniforms in registers.
constexpr int kClCtas = 8;
constexpr int kClHalo = 8;                // rows, at most: 8 PCA sweeps, 4 (2) Gibbs sweeps
constexpr int kClThreads = 768;           // at most

inline int cl_smem_bytes(bool gibbs, int band, int h, int W)
{
    const int Wq4 = (W + 3) & ~3;
    return kThrBytes + (gibbs ? 1 : 2) * (band + 2 * h) * (Wq4 + 8) + 4 * h * Wq4;
}

__device__ __forceinline__ uint32_t cluster_rank()
{
    uint32_t r;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release;\n\t"
                 "barrier.cluster.wait.acquire;" ::: "memory");
}

// Store v at the shared-memory word `local` of CTA `rank` of the cluster.
__device__ __forceinline__ void st_cluster(const uint32_t *local, uint32_t rank, uint32_t v)
{
    uint32_t addr;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;"
                 : "=r"(addr)
                 : "r"((uint32_t)__cvta_generic_to_shared(local)), "r"(rank));
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}

template <int NB, bool GIBBS, int QPT, int h>
__global__ void __cluster_dims__(kClCtas, 1, 1) __launch_bounds__(kClThreads, 1)
    resident_cluster_kernel(const SweepArgs a, const uint8_t *xg_in, uint8_t *xg_out, int nsweeps,
                            int band)
{
    extern __shared__ __align__(16) uint8_t sm[];
    constexpr int kCol = !GIBBS ? 1 : (NB == 4 ? 2 : 4);
    constexpr int K = h / kCol;                    // sweeps per exchange
    static_assert(K >= 1, "halo");
    const int tid = (int)threadIdx.x, nt = (int)blockDim.x;
    const int rank = (int)cluster_rank();
    const int H = a.H, W = a.W;
    const int qrow = (W + 3) >> 2, pw = qrow + 2;  // quads, words per staged row
    const int rows = band + 2 * h;                 // staged rows
    const int r0 = rank * band;                    // the band's first image row
    const int own = max(0, min(band, H - r0));     // its rows inside the image
    ThrTab<NB> &tab = *reinterpret_cast<ThrTab<NB> *>(sm);
    uint32_t *const pl0 = reinterpret_cast<uint32_t *>(sm + kThrBytes);
    uint32_t *const pl1 = GIBBS ? pl0 : pl0 + rows * pw;
    uint32_t *const recv = pl1 + rows * pw;        // [2 turns][above, below][h][qrow]
    load_thresholds<NB>(tab, a.m.btab, tid, nt);
    for (int i = tid; i < (GIBBS ? 1 : 2) * rows * pw; i += nt)
        pl0[i] = 0u;   // outside the image, and the padding of rows
    __syncthreads();
    for (int i = tid; i < rows * qrow; i += nt) {
        const int sr = i / qrow, q = i - sr * qrow, r = r0 - h + sr;
        if (r < 0 || r >= H)
            continue;
        uint32_t w = *reinterpret_cast<const uint32_t *>(xg_in + (size_t)r * a.pitch + 4 * q);
        const int nv = W - 4 * q;
        if (nv < 4)
            w &= (1u << (8 * nv)) - 1u;
        pl0[sr * pw + 1 + q] = w;
    }
    // this thread's quads: rows -(h - 1) .. band + h - 2 of the band
    int lr[QPT], qo[QPT], qc[QPT];
    uint32_t qb[QPT], qm[QPT], clo[QPT], chi[QPT], un[QPT][4];
    const int n = (band + 2 * h - 2) * qrow;
#pragma unroll
    for (int i = 0; i < QPT; ++i) {
        const int q = tid + i * nt;
        qb[i] = qm[i] = clo[i] = chi[i] = 0u;
        lr[i] = q < n ? q / qrow - (h - 1) : 1 << 20;
        qc[i] = q < n ? q % qrow : 0;
        qo[i] = (lr[i] + h) * pw + 1 + qc[i];
        const int r = r0 + lr[i];
        if (q >= n || r < 0 || r >= H) {
            lr[i] = 1 << 20;   // never active
            continue;
        }
        const uint32_t gw = *reinterpret_cast<const uint32_t *>(a.g + (size_t)r * a.pitch + 4 * qc[i]);
        const int nv = min(4, W - 4 * qc[i]);
        qm[i] = nv >= 4 ? 0xFFFFFFFFu : (1u << (8 * nv)) - 1u;
        for (int j = 0; j < nv; ++j) {
            const int c = 4 * qc[i] + j;
            int nm = (r == 0) + (r == H - 1) + (c == 0) + (c == W - 1);
            if (NB == 8)
                nm += (r == 0 || c == 0) + (r == 0 || c == W - 1) + (r == H - 1 || c == 0) +
                      (r == H - 1 || c == W - 1);
            qb[i] |= (uint32_t)(((int)((gw >> (8 * j)) & 1u) * (NB + 1) + nm) * (NB + 1)) << (8 * j);
        }
    }
    const uint32_t t0 = sweep_index(a);
    const uint32_t tag = GIBBS ? kTagGibbs : kTagPCA;
    const auto uniforms = [&](uint32_t t) {
#pragma unroll
        for (int i = 0; i < QPT; ++i)
            if (lr[i] < (1 << 20))
                quad_words(a, tag, t, r0 + lr[i], qc[i], un[i]);
    };
    uniforms(t0);
    cluster_sync();   // every CTA has read its rows: the last one may write them back
    uint32_t nre = 0u;
    int cur = 0, nacc = 0;
    // add the counts of the 16-bit lanes to the accumulator and clear them
    const auto flush = [&]() {
#pragma unroll
        for (int i = 0; i < QPT; ++i) {
            if ((unsigned)lr[i] >= (unsigned)own)
                continue;
            const uint32_t cnt[4] = {clo[i] & 0xFFFFu, chi[i] & 0xFFFFu, clo[i] >> 16,
                                     chi[i] >> 16};
            float *accq = a.acc + (size_t)(r0 + lr[i]) * W + 4 * qc[i];
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (((qm[i] >> (8 * j)) & 1u) && cnt[j] != 0u)
                    accq[j] += (float)cnt[j];
            clo[i] = chi[i] = 0u;
        }
    };
    int done = 0;
    for (unsigned int x = 0;; ++x) {               // exchanges
        const int ns = min(K, nsweeps - done);
        for (int s = 0; s < ns; ++s) {
            const uint32_t t = t0 + (uint32_t)(done + s);
            const bool acc_now = accumulate_after(a, t);
            uint32_t u[QPT][4];
#pragma unroll
            for (int i = 0; i < QPT; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    u[i][j] = un[i][j];
            uint32_t *const X = cur ? pl1 : pl0;
            uint32_t *const Y = GIBBS ? X : (cur ? pl0 : pl1);
#pragma unroll 1
            for (int ph = 0; ph < kCol; ++ph) {
                const int e = (ns - s) * kCol - 1 - ph;   // rows beyond the band, each side
#pragma unroll
                for (int i = 0; i < QPT; ++i) {
                    if ((unsigned)(lr[i] + e) >= (unsigned)(band + 2 * e))
                        continue;
                    const bool mine = (unsigned)lr[i] < (unsigned)own;
                    uint32_t act = qm[i];
                    if (GIBBS)
                        act &= phase_mask<NB>(r0 + lr[i], ph);
                    if (act == 0u)
                        continue;
                    uint32_t M;
                    const uint32_t S = quad_counts<NB>(X, qo[i], pw, M) + qb[i];
                    const uint32_t nw = quad_draw<NB>(tab, S, M, u[i], mine ? act : 0u, nre) & act;
                    Y[qo[i]] = GIBBS ? (M & ~act) | nw : nw;
                    if (acc_now && mine) {
                        clo[i] += nw & 0x00FF00FFu;
                        chi[i] += (nw >> 8) & 0x00FF00FFu;
                    }
                }
                if (ph == kCol - 1)
                    uniforms(t + 1u);   // independent of the labels: fills the pass
                __syncthreads();
            }
            if (!GIBBS)
                cur ^= 1;
            if (acc_now && ++nacc == 0xFFFF) {   // a 16-bit lane is full
                flush();
                nacc = 0;
            }
        }
        done += ns;
        if (done == nsweeps)
            break;
        uint32_t *const X = cur ? pl1 : pl0;
        uint32_t *const rv = recv + (x & 1u) * 2 * h * qrow;
        // the band's first rows go below the upper neighbour's band, its last
        // ones above the lower neighbour's (full there: only the last band of
        // the image is short)
        for (int i = tid; i < 2 * h * qrow; i += nt) {
            const int up = i < h * qrow;
            const int k = up ? i : i - h * qrow;
            const int j = k / qrow, q = k - j * qrow;
            const int row = up ? j : band - h + j;
            if (row >= own || (up ? rank == 0 : rank + 1 == kClCtas))
                continue;
            st_cluster(rv + ((up ? h : 0) + j) * qrow + q, (uint32_t)(up ? rank - 1 : rank + 1),
                       X[(row + h) * pw + 1 + q]);
        }
        cluster_sync();
        for (int i = tid; i < 2 * h * qrow; i += nt) {
            const int up = i < h * qrow;
            const int k = up ? i : i - h * qrow;
            const int j = k / qrow, q = k - j * qrow;
            const int row = up ? j - h : band + j;
            if (r0 + row >= 0 && r0 + row < H)
                X[(row + h) * pw + 1 + q] = rv[((up ? 0 : h) + j) * qrow + q];
        }
        __syncthreads();
    }
    flush();
    const uint32_t *fin = cur ? pl1 : pl0;
    for (int i = tid; i < own * qrow; i += nt) {
        const int r = i / qrow, q = i - r * qrow;
        const uint32_t w = fin[(r + h) * pw + 1 + q];
        uint8_t *out = xg_out + (size_t)(r0 + r) * a.pitch + 4 * q;
        const int nv = min(4, W - 4 * q);
        if (nv == 4)
            *reinterpret_cast<uint32_t *>(out) = w;
        else
            for (int j = 0; j < nv; ++j)
                out[j] = (uint8_t)(w >> (8 * j));
    }
    const uint32_t warp_re = __reduce_add_sync(0xFFFFFFFFu, nre);
    if ((tid & 31) == 0 && warp_re != 0u)
        atomicAdd(a.fp64_draws, (unsigned long long)warp_re);
}

// Batched chains: CTA b runs chain idx[b] (a PCA slot) with the table
// tabs + b * kBtabStride, for the sweeps t0 .. t0 + n - 1 below the slot's
// budget (t0 its device sweep counter); the planes follow the counter.
template <int NB>
__global__ void __launch_bounds__(kResThreads, 1)
    resident_batch_kernel(const SlotDesc *slots, const int *idx, const uint4 *tabs, int n)
{
    const SlotDesc &d = slots[idx[blockIdx.x]];
    if (!d.active)
        return;
    const uint32_t t0 = *d.tdev, bud = *d.budget;
    const int nb = bud > t0 ? (int)min((uint32_t)n, bud - t0) : 0;
    if (nb == 0)
        return;
    SweepArgs a;
    slot_args(d, t0, a);
    a.sweep_base = d.tdev;
    a.sweep_off = 0u;
    a.last_phase = 0;
    resident_run<NB, false, kResMaxQuadsPerThread>(a, tabs + (size_t)blockIdx.x * kBtabStride,
                                                   d.x[t0 & 1u], d.x[(t0 + (uint32_t)nb) & 1u],
                                                   nb);
}

template <int NB, bool GIBBS, int QPT>
cudaError_t launch_res_t(const SweepArgs &a, const uint8_t *x_in, uint8_t *x_out, int n,
                         cudaStream_t st)
{
    static bool attr_set[64] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess)
        return e;
    if (dev >= 64)
        return cudaErrorInvalidDevice;
    if (!attr_set[dev]) {
        e = cudaFuncSetAttribute(resident_kernel<NB, GIBBS, QPT>,
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, kResMaxSmem);
        if (e != cudaSuccess)
            return e;
        attr_set[dev] = true;
    }
    const int smem = res_smem_bytes(NB, GIBBS, a.H, a.W);
    resident_kernel<NB, GIBBS, QPT><<<1, kResThreads, smem, st>>>(a, x_in, x_out, n);
    return cudaGetLastError();
}

// Quads of a CTA of the cluster form with bands of `band` rows and a halo of h.
inline int cluster_quads(int band, int h, int W)
{
    return (band + 2 * h - 2) * ((W + 3) >> 2);
}

// Halo of the cluster form: 8 rows (64 x 64: 0.50 us per sweep, Gibbs 0.85,
// against 0.52 and 0.90 with 4, 0.67 and 1.15 with 2), 4 where the bands are
// thinner or a thread would hold more than a quad; 0: not taken (bands thinner
// than that, or few quads, which leave nothing to share).
inline int cluster_halo(int band, int H, int W)
{
    if (band < 4 || H * ((W + 3) >> 2) < 512 || cluster_quads(band, 4, W) > 2 * kClThreads)
        return 0;
    return band >= kClHalo && cluster_quads(band, kClHalo, W) <= kClThreads ? kClHalo : 4;
}

template <int NB, bool GIBBS, int QPT, int h>
cudaError_t launch_cl_t(const SweepArgs &a, const uint8_t *x_in, uint8_t *x_out, int n, int band,
                        cudaStream_t st)
{
    const int threads = ((cluster_quads(band, h, a.W) + QPT - 1) / QPT + 31) & ~31;
    const int smem = cl_smem_bytes(GIBBS, band, h, a.W);
    if (threads > kClThreads || smem > 48 * 1024)
        return cudaErrorInvalidValue;
    resident_cluster_kernel<NB, GIBBS, QPT, h>
        <<<kClCtas, threads, smem, st>>>(a, x_in, x_out, n, band);
    return cudaGetLastError();
}

template <int NB, bool GIBBS>
cudaError_t launch_res_q(const SweepArgs &a, const uint8_t *x_in, uint8_t *x_out, int n,
                         cudaStream_t st)
{
    const int nq = a.H * (((a.W + 3) & ~3) >> 2);
    const int band = (a.H + kClCtas - 1) / kClCtas, h = cluster_halo(band, a.H, a.W);
    if (h == kClHalo)
        return launch_cl_t<NB, GIBBS, 1, kClHalo>(a, x_in, x_out, n, band, st);
    if (h > 0)
        return cluster_quads(band, 4, a.W) <= kClThreads
                   ? launch_cl_t<NB, GIBBS, 1, 4>(a, x_in, x_out, n, band, st)
                   : launch_cl_t<NB, GIBBS, 2, 4>(a, x_in, x_out, n, band, st);
    if (nq <= kResThreads)
        return launch_res_t<NB, GIBBS, 1>(a, x_in, x_out, n, st);
    if (nq <= 2 * kResThreads)
        return launch_res_t<NB, GIBBS, 2>(a, x_in, x_out, n, st);
    return launch_res_t<NB, GIBBS, kResMaxQuadsPerThread>(a, x_in, x_out, n, st);
}

// ------------------------------------------------------- large images
// Two labels on images too large for one CTA: one launch per sweep with the
// same thresholds.  A warp owns a strip of 32 quads (128 columns) and walks
// down its rows, a lane per quad: the label words above, at and below the row
// stay in registers, the words left and right come from the neighbouring
// lanes (lanes 0 and 31 load the strip's outer words), so labels need one
// load per quad and no shared memory.  Neighbour counts by byte-wise adds, one
// Philox call, four threshold reads and compares, one 32-bit label store.
// Sums: a float4 per lane where rows of the accumulator are aligned, else the
// warp's 128 sums as four coalesced words per lane (the labels by shuffles).
// The next row's words are loaded before a row's draws.
//
// Bound by instruction issue (about 58 per site) at 0.55 of the memory rate:
// 8192^2 151 us per sweep (4.44e11 site-updates/s) against 203 us for the
// form that staged tiles of labels in shared memory and read a 16-byte entry
// per draw; 2043 x 3001 17.9 us against 22.7.  256 threads at 75 registers (3
// blocks per SM): held to 5 blocks 157 us and 21.6.
constexpr int kBinThreads = 256;
constexpr int kBinMaxRows = 16;            // rows per strip, at most
constexpr int kBinQW = 32;                 // quads per strip

// Planes: a.xin -> a.xout, or (x0 != nullptr) x0 / x1 holding the states of
// even / odd sweep indices; budget (optional): a sweep with index >= *budget
// is skipped (a chain of a batch or of the server).
template <int NB>
__global__ void __launch_bounds__(kBinThreads)
    pca_binary_kernel(const SweepArgs a, int strips_x, int nstrips, int rows, int acc_vec, uint8_t *x0,
                      uint8_t *x1, const uint32_t *budget)
{
    __shared__ ThrTab<NB> tab;
    grid_dep_launch();
    grid_dep_wait();
    const uint32_t t = sweep_index(a);
    if (budget && t >= *budget)
        return;   // the whole launch, before any barrier
    const uint8_t *xin = x0 ? ((t & 1u) ? x1 : x0) : a.xin;
    uint8_t *xout = x0 ? ((t & 1u) ? x0 : x1) : a.xout;
    load_thresholds<NB>(tab, a.m.btab, (int)threadIdx.x, kBinThreads);
    const bool acc_on = accumulate_after(a, t);
    const int H = a.H, W = a.W, pitch = a.pitch;
    const int Wq = (W + 3) >> 2;
    const int lane = (int)threadIdx.x & 31;
    uint32_t nre = 0u;
    for (int strip = (int)(blockIdx.x * (kBinThreads / 32) + (threadIdx.x >> 5)); strip < nstrips;
         strip += (int)gridDim.x * (kBinThreads / 32)) {
        const int sy = strip / strips_x, sx = strip - sy * strips_x;
        const int r0 = sy * rows, q = sx * kBinQW + lane;
        const int r1 = min(r0 + rows, H);
        const int nv = min(4, W - 4 * q);                 // sites of the quad inside
        const uint32_t act = nv >= 4 ? 0xFFFFFFFFu : (nv > 0 ? (1u << (8 * nv)) - 1u : 0u);
        // lanes 0 and 31 also read the word outside the strip.  Loads are
        // unconditional, at clamped rows and quads, and masked.
        const int qe = lane == 0 ? q - 1 : (lane == 31 ? q + 1 : q);
        const uint32_t acte = qe >= 0 && qe < Wq
                                  ? (W - 4 * qe >= 4 ? 0xFFFFFFFFu : (1u << (8 * (W - 4 * qe))) - 1u)
                                  : 0u;
        const int qc = min(q, Wq - 1), qec = min(max(qe, 0), Wq - 1);
        const auto row_at = [&](int r) -> const uint8_t * {
            return xin + (size_t)min(max(r, 0), H - 1) * pitch;
        };
        const auto ld = [](const uint8_t *p, int qq) -> uint32_t {
            return *reinterpret_cast<const uint32_t *>(p + 4 * qq);
        };
        // the sums left + right of the 4 sites of word w (outer word e)
        const auto sides = [&](uint32_t w, uint32_t e) -> uint32_t {
            uint32_t l = __shfl_up_sync(0xFFFFFFFFu, w, 1), rr = __shfl_down_sync(0xFFFFFFFFu, w, 1);
            l = lane == 0 ? e : l;
            rr = lane == 31 ? e : rr;
            return __funnelshift_l(l, w, 8) + __funnelshift_r(w, rr, 8);
        };
        const bool side = nv > 0 && (q == 0 || 4 * q + 4 >= W);   // a column has a missing side
        const uint8_t *pu = row_at(r0 - 1), *p0 = row_at(r0), *p1 = row_at(r0 + 1);
        uint32_t up = r0 > 0 ? ld(pu, qc) & act : 0u, M = ld(p0, qc) & act;
        uint32_t dn = r0 + 1 < H ? ld(p1, qc) & act : 0u, dne = r0 + 1 < H ? ld(p1, qec) & acte : 0u;
        uint32_t upS = 0u, Ms = sides(M, ld(p0, qec) & acte);
        if (NB == 8)
            upS = sides(up, r0 > 0 ? ld(pu, qec) & acte : 0u);
        const uint8_t *pg = a.g + (size_t)r0 * pitch;
        const uint8_t *p2 = row_at(r0 + 2);
        uint8_t *po = xout + (size_t)r0 * pitch + 4 * q;
        float *pa = a.acc + (size_t)r0 * W + 4 * kBinQW * sx;
        const int left = W - 4 * kBinQW * sx;             // columns of the strip inside
        uint32_t gw = ld(pg, qc);
        for (int r = r0; r < r1; ++r) {
            // in flight during the draws: the row after next, the next
            // observations, this row's sums
            const uint32_t m2 = r + 2 < H ? 0xFFFFFFFFu : 0u;
            const uint32_t dn2 = ld(p2, qc) & act & m2, dne2 = ld(p2, qec) & acte & m2;
            p2 += r + 3 < H ? pitch : 0;
            pg += r + 1 < H ? pitch : 0;
            const uint32_t gw2 = ld(pg, qc);
            float4 A4 = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            if (acc_on) {
                if (acc_vec) {
                    if (nv >= 4)
                        A4 = *reinterpret_cast<const float4 *>(pa + 4 * lane);
                } else {
                    A4.x = lane < left ? pa[lane] : 0.0f;
                    A4.y = 32 + lane < left ? pa[32 + lane] : 0.0f;
                    A4.z = 64 + lane < left ? pa[64 + lane] : 0.0f;
                    A4.w = 96 + lane < left ? pa[96 + lane] : 0.0f;
                }
            }
            const uint32_t dnS = sides(dn, dne);
            uint32_t S = up + dn + Ms;
            if (NB == 8)
                S += upS + dnS;
            S += (gw & act & 0x01010101u) * (uint32_t)((NB + 1) * (NB + 1));
            if (r == 0 || r == H - 1 || side) {
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int c = 4 * q + j;
                    int nm = (r == 0) + (r == H - 1) + (c == 0) + (c == W - 1);
                    if (NB == 8)
                        nm += (r == 0 || c == 0) + (r == 0 || c == W - 1) +
                              (r == H - 1 || c == 0) + (r == H - 1 || c == W - 1);
                    S += (uint32_t)(nm * (NB + 1)) << (8 * j);
                }
            }
            uint32_t u[4];
            quad_words(a, kTagPCA, t, r, q, u);
            const uint32_t nw = quad_draw<NB>(tab, S, M, u, act, nre) & act;
            if (nv >= 4) {
                *reinterpret_cast<uint32_t *>(po) = nw;
            } else {
                for (int j = 0; j < nv; ++j)
                    po[j] = (uint8_t)(nw >> (8 * j));
            }
            po += pitch;
            if (acc_on) {
                // a byte to a float: in the mantissa of 2^23, less 2^23
                const auto fl = [](uint32_t w, uint32_t sel) {
                    return __fadd_rn(__uint_as_float(__byte_perm(w, 0x4B000000u, sel)), -8388608.0f);
                };
                if (acc_vec) {
                    if (nv >= 4)
                        *reinterpret_cast<float4 *>(pa + 4 * lane) =
                            make_float4(A4.x + fl(nw, 0x7440u), A4.y + fl(nw, 0x7441u),
                                        A4.z + fl(nw, 0x7442u), A4.w + fl(nw, 0x7443u));
                } else {
                    const float old[4] = {A4.x, A4.y, A4.z, A4.w};
                    const uint32_t sel = 0x7440u + (uint32_t)(lane & 3);
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const int c = 32 * j + lane;
                        const uint32_t w = __shfl_sync(0xFFFFFFFFu, nw, 8 * j + (lane >> 2));
                        if (c < left)
                            pa[c] = old[j] + fl(w, sel);
                    }
                }
            }
            pa += W;
            up = M;
            upS = Ms;
            M = dn;
            Ms = dnS;
            dn = dn2;
            dne = dne2;
            gw = gw2;
        }
    }
    const uint32_t warp_re = __reduce_add_sync(0xFFFFFFFFu, nre);
    if (lane == 0 && warp_re != 0u)
        atomicAdd(a.fp64_draws, (unsigned long long)warp_re);
}

template <int NB>
cudaError_t launch_binary_t(const SweepArgs &a, uint8_t *x0, uint8_t *x1, const uint32_t *budget,
                            cudaStream_t st)
{
    static int per_sm[64] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess)
        return e;
    if (dev >= 64)
        return cudaErrorInvalidDevice;
    if (per_sm[dev] == 0) {
        int n = 0;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, pca_binary_kernel<NB>, kBinThreads,
                                                          0);
        if (e != cudaSuccess)
            return e;
        per_sm[dev] = n > 0 ? n : 1;
    }
    int sms = 0;
    e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess)
        return e;
    const int Wq = (a.W + 3) >> 2;
    const int strips_x = (Wq + kBinQW - 1) / kBinQW;
    if (a.H <= 0 || strips_x <= 0)
        return cudaSuccess;
    constexpr int per = kBinThreads / 32;
    const long long cap = (long long)per_sm[dev] * sms;
    // rows per strip: whole waves of the resident warps (8 rows at 2043 x 3001
    // left a quarter of a second wave)
    const long long all = (long long)a.H * strips_x, warps = cap * per;
    const long long waves = (all + warps * kBinMaxRows - 1) / (warps * kBinMaxRows);
    const int rows = (int)((all + warps * waves - 1) / (warps * waves));
    const long long nstrips = (long long)strips_x * ((a.H + rows - 1) / rows);
    if (nstrips >= (1ll << 30))
        return cudaErrorInvalidValue;
    const long long need = (nstrips + per - 1) / per;
    const int grid = (int)(need < cap ? need : cap);
    const int acc_vec = (a.W % 4 == 0 && (reinterpret_cast<uintptr_t>(a.acc) & 15u) == 0) ? 1 : 0;
    return launch_dependent(pca_binary_kernel<NB>, grid, kBinThreads, st, a, strips_x, (int)nstrips,
                            rows, acc_vec, x0, x1, budget);
}

}  // namespace

int btab_bytes()
{
    return kBtabStride * 16;
}

cudaError_t launch_btab(const DevModel &m, uint4 *out, cudaStream_t st)
{
    const BtabJob j{m, out};
    return launch_btabs(&j, 1, st);
}

cudaError_t launch_btabs(const BtabJob *jobs, int n, cudaStream_t st)
{
    for (int i = 0; i < n; ++i)
        if (jobs[i].m.L != 2 || (jobs[i].m.nbhd != 4 && jobs[i].m.nbhd != 8))
            return cudaErrorInvalidValue;
    for (int nb = 4; nb <= 8; nb += 4) {
        const int ne = nb == 8 ? btab_entries<8>() : btab_entries<4>();
        const int grid = (ne + 7) / 8;   // 8 warps per block, one per configuration
        constexpr int kMost = 64;
        BtabJobs<kMost> many;
        int k = 0;
        for (int i = 0; i < n; ++i) {
            if (jobs[i].m.nbhd == nb)
                many.job[k++] = jobs[i];
            if (k == 0 || (k < kMost && i + 1 < n))
                continue;
            if (k == 1) {
                const BtabJobs<1> one{{many.job[0]}};
                if (nb == 8)
                    btab_kernel<8, 1><<<grid, 256, 0, st>>>(one);
                else
                    btab_kernel<4, 1><<<grid, 256, 0, st>>>(one);
            } else if (nb == 8) {
                btab_kernel<8, kMost><<<dim3(grid, k), 256, 0, st>>>(many);
            } else {
                btab_kernel<4, kMost><<<dim3(grid, k), 256, 0, st>>>(many);
            }
            k = 0;
        }
    }
    return cudaGetLastError();
}

bool resident_fits(int L, int nbhd, int H, int W)
{
    if (L != 2 || (nbhd != 4 && nbhd != 8))
        return false;
    if ((long long)H * (((W + 3) & ~3) >> 2) > (long long)kResMaxQuadsPerThread * kResThreads)
        return false;
    return res_smem_bytes(nbhd, false, H, W) <= kResMaxSmem;
}

int resident_smem_bytes(int nbhd, int H, int W)
{
    return res_smem_bytes(nbhd, false, H, W);
}

cudaError_t launch_resident_batch(const SlotDesc *slots, const int *idx, const uint4 *tabs,
                                  int count, int nbhd, int n, int smem, cudaStream_t st)
{
    if (count <= 0 || n <= 0)
        return cudaSuccess;
    if ((nbhd != 4 && nbhd != 8) || smem > kResMaxSmem)
        return cudaErrorInvalidValue;
    static bool attr_set[2][64] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess)
        return e;
    if (dev >= 64)
        return cudaErrorInvalidDevice;
    const int k = nbhd == 8 ? 1 : 0;
    if (!attr_set[k][dev]) {
        e = nbhd == 8 ? cudaFuncSetAttribute(resident_batch_kernel<8>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             kResMaxSmem)
                      : cudaFuncSetAttribute(resident_batch_kernel<4>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             kResMaxSmem);
        if (e != cudaSuccess)
            return e;
        attr_set[k][dev] = true;
    }
    if (nbhd == 8)
        resident_batch_kernel<8><<<count, kResThreads, smem, st>>>(slots, idx, tabs, n);
    else
        resident_batch_kernel<4><<<count, kResThreads, smem, st>>>(slots, idx, tabs, n);
    return cudaGetLastError();
}

bool resident_eligible(const DevModel &m, int H, int W)
{
    if (m.L != 2 || m.norm != 0 || (m.nbhd != 4 && m.nbhd != 8) || m.btab == nullptr)
        return false;
    if ((long long)H * (((W + 3) & ~3) >> 2) > (long long)kResMaxQuadsPerThread * kResThreads)
        return false;
    return res_smem_bytes(m.nbhd, false, H, W) <= kResMaxSmem;
}

cudaError_t launch_resident(const SweepArgs &a, const uint8_t *x_in, uint8_t *x_out, int nsweeps,
                            bool gibbs, cudaStream_t st)
{
    if (!resident_eligible(a.m, a.H, a.W) || nsweeps < 0)
        return cudaErrorInvalidValue;
    if (nsweeps == 0)
        return cudaSuccess;
    if (a.m.nbhd == 8)
        return gibbs ? launch_res_q<8, true>(a, x_in, x_out, nsweeps, st)
                     : launch_res_q<8, false>(a, x_in, x_out, nsweeps, st);
    return gibbs ? launch_res_q<4, true>(a, x_in, x_out, nsweeps, st)
                 : launch_res_q<4, false>(a, x_in, x_out, nsweeps, st);
}

bool binary_eligible(const DevModel &m)
{
    return m.L == 2 && m.norm == 0 && (m.nbhd == 4 || m.nbhd == 8) && m.btab != nullptr;
}

cudaError_t launch_pca_binary(const SweepArgs &a, cudaStream_t st, uint8_t *x0, uint8_t *x1,
                              const uint32_t *budget)
{
    if (!binary_eligible(a.m))
        return cudaErrorInvalidValue;
    // word loads and stores of the planes
    const uintptr_t planes = x0 ? (reinterpret_cast<uintptr_t>(x0) | reinterpret_cast<uintptr_t>(x1))
                                : (reinterpret_cast<uintptr_t>(a.xin) |
                                   reinterpret_cast<uintptr_t>(a.xout));
    if ((a.pitch & 3) != 0 || ((planes | reinterpret_cast<uintptr_t>(a.g)) & 3u) != 0)
        return cudaErrorMisalignedAddress;
    return a.m.nbhd == 8 ? launch_binary_t<8>(a, x0, x1, budget, st)
                         : launch_binary_t<4>(a, x0, x1, budget, st);
}

}  // namespace pcad
