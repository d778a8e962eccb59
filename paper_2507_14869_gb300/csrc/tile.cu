// Tile-resident sweeps: images of a few hundred to a few thousand sites per
// SM, whole runs in one cooperative launch (lazy PCA, Section 5.2;
// checkerboard Gibbs, Section 5.1).
//
// A sweep of such an image is shorter than what one launch per sweep costs
// around it: at 256^2, 9 labels and 8 neighbours, the per-sweep small-label
// kernel took 6.3 us per sweep (launch gap, tables, tile staging, four draws
// in a row per thread) and a Gibbs sweep 11.4 us (four launches), for draws
// that fill the SMs' issue slots for 0.5 us.  Here every CTA owns one tile for
// all sweeps of a run: labels, observation, accumulator and tables stay in
// shared memory, and only tile borders travel.
//
//   * Exchange.  Every k sweeps the tile's border words (4 labels) go to an
//     exchange buffer in global memory as 64-bit stores of (labels, tag = the
//     number of sweeps done), and the neighbours' threads poll exactly the
//     words of their halo until the tag is the awaited one: data and flag are
//     one relaxed 64-bit access, so an exchange is one store-to-load trip
//     through L2 and needs no fence.  Two buffers, used in turn, suffice: a
//     tile writes exchange e + 2 only after its neighbours' words of e + 1
//     arrived, which they published after reading this tile's words of e.
//     Tags only grow between two resets of a chain; the buffers are cleared at
//     creation and at a reset.
//   * k sweeps per exchange.  The halo is h = k sites wide (Gibbs: k times the
//     2 or 4 colour phases of a sweep); a sweep (phase) with e more to come
//     before the next exchange also updates the sites up to e beyond the tile.
//     Draws are keyed by (sweep, site), so every owner of such a site draws
//     the same label.  k trades draws for exchanges (tile_geometry).
//   * The uniforms of the next k sweeps are computed while the border words
//     travel.
//   * Lazy PCA on larger tiles draws whole words: a thread takes the 4 sites of
//     a word (words of labels, observations and uniforms; four draws in
//     flight) instead of one site.  Small tiles keep one site per thread: the
//     latency of a pass counts there, not its instructions.
//   * Two-label tiles above 8192 sites are compact: uniforms drawn in the pass
//     instead of staged, sums as bytes (written back every 255 sweeps), so that
//     an image of 8 megapixels fits the SMs' shared memory.  2043 x 3001: 13.1 us
//     per sweep (4.7e11 site-updates/s, bound by instruction issue) against
//     17.7 with a launch per sweep.
//   * A launch holds one chain, or (batches, the server) several small ones,
//     each on CTAs of its own.
//
// The draws are the other kernels': the small-label draw, the segment draw and
// the two-label threshold table.  The CTAs wait on one another, so the launch is cooperative (all resident);
// every poll is bounded (elapsed time, or another wait's error flag).
// Measured times stand at uses_tile in capi.cu.
#include <algorithm>
#include <type_traits>

#include "async_ptx.cuh"
#include "binary_draw.cuh"
#include "seg_draw.cuh"
#include "small_draw.cuh"
#include "tile.h"

namespace pcad {

namespace {

using namespace sld;
using namespace bind;

// Threads of a CTA, two or (at most) one per SM: 64 registers, or 80 for the
// draws that need them (words, segments: spilled at 64; but a Gibbs phase of
// segment draws gains more from one round of 1024 threads: 512^2 13.0 us
// per sweep against 13.5).
constexpr int kTlThreads = 512, kTlThreads1 = 1024;
constexpr int kTlWideThreads = 384, kTlWideThreads1 = 768;
constexpr int kTlMaxSites = 8192;      // sites per tile, if it is not compact
constexpr int kTlMaxSweeps = 4;        // sweeps per exchange
constexpr int kTlMaxSmem = 224 * 1024;    // one CTA per SM
constexpr int kTlMaxSmem2 = 112 * 1024;   // two

__device__ __forceinline__ unsigned long long ld_word(const unsigned long long *p)
{
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void st_word(unsigned long long *p, unsigned long long v)
{
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// The labels of an exchange word once its tag is `tag`; false when the wait
// ran out or another wait of the launch did.
__device__ __forceinline__ bool poll_word(const unsigned long long *p, uint32_t tag, uint32_t &w,
                                          const int *err, long long limit_ns)
{
    unsigned long long v = ld_word(p);
    if ((uint32_t)(v >> 32) != tag) {
        const unsigned long long t0 = globaltimer_ns();
        for (unsigned int i = 1; (uint32_t)((v = ld_word(p)) >> 32) != tag; ++i)
            if ((i & 63u) == 0u &&
                (ld_flag(err) != 0 || (long long)(globaltimer_ns() - t0) > limit_ns))
                return false;
    }
    w = (uint32_t)v;
    return true;
}

// Colour phases of a sweep.
__host__ __device__ constexpr int tile_phases(int nb, bool gibbs)
{
    return !gibbs ? 1 : (nb == 4 ? 2 : 4);
}

// ------------------------------------------------------------------- draws
// A draw policy: kFill, the staged word outside the image; kTabBytes of
// shared tables and kRowBytes of shared scratch per thread; load() fills the
// tables; draw(), called by all lanes of a warp, returns the new label of the
// site at `me` (rows of SB bytes) at image position (r, c).  Re-draws in FP64
// are counted for sites of the tile itself (own).

template <int LMAX, int NB_, bool MASK>
struct SmallPol {
    static constexpr int NB = NB_;
    static constexpr uint32_t kFill = 0x10101010u;   // code 16: missing
    static constexpr int kTabBytes = kPtabWords * 4 + 16 * kAqStride * 4;
    static constexpr int kRowBytes = kPrefixStride * 4;
    static constexpr double kNsSite = NB == 8 ? 1.6 : 1.4;   // one SM's time per draw (ns)
    static constexpr bool kWide = false;
    static constexpr bool kWords = true;                     // draw4()
    // words per tile from which it is used: 512^2 on 216-word tiles 4.3 us per
    // sweep against 4.6, 300^2 on 150 2.6 against 2.45
    static constexpr int kWordsMin = 192;
    static constexpr bool kCompact = false;
    static constexpr double kNsSiteWords = NB == 8 ? 1.5 : 1.3;
    uint32_t *pt;
    float *aq, *pre;

    __device__ __forceinline__ void load(const DevModel &m, uint8_t *tab, uint8_t *row, int tid, int nt)
    {
        pt = reinterpret_cast<uint32_t *>(tab);
        aq = reinterpret_cast<float *>(tab + kPtabWords * 4);
        pre = reinterpret_cast<float *>(row);
        for (int i = tid; i < kPtabWords / 4; i += nt)
            reinterpret_cast<uint4 *>(pt)[i] = __ldg(reinterpret_cast<const uint4 *>(m.ptab) + i);
        fill_aq(m, aq, tid, nt);
    }

    __device__ __forceinline__ int draw(const SweepArgs &a, const uint8_t *me, int SB, int g,
                                        uint32_t ub, int, int, bool valid, bool own)
    {
        int nc[NB], xi = 0, s = 0;
        bool certain = true;
        if (valid) {
            nc[0] = me[-SB];
            nc[1] = me[SB];
            nc[2] = me[-1];
            nc[3] = me[1];
            if constexpr (NB == 8) {
                nc[4] = me[-SB - 1];
                nc[5] = me[-SB + 1];
                nc[6] = me[SB - 1];
                nc[7] = me[SB + 1];
            }
            xi = me[0];
            s = draw_small<LMAX, NB, MASK>(a.m, pt, nc, g, xi, ub, pre, certain, aq);
        }
        if (__any_sync(0xFFFFFFFFu, valid && !certain)) {
            SiteIn<NB> in{};
            in.g = g;
            in.xi = xi;
            in.ub = ub;
#pragma unroll
            for (int j = 0; j < NB; ++j)
                in.xni[j] = valid && nc[j] != 16 ? nc[j] : kMissingLabelI;
            s = warp_redraw_fp64<NB>(a.m, valid && !certain, in, s, a.fp64_draws, own);
        }
        return s;
    }
    // The new labels of word o (4 sites in a row) of the staged plane X: those
    // of the bytes of `act`, fill elsewhere; u: the word's Philox words.
    __device__ __forceinline__ uint32_t draw4(const SweepArgs &a, const uint32_t *X, int o, int SW,
                                              uint32_t G, const uint4 &u, uint32_t act, int, int,
                                              bool own)
    {
        const uint8_t *me = reinterpret_cast<const uint8_t *>(X + o);
        const int SB = 4 * SW;
        const uint32_t M = X[o], Up = X[o - SW], Dn = X[o + SW];
        const uint32_t Le = __byte_perm(M, me[-1], 0x2104), Ri = __byte_perm(M, me[4], 0x4321);
        uint32_t UL = 0u, UR = 0u, DL = 0u, DR = 0u;
        if constexpr (NB == 8) {
            UL = __byte_perm(Up, me[-SB - 1], 0x2104);
            UR = __byte_perm(Up, me[-SB + 4], 0x4321);
            DL = __byte_perm(Dn, me[SB - 1], 0x2104);
            DR = __byte_perm(Dn, me[SB + 4], 0x4321);
        }
        uint32_t packed = kFill;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const auto at = [&](uint32_t w) { return (int)((w >> (8 * q)) & 0xFFu); };
            int nc[NB];
            nc[0] = at(Up);
            nc[1] = at(Dn);
            nc[2] = at(Le);
            nc[3] = at(Ri);
            if constexpr (NB == 8) {
                nc[4] = at(UL);
                nc[5] = at(UR);
                nc[6] = at(DL);
                nc[7] = at(DR);
            }
            const bool valid = ((act >> (8 * q)) & 1u) != 0u;
            const uint32_t ub = (q == 0 ? u.x : (q == 1 ? u.y : (q == 2 ? u.z : u.w))) >> 8;
            int s = 16;
            bool certain = true;
            if (valid)
                s = draw_small<LMAX, NB, MASK>(a.m, pt, nc, at(G), at(M), ub, pre, certain, aq);
            if (__any_sync(0xFFFFFFFFu, !certain)) {
                SiteIn<NB> in{};
                in.g = at(G);
                in.xi = at(M);
                in.ub = ub;
#pragma unroll
                for (int j = 0; j < NB; ++j)
                    in.xni[j] = nc[j] != 16 ? nc[j] : kMissingLabelI;
                s = warp_redraw_fp64<NB>(a.m, !certain, in, s, a.fp64_draws, own);
            }
            packed ^= (uint32_t)(s ^ 16) << (8 * q);
        }
        return packed;
    }
    __device__ __forceinline__ void finish(const SweepArgs &) {}
};

struct SegPol {
    static constexpr int NB = 4;
    static constexpr uint32_t kFill = 0u;
    static constexpr int kTabBytes = seg::kSegFloats * 4;
    static constexpr int kRowBytes = 0;
    static constexpr double kNsSite = 4.5, kNsSiteWords = 4.5;
    static constexpr bool kWords = false, kCompact = false;
    static constexpr bool kWide = true;   // 80 registers
    float *tab;

    __device__ __forceinline__ void load(const DevModel &m, uint8_t *t, uint8_t *, int tid, int nt)
    {
        tab = reinterpret_cast<float *>(t);
        for (int i = tid; i < seg::kSegFloats / 4; i += nt)
            reinterpret_cast<float4 *>(tab)[i] =
                __ldg(reinterpret_cast<const float4 *>(m.stab) + i);
    }

    __device__ __forceinline__ int draw(const SweepArgs &a, const uint8_t *me, int SB, int g,
                                        uint32_t ub, int r, int c, bool valid, bool own)
    {
        SiteIn<4> in{};
        bool certain = true;
        int s = 0;
        if (valid) {
            in.g = g;
            in.xi = me[0];
            in.ub = ub;
            in.xni[0] = r > 0 ? (int)me[-SB] : kMissingLabelI;
            in.xni[1] = r + 1 < a.H ? (int)me[SB] : kMissingLabelI;
            in.xni[2] = c > 0 ? (int)me[-1] : kMissingLabelI;
            in.xni[3] = c + 1 < a.W ? (int)me[1] : kMissingLabelI;
            s = seg::draw_seg(a.m, tab, in, certain);
        }
        return warp_redraw_fp64<4>(a.m, valid && !certain, in, s, a.fp64_draws, own);
    }
    __device__ __forceinline__ void finish(const SweepArgs &) {}
};

template <int NB_>
struct BinPol {
    static constexpr int NB = NB_;
    static constexpr uint32_t kFill = 0u;   // a missing neighbour is no label-1 neighbour
    static constexpr int kTabBytes = kThrBytes;
    static constexpr int kRowBytes = 0;
    static constexpr double kNsSite = 0.5;
    static constexpr bool kWide = false;
    static constexpr bool kWords = true;
    static constexpr int kWordsMin = 32;   // 300^2 1.0 us against 1.3, 1000^2 3.7 against 5.6
    static constexpr double kNsSiteWords = 0.25;
    static constexpr bool kCompact = true;
    ThrTab<NB> *tab;
    uint32_t nre;

    __device__ __forceinline__ void load(const DevModel &m, uint8_t *t, uint8_t *, int tid, int nt)
    {
        tab = reinterpret_cast<ThrTab<NB> *>(t);
        load_thresholds<NB>(*tab, m.btab, tid, nt);
        nre = 0u;
    }

    __device__ __forceinline__ int draw(const SweepArgs &a, const uint8_t *me, int SB, int g,
                                        uint32_t ub, int r, int c, bool valid, bool own)
    {
        if (!valid)
            return 0;
        int n1 = me[-SB] + me[SB] + me[-1] + me[1];
        const int top = r == 0, bot = r + 1 == a.H, le = c == 0, ri = c + 1 == a.W;
        int nm = top + bot + le + ri;
        if constexpr (NB == 8) {
            n1 += me[-SB - 1] + me[-SB + 1] + me[SB - 1] + me[SB + 1];
            nm += (top | le) + (top | ri) + (bot | le) + (bot | ri);
        }
        const uint4 e = tab->full[((g * (NB + 1) + nm) * (NB + 1) + n1) * 2 + me[0]];
        nre += own && ub - e.y < e.z ? 1u : 0u;
        return ub >= e.x ? 1 : 0;
    }
    __device__ __forceinline__ uint32_t draw4(const SweepArgs &a, const uint32_t *X, int o, int SW,
                                              uint32_t G, const uint4 &u, uint32_t act, int r, int c,
                                              bool own)
    {
        const uint32_t M = X[o], U = X[o - SW], D = X[o + SW];
        uint32_t S = U + D + __funnelshift_l(X[o - 1], M, 8) + __funnelshift_r(M, X[o + 1], 8);
        if constexpr (NB == 8)
            S += __funnelshift_l(X[o - SW - 1], U, 8) + __funnelshift_r(U, X[o - SW + 1], 8) +
                 __funnelshift_l(X[o + SW - 1], D, 8) + __funnelshift_r(D, X[o + SW + 1], 8);
        S += G * (uint32_t)((NB + 1) * (NB + 1));
        const bool top = r == 0, bot = r + 1 == a.H;
        if (top || bot || c == 0 || c + 4 >= a.W) {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int le = c + q == 0, ri = c + q + 1 == a.W;
                int nm = top + bot + le + ri;
                if constexpr (NB == 8)
                    nm += (top | le) + (top | ri) + (bot | le) + (bot | ri);
                S += (uint32_t)(nm * (NB + 1)) << (8 * q);
            }
        }
        const uint32_t w[4] = {u.x, u.y, u.z, u.w};
        return quad_draw<NB>(*tab, S, M, w, own ? act : 0u, nre) & act;
    }
    __device__ __forceinline__ void finish(const SweepArgs &a)
    {
        const uint32_t n = __reduce_add_sync(0xFFFFFFFFu, nre);
        if ((threadIdx.x & 31u) == 0u && n != 0u)
            atomicAdd(a.fp64_draws, (unsigned long long)n);
    }
};

template <class P, bool GIBBS>
__host__ __device__ constexpr int tile_threads(bool two)
{
    return P::kWide && !GIBBS ? (two ? kTlWideThreads : kTlWideThreads1)
                              : (two ? kTlThreads : kTlThreads1);
}

// Words of a staged plane: what follows is 16-byte aligned, and a zero word lies
// before and behind each (draws of whole words read the words around theirs; a
// byte-wise sum must not carry from an undefined one).
__host__ __device__ constexpr int tile_plane(int words)
{
    return (words + 4) & ~3;
}

// Shared memory of a tile (bytes), in the order of the kernel's pointers:
// tables, thread scratch, uniforms of k sweeps, label planes, observation,
// counts.
template <class P, bool GIBBS>
size_t tile_smem(const TileGeom &tg, int nt)
{
    const size_t words = (size_t)(tg.th + 2 * tg.h) * (tg.twq + 2 * tg.hq);
    const size_t plane = tile_plane((int)words) * 4;
    return (size_t)P::kTabBytes + (size_t)nt * P::kRowBytes +
           (tg.compact ? 0 : words * 16 * tg.k) + 16 + plane * (GIBBS ? 1 : 2) + plane +
           (size_t)tg.th * tg.twq * (tg.compact ? 4 : 16);
}

// WORDS (lazy PCA): a thread draws the 4 sites of a word (large tiles), else
// one site.
template <class P, bool GIBBS, int JOBS, bool WORDS>
__global__ void __launch_bounds__(WORDS ? kTlWideThreads1 : tile_threads<P, GIBBS>(false), 1)
    tile_kernel(const __grid_constant__ TileLaunchT<JOBS> L)
{
    constexpr bool MULTI = JOBS > 1;
    extern __shared__ __align__(16) uint8_t sm[];
    constexpr int NB = P::NB;
    constexpr int kCol = tile_phases(NB, GIBBS);
    int j = 0;
    if (MULTI)
        while (j + 1 < L.njobs && (int)blockIdx.x >= L.job[j + 1].cta0)
            ++j;
    const TileJob &J = L.job[MULTI ? j : 0];
    const SweepArgs &a = J.a;
    int *const err = L.err;
    const int cta = (int)blockIdx.x - (MULTI ? J.cta0 : 0);
    const int tid = (int)threadIdx.x, nt = (int)blockDim.x;
    const int TH = J.tg.th, TWq = J.tg.twq, TW = 4 * TWq;
    const int h = J.tg.h, hq = J.tg.hq, hb = 4 * hq;  // halo: rows, words, columns
    const int SW = TWq + 2 * hq, SB = 4 * SW;         // words and bytes per staged row
    const int words = (TH + 2 * h) * SW;
    const int H = a.H, W = a.W, Wq = (W + 3) >> 2;
    const int ty = cta / J.tg.tiles_x, tx = cta - ty * J.tg.tiles_x;
    const int r0 = ty * TH, q0 = tx * TWq, c0 = 4 * q0;
    const uint32_t t0 = sweep_index(a);
    int nsweeps = L.nsweeps;
    if (J.budget) {   // a slot runs up to its budget (the same for all its CTAs)
        const uint32_t b = *J.budget;
        nsweeps = b > t0 ? (int)min((uint32_t)nsweeps, b - t0) : 0;
    }
    if (nsweeps == 0)
        return;
    // planes: in and out, or those of even and odd sweep indices
    const uint8_t *xg_in = J.par_from_t && (t0 & 1u) ? J.x1 : J.x0;
    uint8_t *xg_out = J.par_from_t ? (((t0 + (uint32_t)nsweeps) & 1u) ? J.x1 : J.x0) : J.x1;

    uint8_t *const row = sm + P::kTabBytes + tid * P::kRowBytes;
    uint32_t *U = reinterpret_cast<uint32_t *>(sm + P::kTabBytes + nt * P::kRowBytes);
    const bool compact = WORDS && P::kCompact && J.tg.compact;
    uint32_t *pl0 = U + (compact ? 0 : 4 * words * J.tg.k) + 4;
    const int plane = tile_plane(words);
    uint32_t *pl1 = GIBBS ? pl0 : pl0 + plane;
    uint32_t *gw = pl1 + plane;
    uint32_t *cnt = gw + plane;   // [TH][TW] label sums of this launch (compact: as bytes)
    P pol;
    pol.load(a.m, sm, row, tid, nt);
    // labels and observation with the halo
    for (int i = tid; i < words; i += nt) {
        const int sr = i / SW, sq = i - sr * SW;
        const int r = r0 - h + sr, q = q0 - hq + sq;
        uint32_t x = P::kFill, g = 0u;
        if (r >= 0 && r < H && q >= 0 && q < Wq) {
            x = *reinterpret_cast<const uint32_t *>(xg_in + (size_t)r * a.pitch + 4 * q);
            g = *reinterpret_cast<const uint32_t *>(a.g + (size_t)r * a.pitch + 4 * q);
            const int nv = W - 4 * q;
            if (nv < 4) {
                const uint32_t mask = (1u << (8 * nv)) - 1u;
                x = (x & mask) | (P::kFill & ~mask);
                g &= mask;
            }
        }
        pl0[i] = x;
        if (!GIBBS)
            pl1[i] = P::kFill;
        gw[i] = g;
    }
    for (int i = tid; i < (compact ? TH * TWq : TH * TW); i += nt)
        cnt[i] = 0u;
    if (tid < plane - words) {
        pl0[words + tid] = 0u;
        pl1[words + tid] = 0u;
        pl0[-1] = 0u;
    }

    const long long limit = wait_limit(a.wait_ns);
    const uint32_t key0 = (uint32_t)(a.seed & 0xFFFFFFFFull), key1 = (uint32_t)(a.seed >> 32);
    const uint32_t ctr3 = ((GIBBS ? kTagGibbs : kTagPCA) << 24) | (a.chain & 0xFFFFFFu);
    // 2^32 / divisor of a pass's and the uniforms' places, by e (an integer
    // division per thread and pass costs a fifth of a small tile's pass)
    constexpr int kMaxE = (GIBBS ? 2 : kTlMaxSweeps) * kCol;
    __shared__ unsigned int inv_pass[kMaxE], inv_uni[kMaxE];
    if (tid < kMaxE) {
        const int e = tid, q = kCol - 1 - e % kCol;
        const int words_row = TWq + 2 * ((e + 3) >> 2);
        int per = words_row;
        if (!WORDS)
            per = !GIBBS ? TW + 2 * e
                         : (NB == 4 ? (TW + 2 * e + 1) >> 1 : (TW + 2 * e - ((-e + q) & 1) + 1) >> 1);
        inv_pass[e] = 0xFFFFFFFFu / (unsigned int)per + 1u;
        inv_uni[e] = 0xFFFFFFFFu / (unsigned int)words_row + 1u;
    }
    __syncthreads();
    // the uniforms of `ns` sweeps from t on, at their staged words: sweep s
    // updates up to (ns - s) kCol - 1 sites beyond the tile
    const auto uniforms = [&](uint32_t t, int ns) {
        for (int s = 0; s < (compact ? 0 : ns); ++s) {
            const int e = (ns - s) * kCol - 1, eq = (e + 3) >> 2;
            const int per = TWq + 2 * eq, n = (TH + 2 * e) * per;
            const unsigned int inv = inv_uni[e];
            for (int i = tid; i < n; i += nt) {
                // (per == 1: the reciprocal does not fit 32 bits)
                const int ir = per == 1 ? i : (int)__umulhi((unsigned int)i, inv);
                const int lr = ir - e, lq = i - ir * per - eq;
                uint32_t o0, o1, o2, o3;
                philox4x32_10((uint32_t)(q0 + lq), (uint32_t)(r0 + lr + a.row_off),
                              t + (uint32_t)s, ctr3, key0, key1, o0, o1, o2, o3);
                reinterpret_cast<uint4 *>(U)[s * words + (lr + h) * SW + lq + hq] =
                    WORDS ? make_uint4(o0, o1, o2, o3)
                          : make_uint4(o0 >> 8, o1 >> 8, o2 >> 8, o3 >> 8);
            }
        }
    };
    // the byte counts to the accumulator
    const auto flush = [&]() {
        for (int i = tid; i < TH * TWq; i += nt) {
            const int lr = i / TWq, lq = i - lr * TWq;
            const uint32_t n4 = cnt[i];
            if (n4 == 0u)   // (always, outside the image)
                continue;
            cnt[i] = 0u;
            float *pa = a.acc + (size_t)(r0 + lr) * W + c0 + 4 * lq;
#pragma unroll
            for (int b = 0; b < 4; ++b)
                if ((n4 >> (8 * b)) & 0xFFu)
                    pa[b] += (float)((n4 >> (8 * b)) & 0xFFu);
        }
    };
    int nacc = 0;   // sweeps in the byte counts
    uniforms(t0, min(J.tg.k, nsweeps));
    bool ok = true;
    uint32_t *X = pl0;
    int done = 0;
    const bool ring = TH > 2 * h && TWq > 2 * hq;   // some words are not border words
    const int nrows = ring ? 2 * h * TWq : TH * TWq;
    const int nborder = ring ? nrows + (TH - 2 * h) * 2 * hq : nrows;
    for (unsigned int x = 1;; ++x) {                // exchanges
        const int ns = min(J.tg.k, nsweeps - done);
        // halo words and uniforms in place; leave together when a wait gave up
        if (__syncthreads_or(!ok)) {
            if (tid == 0)
                report_wait(err, a.gave_up);
            return;
        }
        // A pass computes its first sites' places and reads their inputs before
        // the barrier that ends the pass before it.
        bool fresh = true;   // no pass since the last barrier
        // (a run of one exchange's sweeps, written back in place, still waits
        // for the neighbours: they have then read their halo of the initial
        // labels)
        const bool more = done + ns < nsweeps || (x == 1 && xg_in == xg_out);
        const bool pub = more && (int)blockIdx.x != a.stall_tile - 1;
        const uint32_t tag = t0 + (uint32_t)(done + ns);
        unsigned long long *buf = J.xch + (size_t)(x & 1u) * H * Wq;
        for (int s = 0; s < ns; ++s) {
            const uint32_t t = t0 + (uint32_t)(done + s);
            const bool acc_now = accumulate_after(a, t);
            const uint32_t *Us = U + 4 * s * words;
            uint32_t *Y = GIBBS ? X : (X == pl0 ? pl1 : pl0);
#pragma unroll 1
            for (int q = 0; q < kCol; ++q) {
                // sites of colour q of rows [-e, TH + e), columns [-e, TW + e)
                const int e = (ns - s) * kCol - 1 - q;
                if constexpr (WORDS) {
                    // the words that hold them; labels of other sites in
                    // those words stay undefined
                    const int eq = (e + 3) >> 2, per = TWq + 2 * eq, n = (TH + 2 * e) * per;
                    const unsigned int inv = inv_pass[e];
                    for (int b = 0; b < n; b += nt) {
                        const int i = b + tid;
                        const int ir = per == 1 ? i : (int)__umulhi((unsigned int)i, inv);
                        const int lr = ir - e, lq = i - ir * per - eq, lc = 4 * lq;
                        const int lo = max(-e - lc, 0), hi = min(min(TW + e, W - c0) - lc, 4);
                        const bool valid = i < n && (unsigned)(r0 + lr) < (unsigned)H &&
                                           c0 + lc >= 0 && lo < hi;
                        const uint32_t act = valid ? (0xFFFFFFFFu << (8 * lo)) &
                                                         (0xFFFFFFFFu >> (8 * (4 - hi)))
                                                   : 0u;
                        const bool own = (unsigned)lr < (unsigned)TH && (unsigned)lq < (unsigned)TWq;
                        const int o = valid ? (lr + h) * SW + lq + hq : SW + 1;
                        uint4 u;
                        if (compact)
                            philox4x32_10((uint32_t)(q0 + lq), (uint32_t)(r0 + lr + a.row_off), t, ctr3,
                                          key0, key1, u.x, u.y, u.z, u.w);
                        else
                            u = reinterpret_cast<const uint4 *>(Us)[o];
                        const uint32_t G = gw[o];
                        if (b == 0 && !fresh)
                            __syncthreads();
                        fresh = false;
                        const uint32_t v = pol.draw4(a, X, o, SW, G, u, act, r0 + lr, c0 + lc, own);
                        if (valid) {
                            Y[o] = v;
                            if (compact) {
                                if (own && acc_now)
                                    cnt[lr * TWq + lq] += v & act;
                            } else if (own && acc_now) {
                                uint4 *pc = reinterpret_cast<uint4 *>(cnt + lr * TW + lc);
                                const uint32_t w = v & act;
                                uint4 n4 = *pc;
                                n4.x += w & 0xFFu;
                                n4.y += (w >> 8) & 0xFFu;
                                n4.z += (w >> 16) & 0xFFu;
                                n4.w += w >> 24;
                                *pc = n4;
                            }
                        }
                    }
                    continue;
                }
                int nr, per, sr0, sc0;   // rows, sites per row, first row and column
                if (!GIBBS) {
                    nr = TH + 2 * e;
                    per = TW + 2 * e;
                    sr0 = -e;
                    sc0 = -e;
                } else if (NB == 4) {
                    nr = TH + 2 * e;
                    per = (TW + 2 * e + 1) >> 1;
                    sr0 = -e;
                    sc0 = -e;
                } else {
                    sr0 = -e + ((r0 - e + (q >> 1)) & 1);
                    sc0 = -e + ((-e + q) & 1);
                    nr = (TH + e - sr0 + 1) >> 1;
                    per = (TW + e - sc0 + 1) >> 1;
                }
                const unsigned int inv = inv_pass[e];   // per >= 2
                for (int b = 0; b < nr * per; b += nt) {
                    const int i = b + tid;
                    const int ir = (int)__umulhi((unsigned int)i, inv), ic = i - ir * per;
                    const int lr = GIBBS && NB == 8 ? sr0 + 2 * ir : sr0 + ir;
                    int lc = GIBBS ? sc0 + 2 * ic : sc0 + ic;
                    if (GIBBS && NB == 4)
                        lc += (r0 + lr + c0 + lc + q) & 1;
                    const bool valid = ir < nr && lc < TW + e &&
                                       (unsigned)(r0 + lr) < (unsigned)H &&
                                       (unsigned)(c0 + lc) < (unsigned)W;
                    const bool own = (unsigned)lr < (unsigned)TH && (unsigned)lc < (unsigned)TW;
                    const int o = (lr + h) * SB + lc + hb;
                    const int g = valid ? (int)reinterpret_cast<const uint8_t *>(gw)[o] : 0;
                    const uint32_t ub = valid ? Us[o] : 0u;
                    if (b == 0 && !fresh)
                        __syncthreads();
                    fresh = false;
                    const int v = pol.draw(a, reinterpret_cast<const uint8_t *>(X) + o, SB, g, ub,
                                           r0 + lr, c0 + lc, valid, own);
                    if (valid) {
                        reinterpret_cast<uint8_t *>(Y)[o] = (uint8_t)v;
                        if (own && acc_now)
                            cnt[lr * TW + lc] += (uint32_t)v;
                    }
                }
            }
            X = Y;
            if (compact && acc_now && ++nacc == 255) {   // the counts are full
                __syncthreads();
                flush();
                nacc = 0;   // (each count is its own thread's again after the next barrier)
            }
        }
        __syncthreads();
        done += ns;
        if (!more)
            break;
        if (pub)   // publish the border words: whole rows, then the sides of the others
            for (int i = tid; i < nborder; i += nt) {
                int lr, lq;
                if (i < nrows) {
                    lr = i / TWq;
                    lq = i - lr * TWq;
                    lr += ring && lr >= h ? TH - 2 * h : 0;
                } else {
                    lr = (i - nrows) / (2 * hq);
                    lq = i - nrows - lr * 2 * hq;
                    lr += h;
                    lq += lq < hq ? 0 : TWq - 2 * hq;
                }
                if (r0 + lr < H && q0 + lq < Wq)
                    st_word(buf + (size_t)(r0 + lr) * Wq + q0 + lq,
                            ((unsigned long long)tag << 32) | X[(lr + h) * SW + lq + hq]);
            }
        uniforms(t0 + (uint32_t)done, min(J.tg.k, nsweeps - done));
        // poll the halo: h rows above and below (with the corners where they
        // are read), hq words left and right of each row
        const bool corners = NB == 8 || GIBBS || h > 1;
        const int nrow = 2 * h * SW, nh = nrow + 2 * hq * TH;
        for (int i = tid; i < nh && ok; i += nt) {
            int sr, sq;
            if (i < nrow) {
                sr = i / SW;
                sq = i - sr * SW;
                if (!corners && (sq < hq || sq >= SW - hq))
                    continue;   // no diagonal neighbours
                sr = sr < h ? sr : sr + TH;
            } else {
                sr = (i - nrow) / (2 * hq);
                sq = (i - nrow) - sr * 2 * hq;
                sr += h;
                sq = sq < hq ? sq : sq + TWq;
            }
            const int r = r0 - h + sr, q = q0 - hq + sq;
            if (r < 0 || r >= H || q < 0 || q >= Wq)
                continue;
            uint32_t w;
            ok = poll_word(buf + (size_t)r * Wq + q, tag, w, err, limit);
            if (ok)
                X[sr * SW + sq] = w;
        }
        if (done == nsweeps)
            break;
    }
    if (__syncthreads_or(!ok)) {
        if (tid == 0)
            report_wait(err, a.gave_up);
        return;
    }
    pol.finish(a);
    // labels and counts back (a label of this plane that a neighbour read at
    // the start was read before it published its first exchange, which this
    // tile awaited, or the planes differ)
    if (compact)
        flush();
    for (int i = tid; i < TH * TWq; i += nt) {
        const int lr = i / TWq, lq = i - lr * TWq;
        const int r = r0 + lr, c = c0 + 4 * lq;
        if (r >= H || c >= W)
            continue;
        const uint32_t w = X[(lr + h) * SW + lq + hq];
        float *pa = a.acc + (size_t)r * W + c;
        const uint32_t *n4 = cnt + lr * TW + 4 * lq;
        const int nv = min(4, W - c);
        if (nv == 4)
            *reinterpret_cast<uint32_t *>(xg_out + (size_t)r * a.pitch + c) = w;
        for (int b = 0; b < nv; ++b) {
            if (nv < 4)
                xg_out[(size_t)r * a.pitch + c + b] = (uint8_t)(w >> (8 * b));
            if (!compact && n4[b])
                pa[b] += (float)n4[b];
        }
    }
}

// Time model of a sweep of a tile (ns; k sweeps per exchange), for the choice
// of the grid and of k only: kNsPass per pass over the sites (block barrier
// and the latency of one draw; kNsPassWords, of four), `site` per site an SM
// draws, kNsExchange per exchange and kNsHaloWord per word of its halo.
constexpr double kNsPass = 350.0, kNsPassWords = 550.0, kNsExchange = 1300.0, kNsHaloWord = 0.5;

double tile_cost(const TileGeom &g, int phases, int per_sm, double site, bool words)
{
    double ns = kNsExchange + kNsHaloWord * per_sm * (2 * g.h * (g.twq + 2 * g.hq) + 2 * g.hq * g.th);
    for (int s = 0; s < g.k; ++s)
        for (int q = 0; q < phases; ++q) {
            const int e = (g.k - s) * phases - 1 - q;
            const double row = words ? 4.0 * (g.twq + 2 * ((e + 3) / 4)) : 4.0 * g.twq + 2 * e;
            ns += (words ? kNsPassWords : kNsPass) + site * per_sm * (g.th + 2 * e) * row / phases;
        }
    return ns / g.k;
}

// Tiles of which a lazy-PCA sweep draws whole words.
template <class P, bool GIBBS>
bool draws_words(const TileGeom &g)
{
    if constexpr (P::kWords && !GIBBS)
        return g.th * g.twq >= P::kWordsMin;
    return false;
}

// The tile grid of an image: at most `ctas` tiles of at least h rows and
// columns, k sweeps per exchange.
template <class P, bool GIBBS>
bool tile_geometry(int H, int W, int ctas, int per_sm, bool compact, TileGeom &best)
{
    constexpr int phases = tile_phases(P::NB, GIBBS);
    const size_t most = per_sm == 2 ? kTlMaxSmem2 : kTlMaxSmem;
    const int Wq = (W + 3) / 4;
    double best_cost = -1.0;
    for (int k = 1; k <= (GIBBS ? 2 : kTlMaxSweeps); ++k)
        for (int nx = 1, wide = 0; nx <= ctas && nx <= Wq; ++nx) {
            if ((Wq + nx - 1) / nx == wide)
                continue;   // the same tiles as with fewer columns of them
            wide = (Wq + nx - 1) / nx;
            TileGeom g{};
            g.k = k;
            g.two = per_sm == 2;
            g.h = k * phases;
            g.hq = (g.h + 3) / 4;
            g.twq = wide;
            if (g.twq < g.hq)
                g.twq = g.hq;
            g.tiles_x = (Wq + g.twq - 1) / g.twq;
            const int rows = ctas / g.tiles_x;
            g.th = (H + rows - 1) / rows;
            if (g.th < g.h)
                g.th = g.h;
            g.tiles_y = (H + g.th - 1) / g.th;
            g.compact = compact && P::kCompact && !GIBBS && g.th * g.twq * 4 > kTlMaxSites;
            if ((!g.compact && (long)g.th * g.twq * 4 > kTlMaxSites) || g.tiles_x * g.tiles_y > ctas)
                continue;
            // one CTA per SM: a thread per site of the widest pass, if they are
            // few (idle warps still take every barrier)
            const long most_sites = (long)(g.th + 2 * g.h - 2) * (4 * g.twq + 2 * g.h - 2) / phases;
            g.threads = per_sm == 2 ? tile_threads<P, GIBBS>(true)
                                    : (int)std::min<long>(tile_threads<P, GIBBS>(false),
                                                          std::max<long>(256, (most_sites + 127) / 128 * 128));
            // (the scratch of the widest launch: a pack has its widest job's threads)
            if (tile_smem<P, GIBBS>(g, tile_threads<P, GIBBS>(per_sm == 2)) > most)
                continue;
            const bool words = draws_words<P, GIBBS>(g);
            const double cost =
                tile_cost(g, phases, per_sm, words ? P::kNsSiteWords : P::kNsSite, words);
            if (best_cost < 0.0 || cost < best_cost) {
                best_cost = cost;
                best = g;
            }
        }
    return best_cost >= 0.0;
}

// Threads of a launch that draws words: one per word of the widest pass, as
// far as they go.
inline int word_threads(const TileGeom &g)
{
    if (g.two)
        return kTlWideThreads;
    const int wide = (g.th + 2 * g.h - 2) * (g.twq + 2 * ((g.h + 2) / 4));
    return std::min(kTlWideThreads1, std::max(256, (wide + 127) / 128 * 128));
}

template <class P, bool GIBBS, int JOBS, bool WORDS>
cudaError_t launch_w(const TileLaunchT<JOBS> &L, int ctas, cudaStream_t st)
{
    static bool attr_set[64] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess)
        return e;
    if (dev >= 64)
        return cudaErrorInvalidDevice;
    auto kern = tile_kernel<P, GIBBS, JOBS, WORDS>;
    if (!attr_set[dev]) {
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kTlMaxSmem);
        if (e != cudaSuccess)
            return e;
        attr_set[dev] = true;
    }
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(ctas);
    int threads = 0;   // the widest job's; shared memory for every job with them
    size_t smem = 0;
    for (int i = 0; i < L.njobs; ++i)
        threads = std::max(threads, WORDS ? word_threads(L.job[i].tg) : L.job[i].tg.threads);
    for (int i = 0; i < L.njobs; ++i)
        smem = std::max(smem, tile_smem<P, GIBBS>(L.job[i].tg, threads));
    if (threads < 1 || smem > (size_t)kTlMaxSmem)
        return cudaErrorInvalidValue;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;   // the CTAs wait on one another
    at[0].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, L);
}

// Draws of words where the tiles of every chain of the launch hold enough of
// them; results do not depend on the choice.
template <class P, bool GIBBS, int JOBS>
cudaError_t launch_t(const TileLaunchT<JOBS> &L, int ctas, cudaStream_t st)
{
    if constexpr (P::kWords && !GIBBS) {
        bool words = true;
        for (int i = 0; i < L.njobs; ++i)
            words = words && draws_words<P, GIBBS>(L.job[i].tg);
        if (words)
            return launch_w<P, GIBBS, JOBS, true>(L, ctas, st);
    }
    return launch_w<P, GIBBS, JOBS, false>(L, ctas, st);
}

// f(policy, GIBBS) for the kind's instance.
template <class F>
auto with_policy(const TileKind &k, F f)
{
    const auto g = [&](auto pol) {
        return k.gibbs ? f(pol, std::true_type{}) : f(pol, std::false_type{});
    };
    if (k.draw == TileKind::kBinary)
        return k.nbhd == 8 ? g(static_cast<BinPol<8> *>(nullptr))
                           : g(static_cast<BinPol<4> *>(nullptr));
    if (k.draw == TileKind::kSegment)
        return g(static_cast<SegPol *>(nullptr));
    if (k.nbhd == 8)
        return k.lmax == 8 ? (k.mask ? g(static_cast<SmallPol<8, 8, true> *>(nullptr))
                                     : g(static_cast<SmallPol<8, 8, false> *>(nullptr)))
                           : (k.mask ? g(static_cast<SmallPol<16, 8, true> *>(nullptr))
                                     : g(static_cast<SmallPol<16, 8, false> *>(nullptr)));
    return k.lmax == 8 ? (k.mask ? g(static_cast<SmallPol<8, 4, true> *>(nullptr))
                                 : g(static_cast<SmallPol<8, 4, false> *>(nullptr)))
                       : (k.mask ? g(static_cast<SmallPol<16, 4, true> *>(nullptr))
                                 : g(static_cast<SmallPol<16, 4, false> *>(nullptr)));
}

}  // namespace

bool tile_kind(const DevModel &m, bool gibbs, TileKind &k)
{
    k = TileKind{};
    k.nbhd = m.nbhd;
    k.gibbs = gibbs;
    if (m.norm != 0 || (m.nbhd != 4 && m.nbhd != 8))
        return false;
    if (m.L == 2) {
        k.draw = TileKind::kBinary;
        return true;
    }
    if (m.L >= kSmallMinLabels && m.L <= kSmallMaxLabels && m.gam <= 0.0f && m.alpha <= 0.0f) {
        k.draw = TileKind::kSmall;
        k.lmax = m.L <= 8 ? 8 : 16;
        k.mask = m.L != k.lmax;
        return true;
    }
    k.draw = TileKind::kSegment;
    return seg_eligible(m);
}

namespace {

bool plan_geometry(const TileKind &k, int H, int W, int ctas, bool two, bool compact, TileGeom &tg)
{
    if (ctas <= 0)
        return false;
    return with_policy(k, [&](auto pol, auto gibbs) {
        using P = std::remove_pointer_t<decltype(pol)>;
        return tile_geometry<P, decltype(gibbs)::value>(H, W, ctas, two ? 2 : 1, compact, tg);
    });
}

}  // namespace

bool tile_plan(const TileKind &k, int H, int W, int sms, TilePlan &p)
{
    const bool two = (long long)H * W > (long long)sms * kTlThreads1;
    if (!(two && plan_geometry(k, H, W, 2 * sms, true, false, p.tg)) &&
        !plan_geometry(k, H, W, sms, false, true, p.tg))
        return false;
    p.ctas = p.tg.tiles_x * p.tg.tiles_y;
    return true;
}

bool tile_plan_ctas(const TileKind &k, int H, int W, int ctas, bool two, TileGeom &tg)
{
    return plan_geometry(k, H, W, ctas, two, false, tg);
}

size_t tile_xch_bytes(int H, int W)
{
    return (size_t)2 * H * ((W + 3) / 4) * sizeof(unsigned long long);
}

namespace {

template <int JOBS>
cudaError_t launch_checked(const TileKind &k, const TileLaunchT<JOBS> &L, int ctas,
                           cudaStream_t st)
{
    if (L.njobs < 1 || L.njobs > JOBS || ctas < 1)
        return cudaErrorInvalidValue;
    if (L.nsweeps <= 0)
        return cudaSuccess;
    for (int i = 0; i < L.njobs; ++i) {
        const TileJob &J = L.job[i];
        TileKind kk;
        if (!tile_kind(J.a.m, k.gibbs, kk) || !(kk == k) || J.xch == nullptr)
            return cudaErrorInvalidValue;
        if ((k.draw == TileKind::kSmall && !J.a.m.ptab) ||
            (k.draw == TileKind::kBinary && !J.a.m.btab) ||
            (k.draw == TileKind::kSegment && !J.a.m.stab))
            return cudaErrorInvalidValue;
        // word loads and stores of the planes
        if ((J.a.pitch & 3) != 0 ||
            ((reinterpret_cast<uintptr_t>(J.x0) | reinterpret_cast<uintptr_t>(J.x1) |
              reinterpret_cast<uintptr_t>(J.a.g)) & 3u) != 0)
            return cudaErrorMisalignedAddress;
    }
    return with_policy(k, [&](auto pol, auto gibbs) {
        using P = std::remove_pointer_t<decltype(pol)>;
        if constexpr (JOBS > 1 && decltype(gibbs)::value)
            return cudaErrorInvalidValue;   // batches and the server run the PCA sampler
        else
            return launch_t<P, decltype(gibbs)::value, JOBS>(L, ctas, st);
    });
}

}  // namespace

cudaError_t launch_tile(const TileKind &k, const TileLaunch &L, int ctas, cudaStream_t st)
{
    return launch_checked(k, L, ctas, st);
}

cudaError_t launch_tile(const TileKind &k, const TilePack &L, int ctas, cudaStream_t st)
{
    return launch_checked(k, L, ctas, st);
}

}  // namespace pcad
