// Lazy-PCA sweeps (Section 5.2, Eq. posterior_pca_transition_matrix) and
// checkerboard Gibbs colour phases (Section 5.1) with the segment draw
// (seg_draw.cuh): 4 neighbours, c >= 0, many labels.  They run in place of
// the windowed draw (win.cu) for the models seg_eligible accepts, in the same
// two launch forms:
//
//   * one launch per sweep (per colour phase): one persistent block per SM (24
//     warps, 80 registers; colour phases 32 warps, 64), its warps taking tiles
//     of 4 x 32 sites (64 columns x 4 rows of cells for Gibbs) as they come
//     free.  A block copies the model's prefix tables (18 KB) into shared
//     memory once per launch; there is no other block barrier.  A lane owns a
//     column of the tile and walks its 4 rows with the labels above, at and
//     below it in registers; one Philox call per lane and tile serves the tile's
//     128 sites.
//     Bound by instruction issue: 842 warp instructions per 32 site-updates (700
//     in the draw) at 88 % issue, ALU pipe 65 %, DRAM 5 %.
//     L = 256, T = 30, sigma = 25, 8192^2: 1.60 ms per sweep (4.19e10
//     site-updates/s) against 4.05 ms for the windowed draw.  Gibbs at 4096^2:
//     434 us per sweep (3.9e10; 479 with a fixed share per warp).
//   * the wavefront for images of few tiles: the sweeps of a block in one
//     persistent launch, items and waits as in win.cu's wavefront, one site
//     per thread.  512^2: 9.4 us per sweep against 17.9 us (Gibbs 14.4 against
//     26 us).
#include <algorithm>

#include "seg_draw.cuh"

namespace pcad {

namespace {

using namespace seg;

constexpr int kSX = 32;
constexpr int kSY = 4;
constexpr int kSegWarps = 24;                // per-sweep blocks: one per SM (80 registers)
constexpr int kSegThreads = 32 * kSegWarps;
constexpr int kSegGibbsWarps = 32;           // per colour phase (64 registers)
constexpr int kSegGibbsThreads = 32 * kSegGibbsWarps;
constexpr int kSegwThreads = kSX * kSY;      // wavefront blocks
constexpr double kBias = 3.9443045261050590e-31;   // 2^-101

// Row blockIdx.x - 4 of the prefix tables of job blockIdx.y, one thread per entry:
// FP64 terms (the model's data factors times 2^(mu k d), mu the FP32 coefficient
// the sweeps use), an FP64 scan, one rounding.
template <int N>
struct SegTabJobs {
    SegTabJob job[N];
};

template <int N>
__global__ void __launch_bounds__(kSegRow)
    seg_table_kernel(const __grid_constant__ SegTabJobs<N> jobs)
{
    const DevModel &m = jobs.job[N > 1 ? blockIdx.y : 0].m;
    float *const out = jobs.job[N > 1 ? blockIdx.y : 0].out;
    __shared__ double v[2][kSegRow];
    const int k = (int)blockIdx.x - 4, j = (int)threadIdx.x;
    const int d = j - 256;
    // k >= 0: sum over d' <= d; k < 0: sum over d' > d, scanned from the top
    const int at = k >= 0 ? j : kSegRow - 1 - j;
    double x = 0.0;
    if (d > -m.L && d < m.L)   // a label's d = s - g; no other entry is read
        x = m.ta64[kTableOffset + d] *
            exp2((double)(-m.gam) * (double)k * (double)d - rint((double)m.cbs - (double)m.cb));
    v[0][at] = x;
    __syncthreads();
    int cur = 0;
    for (int o = 1; o < kSegRow; o <<= 1) {
        v[cur ^ 1][j] = v[cur][j] + (j >= o ? v[cur][j - o] : 0.0);
        cur ^= 1;
        __syncthreads();
    }
    const double F = k >= 0 ? v[cur][at] + kBias
                            : -((at > 0 ? v[cur][at - 1] : 0.0) + kBias);
    out[(size_t)blockIdx.x * kSegRow + j] = (float)F;
}

__device__ __forceinline__ void load_tab(float *tab, const float *src, int tid, int n)
{
    for (int i = tid; i < kSegFloats / 4; i += n)
        reinterpret_cast<float4 *>(tab)[i] = __ldg(reinterpret_cast<const float4 *>(src) + i);
}

// A warp's next tile: groups of WARPS tiles go to the blocks in turn, and a
// block's warps take its tiles as they come free.  With a fixed share per warp
// and three blocks of 8 warps per SM the scheduler ran the oldest warps ahead,
// and the last part of a sweep had few left (30 % of warps active on average
// against 37.5 % resident): one block per SM whose warps share its tiles, 8192^2,
// L = 256 1773 -> 1603 us per sweep (three such blocks per SM: 1786).
template <int WARPS>
__device__ __forceinline__ int next_tile(int *taken, int lane)
{
    int n = 0;
    if (lane == 0)
        n = atomicAdd(taken, 1);
    n = __shfl_sync(0xFFFFFFFFu, n, 0);
    return ((n / WARPS) * (int)gridDim.x + (int)blockIdx.x) * WARPS + n % WARPS;
}

// One lazy-PCA sweep: a.xin -> a.xout (or the planes x0 / x1 by the parity of
// the sweep index), skipped at or past *budget.
__global__ void __launch_bounds__(kSegThreads, 1)
    pca_seg_kernel(const SweepArgs a, int tiles_x, int ntiles, uint8_t *x0,
                   uint8_t *x1, const uint32_t *budget)
{
    __shared__ __align__(16) float tab[kSegFloats];
    __shared__ __align__(16) uint32_t U_s[kSegWarps][kSY * kSX];
    __shared__ int s_taken;
    const uint32_t t = sweep_index(a);
    if (budget && t >= *budget)
        return;   // the whole launch, before any barrier
    const uint8_t *xin = x0 ? ((t & 1u) ? x1 : x0) : a.xin;
    uint8_t *xout = x0 ? ((t & 1u) ? x0 : x1) : a.xout;
    const int lane = (int)threadIdx.x & 31, wp = (int)threadIdx.x >> 5;
    load_tab(tab, a.m.stab, (int)threadIdx.x, kSegThreads);
    if (threadIdx.x == 0)
        s_taken = 0;
    __syncthreads();
    const bool acc_on = accumulate_after(a, t);
    const int H = a.H, W = a.W;
    uint32_t *U = U_s[wp];
    for (int tile; (tile = next_tile<kSegWarps>(&s_taken, lane)) < ntiles;) {
        const int ty = tile / tiles_x, tx = tile - ty * tiles_x;
        const int r0 = ty * kSY, c = tx * kSX + lane;
        block_uniforms(a, r0, tx * kSX, t, U);
        __syncwarp();
        const bool cv = c < W;
        // tiles whose halo lies inside the image load without bounds tests
        const bool inner = r0 >= 1 && r0 + kSY < H && tx >= 1 && (tx + 1) * kSX < W;
        const auto at = [&](int r, int cc) -> int {
            return (unsigned)r < (unsigned)H && (unsigned)cc < (unsigned)W
                       ? (int)xin[(size_t)r * a.pitch + cc] : kMissingLabelI;
        };
        const uint8_t *px = xin + (size_t)r0 * a.pitch + c, *pg = a.g + (size_t)r0 * a.pitch + c;
        int up, cur, dn, le, ri, g;
        if (inner) {
            up = px[-(ptrdiff_t)a.pitch];
            cur = px[0];
            dn = px[a.pitch];
            le = px[-1];
            ri = px[1];
            g = pg[0];
        } else {
            up = at(r0 - 1, c);
            cur = at(r0, c);
            dn = at(r0 + 1, c);
            le = at(r0, c - 1);
            ri = at(r0, c + 1);
            g = cv && r0 < H ? (int)pg[0] : 0;
        }
#pragma unroll 1
        for (int i = 0; i < kSY; ++i) {
            const int r = r0 + i;
            const bool valid = inner || (cv && r < H);
            SiteIn<4> in;
            in.g = g;
            in.xi = valid ? cur : 0;
            in.xni[0] = up;
            in.xni[1] = dn;
            in.xni[2] = le;
            in.xni[3] = ri;
            in.ub = U[i * kSX + lane];
            // the next row's labels and observation, in flight during the draw
            up = cur;
            cur = dn;
            px += a.pitch;
            pg += a.pitch;
            if (i + 1 < kSY) {
                if (inner) {
                    dn = px[a.pitch];
                    le = px[-1];
                    ri = px[1];
                    g = pg[0];
                } else {
                    dn = at(r + 2, c);
                    le = at(r + 1, c - 1);
                    ri = at(r + 1, c + 1);
                    g = cv && r + 1 < H ? (int)pg[0] : 0;
                }
            }
            float *pa = a.acc + (size_t)r * W + c;
            const float old = valid && acc_on ? *pa : 0.0f;
            bool certain = true;
            int s = 0;
            if (valid)
                s = draw_seg(a.m, tab, in, certain);
            s = warp_redraw_fp64<4>(a.m, valid && !certain, in, s, a.fp64_draws);
            if (valid) {
                xout[(size_t)r * a.pitch + c] = (uint8_t)s;
                if (acc_on)
                    *pa = old + (float)s;
            }
        }
        __syncwarp();   // U is read
    }
}

// Wavefront form: items, waits and planes as pca_winw_kernel's.
__global__ void __launch_bounds__(kSegwThreads, 8)
    pca_segw_kernel(const SweepArgs a, uint8_t *x0, uint8_t *x1, int nsweeps,
                    int tiles_x, int tiles_y, unsigned int *done, unsigned int *grab, int *err,
                    int par_from_t, const uint32_t *budget)
{
    __shared__ __align__(16) float tab[kSegFloats];
    __shared__ __align__(16) uint32_t U_s[kSY * kSX];
    __shared__ unsigned int s_next;
    const int lane = (int)threadIdx.x, wp = (int)threadIdx.y;
    const int tid = wp * kSX + lane;
    const unsigned int ntiles = (unsigned int)(tiles_x * tiles_y);
    const unsigned int total = ntiles * (unsigned int)nsweeps;
    const uint32_t t0 = sweep_index(a);
    const long long limit = wait_limit(a.wait_ns);
    load_tab(tab, a.m.stab, tid, kSegwThreads);
    if (tid == 0)
        s_next = atomicAdd(grab, 1u);
    __syncthreads();
    unsigned int item = s_next;
    while (item < total) {
        const int k = (int)(item / ntiles);
        const int j = (int)(item - (unsigned int)k * ntiles);
        const int ty = j / tiles_x;
        const int tx = j - ty * tiles_x;
        const uint32_t t = t0 + (uint32_t)k;
        const bool run = budget == nullptr || t < *budget;   // the same for the whole block
        __syncthreads();   // s_next read; the previous item's uniforms are read
        if (wp == 0) {
            // lane 31 takes the following item (none once a wait of the
            // launch gave up); lanes 0-8 wait for the 3 x 3 tiles around j
            if (lane == 31)
                s_next = ld_flag(err) ? total : atomicAdd(grab, 1u);
            bool ok = true;
            if (run && k > 0 && lane < 9) {
                const int yy = ty + lane / 3 - 1;
                const int xx = tx + lane % 3 - 1;
                if (yy >= 0 && yy < tiles_y && xx >= 0 && xx < tiles_x) {
                    const unsigned int *d = done + (size_t)yy * tiles_x + xx;
                    ok = wait_ge(d, (unsigned int)k, ld_acquire_u32(d), err, limit);
                }
            }
            if (!ok)
                report_wait(err, a.gave_up);
            __syncwarp();
        } else if (wp == 1 && run) {
            block_uniforms(a, ty * kSY, tx * kSX, t, U_s);
        }
        __syncthreads();
        if (run) {
            const uint32_t ph = par_from_t ? (t & 1u) : (uint32_t)(k & 1);
            const uint8_t *xin = ph ? x1 : x0;
            uint8_t *xout = ph ? x0 : x1;
            const int r = ty * kSY + wp, c = tx * kSX + lane;
            const bool valid = r < a.H && c < a.W;
            SiteIn<4> in{};
            bool certain = true;
            int s = 0;
            if (valid) {
                load_site<4, true, false>(a, xin, r, c, kTagPCA, t, in);
                in.ub = U_s[tid];
                s = draw_seg(a.m, tab, in, certain);
            }
            s = warp_redraw_fp64<4>(a.m, valid && !certain, in, s, a.fp64_draws);
            if (valid) {
                xout[(size_t)r * a.pitch + c] = (uint8_t)s;
                if (accumulate_after(a, t)) {
                    float *p = a.acc + (size_t)r * a.W + c;
                    *p = __ldcg(p) + (float)s;
                }
            }
        }
        __syncthreads();
        // a skipped item publishes nothing (see pca_winw_kernel)
        if (run && tid == 0 && j != a.stall_tile - 1) {
            __threadfence();   // the tile's labels and sums before its counter
            atomicExch(done + j, (unsigned int)(k + 1));
        }
        item = s_next;
    }
}

// The uniforms of Gibbs tile rows [row0, row0 + 4), columns 64 tx ..: call i
// (0 .. 63) serves row row0 + i / 16, columns 64 tx + 4 (i % 16) .. + 3.
__device__ __forceinline__ void gibbs_uniforms(const SweepArgs &a, int row0, int tx, uint32_t t,
                                               int i, uint32_t *U)
{
    uint32_t o0, o1, o2, o3;
    philox4x32_10((uint32_t)(16 * tx + (i & 15)), (uint32_t)(row0 + (i >> 4) + a.row_off), t,
                  (kTagGibbs << 24) | (a.chain & 0xFFFFFFu), (uint32_t)(a.seed & 0xFFFFFFFFull),
                  (uint32_t)(a.seed >> 32), o0, o1, o2, o3);
    reinterpret_cast<uint4 *>(U)[i] = make_uint4(o0 >> 8, o1 >> 8, o2 >> 8, o3 >> 8);
}

// Colour phase q in place on a.xin: warp tiles of 64 columns x 4 rows, lane l
// the column pair 2 l; after the last phase (a.last_phase) the pairs are
// accumulated.  A phase writes one colour and reads the other, but for the
// site's own label, which only the accumulation reads, after its own write.
__global__ void __launch_bounds__(kSegGibbsThreads, 1)
    gibbs_seg_kernel(const SweepArgs a, int q, int tiles_x, int ntiles)
{
    __shared__ __align__(16) float tab[kSegFloats];
    __shared__ __align__(16) uint32_t U_s[kSegGibbsWarps][kSY * 2 * kSX];
    __shared__ int s_taken;
    uint8_t *x = const_cast<uint8_t *>(a.xin);
    const uint32_t t = sweep_index(a);
    const int lane = (int)threadIdx.x & 31, wp = (int)threadIdx.x >> 5;
    load_tab(tab, a.m.stab, (int)threadIdx.x, kSegGibbsThreads);
    if (threadIdx.x == 0)
        s_taken = 0;
    __syncthreads();
    const bool acc_on = a.last_phase && accumulate_after(a, t);
    uint32_t *U = U_s[wp];
    for (int tile; (tile = next_tile<kSegGibbsWarps>(&s_taken, lane)) < ntiles;) {
        const int ty = tile / tiles_x, tx = tile - ty * tiles_x;
        const int r0 = ty * kSY, c0 = 2 * (tx * kSX + lane);
        gibbs_uniforms(a, r0, tx, t, lane, U);
        gibbs_uniforms(a, r0, tx, t, lane + 32, U);
        __syncwarp();
#pragma unroll 1
        for (int i = 0; i < kSY; ++i) {
            const int r = r0 + i, c = c0 + ((r + q) & 1);
            const bool valid = r < a.H && c < a.W;
            SiteIn<4> in{};
            bool certain = true;
            int s = 0;
            if (valid) {
                load_site<4, false, false>(a, x, r, c, kTagGibbs, t, in);
                in.ub = U[i * 2 * kSX + (c - 2 * kSX * tx)];
                s = draw_seg(a.m, tab, in, certain);
            }
            s = warp_redraw_fp64<4>(a.m, valid && !certain, in, s, a.fp64_draws);
            if (valid)
                x[(size_t)r * a.pitch + c] = (uint8_t)s;
            if (acc_on && r < a.H) {
#pragma unroll
                for (int dc = 0; dc < 2; ++dc) {
                    const int cc = c0 + dc;
                    if (cc < a.W)
                        a.acc[(size_t)r * a.W + cc] +=
                            (float)(cc == c ? s : (int)x[(size_t)r * a.pitch + cc]);
                }
            }
        }
        __syncwarp();   // U is read
    }
}

// Wavefront of colour phases: items and waits as gibbs_winw_kernel's.
__global__ void __launch_bounds__(kSegwThreads, 7)
    gibbs_segw_kernel(const SweepArgs a, uint8_t *x, int nphases, int tiles_x,
                      int tiles_y, unsigned int *done, unsigned int *grab, int *err)
{
    __shared__ __align__(16) float tab[kSegFloats];
    __shared__ __align__(16) uint32_t U_s[kSY * 2 * kSX];
    __shared__ unsigned int s_next;
    const int lane = (int)threadIdx.x, wp = (int)threadIdx.y;
    const int tid = wp * kSX + lane;
    const unsigned int ntiles = (unsigned int)(tiles_x * tiles_y);
    const unsigned int total = ntiles * (unsigned int)nphases;
    const uint32_t t0 = sweep_index(a);
    const long long limit = wait_limit(a.wait_ns);
    load_tab(tab, a.m.stab, tid, kSegwThreads);
    if (tid == 0)
        s_next = atomicAdd(grab, 1u);
    __syncthreads();
    unsigned int item = s_next;
    while (item < total) {
        const int k = (int)(item / ntiles);
        const int j = (int)(item - (unsigned int)k * ntiles);
        const int ty = j / tiles_x;
        const int tx = j - ty * tiles_x;
        const int q = k & 1;
        const uint32_t t = t0 + (uint32_t)(k >> 1);
        __syncthreads();   // s_next read; the previous item's uniforms are read
        if (wp == 0) {
            if (lane == 31)
                s_next = ld_flag(err) ? total : atomicAdd(grab, 1u);
            bool ok = true;
            if (k > 0 && lane < 9) {
                const int yy = ty + lane / 3 - 1;
                const int xx = tx + lane % 3 - 1;
                if (yy >= 0 && yy < tiles_y && xx >= 0 && xx < tiles_x) {
                    const unsigned int *d = done + (size_t)yy * tiles_x + xx;
                    ok = wait_ge(d, (unsigned int)k, ld_acquire_u32(d), err, limit);
                }
            }
            if (!ok)
                report_wait(err, a.gave_up);
            __syncwarp();
        } else if (wp == 1 || wp == 2) {
            gibbs_uniforms(a, ty * kSY, tx, t, (wp - 1) * 32 + lane, U_s);
        }
        __syncthreads();
        const int r = ty * kSY + wp, c0 = 2 * (tx * kSX + lane);
        const int c = c0 + ((r + q) & 1);
        const bool valid = r < a.H && c < a.W;
        SiteIn<4> in{};
        bool certain = true;
        int s = 0;
        if (valid) {
            load_site<4, true, false>(a, x, r, c, kTagGibbs, t, in);
            in.ub = U_s[wp * 2 * kSX + (c - 2 * kSX * tx)];
            s = draw_seg(a.m, tab, in, certain);
        }
        s = warp_redraw_fp64<4>(a.m, valid && !certain, in, s, a.fp64_draws);
        if (valid)
            x[(size_t)r * a.pitch + c] = (uint8_t)s;
        if (q == 1 && r < a.H && accumulate_after(a, t)) {
#pragma unroll
            for (int dc = 0; dc < 2; ++dc) {
                const int cc = c0 + dc;
                if (cc < a.W) {
                    float *p = a.acc + (size_t)r * a.W + cc;
                    const int v = cc == c ? s : (int)__ldcg(x + (size_t)r * a.pitch + cc);
                    *p = __ldcg(p) + (float)v;
                }
            }
        }
        __syncthreads();
        if (tid == 0 && j != a.stall_tile - 1) {
            __threadfence();   // the tile's labels and sums before its counter
            atomicExch(done + j, (unsigned int)(k + 1));
        }
        item = s_next;
    }
}

// Resident blocks of a kernel on the current device (queried once per device).
template <typename K>
cudaError_t resident(K kernel, int threads, int (&per_sm)[64], int &blocks)
{
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess)
        return e;
    if (dev >= 64)
        return cudaErrorInvalidDevice;
    if (per_sm[dev] == 0) {
        int n = 0;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kernel, threads, 0);
        if (e != cudaSuccess)
            return e;
        per_sm[dev] = n > 0 ? n : 1;
    }
    e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    blocks = per_sm[dev] * sms;
    return e;
}

}  // namespace

int seg_table_floats()
{
    return kSegFloats;
}

// c >= 0, Gaussian or no likelihood, L0 price, 4 neighbours, and exponents
// that fit FP32.  A line's value at d = 0 lies within +-B, B = 4 mu (L - 1 + T)
// + A bits; the scales 2^(c + S) carry an offset S (the tables 2^-S) that
// keeps them from being flushed below 2^-126, S = 0 for B <= 125 (c_T <=
// 0.068 at L = 256, T = 30).  A scale above 2^127 turns Z into an infinity or
// a NaN, which certifies nothing: such a site is re-drawn in FP64.  It takes
// four neighbours more than (127 - S) / (4 mu) labels away from the
// observation, so that distance must be one the noise does not reach.  The
// rows' sums must stay below 2^127.
bool seg_structure(const DevModel &m)
{
    return m.nbhd == 4 && m.T >= 1 && m.L >= 9 && m.L <= 256;
}

float seg_offset(const DevModel &m)
{
    const float no = NAN;
    if (!seg_structure(m) || m.norm != 0 || m.gam > 0.0f || m.alpha > 0.0f)
        return no;
    const double mu = -(double)m.gam, A = mu * 4.0 * m.T, range = m.L - 1 + m.T;
    const double S = std::ceil(std::fmax(0.0, 4.0 * mu * range + A - 125.0));
    const double sigma = m.alpha < 0.0f ? std::sqrt(0.5 * 1.4426950408889634 / -(double)m.alpha)
                                        : 1e9;
    if (S > 0.0 && (127.0 - S) / (4.0 * mu) < std::fmin(range, 5.0 * sigma + m.T))
        return no;
    // the largest alpha d^2 + 4 mu d over d < L
    double d = m.L - 1;
    if (m.alpha < 0.0f && 2.0 * mu / -(double)m.alpha < d)
        d = 2.0 * mu / -(double)m.alpha;
    if ((double)m.alpha * d * d + 4.0 * mu * d - S > 117.0)
        return no;
    return (float)((double)m.cb + S);
}

bool seg_eligible(const DevModel &m)
{
    return !std::isnan(m.cbs);
}

cudaError_t launch_seg_table(const DevModel &m, float *out, cudaStream_t st)
{
    const SegTabJob j{m, out};
    return launch_seg_tables(&j, 1, st);
}

cudaError_t launch_seg_tables(const SegTabJob *jobs, int n, cudaStream_t st)
{
    for (int i = 0; i < n; ++i)
        if (!seg_eligible(jobs[i].m) || jobs[i].m.ta64 == nullptr)
            return cudaErrorInvalidValue;
    constexpr int kMost = 64;
    for (int i = 0; i < n; i += kMost) {
        const int k = n - i < kMost ? n - i : kMost;
        if (k == 1) {
            const SegTabJobs<1> one{{jobs[i]}};
            seg_table_kernel<1><<<kSegRows, kSegRow, 0, st>>>(one);
            continue;
        }
        SegTabJobs<kMost> many;
        std::copy(jobs + i, jobs + i + k, many.job);
        seg_table_kernel<kMost><<<dim3(kSegRows, k), kSegRow, 0, st>>>(many);
    }
    return cudaGetLastError();
}

cudaError_t launch_pca_seg(const SweepArgs &a, uint8_t *x0, uint8_t *x1,
                           const uint32_t *budget, cudaStream_t st)
{
    static int per_sm[64] = {};
    int cap = 0;
    cudaError_t e = resident(pca_seg_kernel, kSegThreads, per_sm, cap);
    if (e != cudaSuccess)
        return e;
    const int tiles_x = (a.W + kSX - 1) / kSX;
    const long long ntiles = (long long)tiles_x * ((a.H + kSY - 1) / kSY);
    if (ntiles >= (1ll << 30))
        return cudaErrorInvalidValue;
    const long long need = (ntiles + kSegWarps - 1) / kSegWarps;
    pca_seg_kernel<<<(int)(need < cap ? need : cap), kSegThreads, 0, st>>>(
        a, tiles_x, (int)ntiles, x0, x1, budget);
    return cudaGetLastError();
}

cudaError_t launch_gibbs_seg(const SweepArgs &a, int q, cudaStream_t st)
{
    static int per_sm[64] = {};
    int cap = 0;
    cudaError_t e = resident(gibbs_seg_kernel, kSegGibbsThreads, per_sm, cap);
    if (e != cudaSuccess)
        return e;
    const int tiles_x = (a.W + 2 * kSX - 1) / (2 * kSX);
    const long long ntiles = (long long)tiles_x * ((a.H + kSY - 1) / kSY);
    if (ntiles >= (1ll << 30))
        return cudaErrorInvalidValue;
    const long long need = (ntiles + kSegGibbsWarps - 1) / kSegGibbsWarps;
    gibbs_seg_kernel<<<(int)(need < cap ? need : cap), kSegGibbsThreads, 0, st>>>(a, q, tiles_x,
                                                                             (int)ntiles);
    return cudaGetLastError();
}

cudaError_t launch_pca_segw(const SweepArgs &a, uint8_t *x0, uint8_t *x1, int n,
                            unsigned int *done, unsigned int *grab, int *err, bool par_from_t,
                            const uint32_t *budget, cudaStream_t st)
{
    static int per_sm[64] = {};
    int cap = 0;
    cudaError_t e = resident(pca_segw_kernel, kSegwThreads, per_sm, cap);
    if (e != cudaSuccess)
        return e;
    const int tiles_x = (a.W + kSX - 1) / kSX, tiles_y = (a.H + kSY - 1) / kSY;
    const long long items = (long long)tiles_x * tiles_y * n;
    if (items >= (1ll << 32))
        return cudaErrorInvalidValue;
    // at most the resident capacity: every block that takes an item runs
    pca_segw_kernel<<<(int)(items < cap ? items : cap), dim3(kSX, kSY), 0, st>>>(
        a, x0, x1, n, tiles_x, tiles_y, done, grab, err, par_from_t ? 1 : 0, budget);
    return cudaGetLastError();
}

cudaError_t launch_gibbs_segw(const SweepArgs &a, uint8_t *x, int nsweeps,
                              unsigned int *done, unsigned int *grab, int *err, cudaStream_t st)
{
    static int per_sm[64] = {};
    int cap = 0;
    cudaError_t e = resident(gibbs_segw_kernel, kSegwThreads, per_sm, cap);
    if (e != cudaSuccess)
        return e;
    const int tiles_x = (a.W + 2 * kSX - 1) / (2 * kSX), tiles_y = (a.H + kSY - 1) / kSY;
    const long long items = (long long)tiles_x * tiles_y * 2 * nsweeps;
    if (items >= (1ll << 32))
        return cudaErrorInvalidValue;
    gibbs_segw_kernel<<<(int)(items < cap ? items : cap), dim3(kSX, kSY), 0, st>>>(
        a, x, 2 * nsweeps, tiles_x, tiles_y, done, grab, err);
    return cudaGetLastError();
}

}  // namespace pcad
