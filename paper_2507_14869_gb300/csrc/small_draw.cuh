// The small-label draw (3 <= L <= 16, Section 5.2, Eq.
// posterior_pca_transition_matrix): prior sums of all labels from a table of
// neighbour pairs, weights two labels per packed FP32x2 instruction, inverse
// CDF over chunks of 4 labels with the per-site certified margin.  Shared by
// the small-label sweep (small.cu) and the TMA-tiled k-sweep kernel (tb.cu).
#pragma once

#include "pcad_internal.h"

namespace pcad {
namespace sld {

constexpr int kCodes = 17;                       // labels 0..15 and "missing"
constexpr int kPtabWords = kCodes * kCodes * 4;  // 16 bytes per pair
constexpr int kPrefixStride = 20;                // floats per thread row (conflict-free)
constexpr int kAqStride = 20;                    // floats per row of the data-term table

// Row g of the data-term table: fl(alpha (g - s)^2) for s = 0..15 (observations
// g < 16; every chain checks g < L at creation).
__device__ __forceinline__ void fill_aq(const DevModel &m, float *aq, int tid, int nthreads)
{
    for (int i = tid; i < 16 * 16; i += nthreads) {
        const int g = i >> 4, sl = i & 15;
        aq[g * kAqStride + sl] = __fmul_rn(m.alpha, (float)((g - sl) * (g - sl)));
    }
}

// The draw of one site from its neighbour codes nc[] and observation g (below
// 16).  Returns the label; `certain` is false when the uniform lies within the
// certified margin of an end of the chosen label's CDF interval, or of 0 or Z
// (the caller re-draws it in FP64).  pt: the pair table in shared memory; pre:
// this thread's row of shared memory (kPrefixStride floats), which receives
// the weights; aq: the data-term table (fill_aq): the exponent is
// fl(gam P + fl(alpha q)), both terms non-positive, so within 3u |v| of the
// exact one, the per-site margin's bound.
//
// The inertia atom delta is added to w(x_i) in the thread's row and to the
// chunk prefixes at and above x_i's chunk, so neither the chunk nor the label
// search looks at x_i again.  Roundings: chunk sums 2, chunk prefix 3, delta's
// join 1, the label prefix 4 and w(x_i) + delta 1: every C_k within 11u, Z
// within 6u, t 1u, inside the 22u of summation in the margin.  A chunk chosen
// off by one through these roundings leaves t within a few u Z of the tested
// interval's end, inside the margin.
template <int LMAX, int NB, bool MASK>
__device__ __forceinline__ int draw_small(const DevModel &m, const uint32_t *pt, const int (&nc)[NB],
                                          int g, int xi, uint32_t ub, float *pre, bool &certain,
                                          const float *aq)
{
    constexpr int NW = LMAX / 4;      // table words used per pair = chunks of 4 labels
    uint32_t P[NW];
    {
        const int e0 = (nc[0] * kCodes + nc[1]) * 4;
        const int e1 = (nc[2] * kCodes + nc[3]) * 4;
        if constexpr (NW == 4) {
            uint4 a = *reinterpret_cast<const uint4 *>(pt + e0);
            const uint4 b = *reinterpret_cast<const uint4 *>(pt + e1);
            a.x += b.x;
            a.y += b.y;
            a.z += b.z;
            a.w += b.w;
            if constexpr (NB == 8) {
                const uint4 c = *reinterpret_cast<const uint4 *>(pt + (nc[4] * kCodes + nc[5]) * 4);
                const uint4 d = *reinterpret_cast<const uint4 *>(pt + (nc[6] * kCodes + nc[7]) * 4);
                a.x += c.x + d.x;
                a.y += c.y + d.y;
                a.z += c.z + d.z;
                a.w += c.w + d.w;
            }
            P[0] = a.x;
            P[1] = a.y;
            P[2] = a.z;
            P[3] = a.w;
        } else {
            uint2 a = *reinterpret_cast<const uint2 *>(pt + e0);
            const uint2 b = *reinterpret_cast<const uint2 *>(pt + e1);
            a.x += b.x;
            a.y += b.y;
            if constexpr (NB == 8) {
                const uint2 c = *reinterpret_cast<const uint2 *>(pt + (nc[4] * kCodes + nc[5]) * 4);
                const uint2 d = *reinterpret_cast<const uint2 *>(pt + (nc[6] * kCodes + nc[7]) * 4);
                a.x += c.x + d.x;
                a.y += c.y + d.y;
            }
            P[0] = a.x;
            P[1] = a.y;
        }
    }
    const float2 g2 = make_float2(m.gam, m.gam);
    const float2 off2 = make_float2(-8388608.0f, -8388608.0f);
    const float4 *aqr = reinterpret_cast<const float4 *>(aq + g * kAqStride);
    const float gf = __uint_as_float(0x4B000000u + (uint32_t)g) - 8388608.0f;
    const float2 gf2 = make_float2(gf, gf), al2 = make_float2(m.alpha, m.alpha);
    float S[NW];
#pragma unroll
    for (int c = 0; c < NW; ++c) {
        const uint32_t p = P[c];
        // fl(alpha (g - s)^2): half the chunks from the table, half computed (the
        // same bits), between the shared-memory and the issue limits: 8192^2 549
        // -> 538 us per sweep, 1024^2 11.3 -> 10.9; all computed 561 and 11.1
        float4 q;
        if (c < (NW + 1) / 2) {
            q = aqr[c];
        } else {
            const float2 da = __fadd2_rn(gf2, make_float2(-(float)(4 * c), -(float)(4 * c + 1)));
            const float2 db = __fadd2_rn(gf2, make_float2(-(float)(4 * c + 2), -(float)(4 * c + 3)));
            const float2 qa = __fmul2_rn(al2, __fmul2_rn(da, da));
            const float2 qb = __fmul2_rn(al2, __fmul2_rn(db, db));
            q = make_float4(qa.x, qa.y, qb.x, qb.y);
        }
        // bytes to floats: the byte in the mantissa of 2^23, less 2^23
        const float2 p0 = __fadd2_rn(
            make_float2(__uint_as_float(__byte_perm(p, 0x4B000000u, 0x7440u)),
                        __uint_as_float(__byte_perm(p, 0x4B000000u, 0x7441u))), off2);
        const float2 p1 = __fadd2_rn(
            make_float2(__uint_as_float(__byte_perm(p, 0x4B000000u, 0x7442u)),
                        __uint_as_float(__byte_perm(p, 0x4B000000u, 0x7443u))), off2);
        const float2 v0 = __ffma2_rn(g2, p0, make_float2(q.x, q.y));
        const float2 v1 = __ffma2_rn(g2, p1, make_float2(q.z, q.w));
        float2 w0 = make_float2(ex2_ftz(v0.x), ex2_ftz(v0.y));
        float2 w1 = make_float2(ex2_ftz(v1.x), ex2_ftz(v1.y));
        if (MASK) {
            w0.x = 4 * c < m.L ? w0.x : 0.0f;
            w0.y = 4 * c + 1 < m.L ? w0.y : 0.0f;
            w1.x = 4 * c + 2 < m.L ? w1.x : 0.0f;
            w1.y = 4 * c + 3 < m.L ? w1.y : 0.0f;
        }
        reinterpret_cast<float4 *>(pre)[c] = make_float4(w0.x, w0.y, w1.x, w1.y);
        const float2 h = __fadd2_rn(w0, w1);
        S[c] = __fadd_rn(h.x, h.y);
    }
    // the inertia atom joins w(x_i) in the row and the prefixes from its chunk on
    float delta = 0.0f;
    if (m.em1 != 0.0f) {
        const float wx = pre[xi];
        delta = __fmul_rn(wx, m.em1);
        pre[xi] = __fadd_rn(wx, delta);
    }
    float G[NW];
    G[0] = S[0];
#pragma unroll
    for (int c = 1; c < NW; ++c)
        G[c] = __fadd_rn(G[c - 1], S[c]);
#pragma unroll
    for (int c = 0; c < NW; ++c)
        G[c] = 4 * c + 3 >= xi ? __fadd_rn(G[c], delta) : G[c];   // (always for the last)
    const float Z = G[NW - 1];
    const float t = __fmul_rn((float)ub, __fmul_rn(Z, 1.0f / 16777216.0f));
    // site_margin times Z
    const float margin =
        __fmaf_rn(__fmaf_rn(m.kb1, __fsub_rn(m.hb, lg2_ftz(Z)), m.kb0), Z, m.kbr * delta);
    int cs = 0;
    float Gp = 0.0f;
#pragma unroll
    for (int c = 0; c + 1 < NW; ++c) {
        const bool below = G[c] <= t;
        cs += below ? 1 : 0;
        Gp = below ? G[c] : Gp;
    }
    const float4 wc = reinterpret_cast<const float4 *>(pre)[cs];
    const float C0 = __fadd_rn(Gp, wc.x), C1 = __fadd_rn(C0, wc.y), C2 = __fadd_rn(C1, wc.z),
                C3 = __fadd_rn(C2, wc.w);
    const bool b0 = C0 <= t, b1 = C1 <= t, b2 = C2 <= t;
    const float hiC = b2 ? C3 : (b1 ? C2 : (b0 ? C1 : C0));
    const float loC = b2 ? C2 : (b1 ? C1 : (b0 ? C0 : Gp));
    certain = fminf(__fsub_rn(hiC, t), __fsub_rn(t, loC)) > margin;
    return 4 * cs + (int)b0 + (int)b1 + (int)b2;
}

}  // namespace sld
}  // namespace pcad
