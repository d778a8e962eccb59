// Tile-resident sweeps (tile.cu): host interface.
#pragma once

#include "pcad_internal.h"

namespace pcad {

// The draw of a tile-resident launch and its template instance.
struct TileKind {
    enum Draw { kSmall, kSegment, kBinary };
    Draw draw = kSmall;
    int nbhd = 4;
    bool gibbs = false;
    int lmax = 0;          // kSmall: 8 or 16 labels evaluated, masked at L
    bool mask = false;
    bool operator==(const TileKind &o) const
    {
        return draw == o.draw && nbhd == o.nbhd && gibbs == o.gibbs && lmax == o.lmax &&
               mask == o.mask;
    }
};

struct TileGeom {
    int th, twq;          // rows and quads (4-site words) per tile
    int tiles_x, tiles_y;
    int k;                // sweeps per exchange
    int h, hq;            // halo: rows (and columns), words
    int threads;          // per CTA
    bool two;             // two CTAs per SM
    bool compact;         // two labels: no staged uniforms, byte counts
};

struct TilePlan {
    TileGeom tg;
    int ctas;
};

// One chain of a launch.  Its sweeps are those at *a.sweep_base + a.sweep_off
// on (up to *budget, if set); planes x0 -> x1 (the same one for Gibbs or an
// even count), or x0 / x1 by the parity of the sweep index (par_from_t).
struct TileJob {
    SweepArgs a;
    uint8_t *x0, *x1;
    const uint32_t *budget;
    unsigned long long *xch;   // border exchange, tile_xch_bytes, no stale tags
    int par_from_t;
    int cta0;                  // first CTA of the chain
    TileGeom tg;
};

// A launch's chains (kernel parameters; small launches keep them small).
constexpr int kTileJobs = 32;
template <int N>
struct TileLaunchT {
    int nsweeps, njobs;
    int *err;                  // set when a bounded wait runs out
    TileJob job[N];
};
using TileLaunch = TileLaunchT<1>;
using TilePack = TileLaunchT<kTileJobs>;
static_assert(sizeof(TilePack) <= 32000, "kernel parameter space");

// The launch kind of a model (false: not taken).  Its tables must be in place
// at the launch: m.ptab (small), m.stab (segment) or m.btab (two labels);
// small and two-label observations are checked against L.
bool tile_kind(const DevModel &m, bool gibbs, TileKind &k);
// Tiles of an image alone on the device, or on at most `ctas` CTAs with two
// or one per SM; false when they do not fit.
bool tile_plan(const TileKind &k, int H, int W, int sms, TilePlan &p);
bool tile_plan_ctas(const TileKind &k, int H, int W, int ctas, bool two, TileGeom &tg);
size_t tile_xch_bytes(int H, int W);
// One cooperative launch of `ctas` CTAs (all the jobs' tiles).
cudaError_t launch_tile(const TileKind &k, const TileLaunch &L, int ctas, cudaStream_t s);
cudaError_t launch_tile(const TileKind &k, const TilePack &L, int ctas, cudaStream_t s);
// Chains, batches and the server take tile-resident launches for images of at
// most this many sites.
constexpr long long kTileMaxSites = 1ll << 20;
// Two-label PCA chains: as long as their tiles fit (about 50000 sites per SM;
// tiles above 8192 sites are compact, for runs of at least kTileCompactSweeps).
constexpr long long kTileMaxBinarySites = 8ll << 20;
constexpr int kTileCompactSweeps = 16;

}  // namespace pcad
