// kmc_internal.h -- shared declarations of the sm_103a kinetic Monte Carlo library
// (device tables, handle, kernel launchers).  Host code and kernels include it;
// nothing outside csrc/ does.
#pragma once

#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <string>

#include "../../include/kmc.h"

namespace kmc {

constexpr int kThreads = 256;          // threads per block of the particle kernels
constexpr int kScanThreads = 256;      // scan: threads per tile
constexpr int kScanItems = 16;         // scan: keys per thread (4 x uint4)
constexpr int kScanTile = kScanThreads * kScanItems;
constexpr uint32_t kSpinCap = 1u << 22;  // bounded waits: iterations before giving up
constexpr int kFoldCap = 64;           // wall folds per coordinate per step
constexpr int kAccFields = 10;         // per c-bin accumulator: N, Sum v (3), Sum v^2 (3), Sum W, collided
constexpr int kTestSlots = 256;        // counters of the pruned tile search's pair tests (blocks spread over them)
constexpr int kCbinRows = 4;           // rows of search cells per c-bin up to which moments go one warp per c-bin
constexpr int kPrunedCap = 1888;       // default staging capacity of the pruned tile search (28 B per slot)
                                       // count, Sum v.r_hat
constexpr int64_t kFineRows = 1 << 18;  // pruned instances from this many particles on: rows of finer cells
constexpr double kSymPassing = 64.0;   // filtered search: passing candidates per particle up to which a pair is tested once
constexpr double kPairsClose = 16.0;   // pair search: passing candidates per particle from which pairs are tested
                                       // against the closest so far
constexpr double kChiHits = 50.0;      // pairs per particle left by one filter from which it filters by criterion 1 too
constexpr int kMomStride = 18;         // per c-bin output: 8 raw, 8 derived, Sum v.r_hat and v_r (an array each)
constexpr uint32_t kCanonMax = 16384;  // search cells up to this many particles are put in id order

// device error flags (DevState::error)
constexpr uint32_t kErrScanTimeout = 1u;
constexpr uint32_t kErrKeyRange = 2u;

constexpr unsigned long long kNoPartner = ~0ull;  // partner key of a particle without candidate
// searches that no option asks for (InstDev::search)
constexpr int kSearchDirect = 0;       // one thread per particle
constexpr int kSearchFilter = 1;       // kmc_filter.cuh
constexpr int kSearchPairs = 2;        // kmc_pairs.cuh, binary32
constexpr int kSearchTile = 3;         // tile search, pruned on half c-bins (small single runs; InstDev::tiled)
constexpr int kMomItems = 4;           // moments: consecutive particles per thread
constexpr int kStageThreads = 256;     // staged search: threads per tile

// Per-instance constants.  Geometry (box, c-bins, walls) is shared; the search
// grid subdivision s[] and the interaction constants are per instance.
struct InstDev {
    int64_t p_off;       // first particle of the instance (global index)
    int64_t n;           // particles of the instance
    uint32_t key_base;   // first search-grid key of the instance
    uint32_t bin_base;   // first c-bin (moment row) of the instance
    int s[3];            // subdivision of a c-bin into search cells per dimension
    int M[3];            // search cells per dimension = n_cells * s
    double R2;           // squared contact distance
    double dt;           // timestep
    float R2f, dtf;      // the same rounded to binary32 (binary32 kernels use these)
    uint32_t seed_lo, seed_hi;
    double w[3];         // search-cell width per dimension
    // staged search (3-D, sparse search cells): tiles of tile_rows consecutive
    // y-rows of one x-slab; the tile's neighbourhood rows are copied to
    // shared memory before the search
    int staged;
    int tiled;           // search cells are the c-bins: one block per cell (tile_search_kernel)
    int prune;           // binary32: searched on cells finer than the c-bins, candidates out of reach skipped
    int search;          // kSearch...: its search, unless tiled or staged
    int chi;             // filtered search: criterion 1 filters too (the same for every instance of a handle)
    int sym;             // filtered search, binary32: each pair tested once, by its lower position
    int close;           // pair search: many candidates pass, pairs are tested against the closest so far
    int adaptive;        // timestep dx_min / v_max(t) per step (Sect. "Simulation setup")
    double dx_min;       // smallest c-bin width over the position dimensions
    int tile_rows;
    int tiles_per_x;     // ceil(M[1] / tile_rows)
    uint32_t tile_base;  // first tile of the instance in the staged launch
    // Lengths for the filtered search's constants in units of 1 / f_unit, the power of two that
    // puts the box's longest side in [1, 2): boxes of any size fit binary32 and binary16
    float f_unit, f_len;    // f_unit and 1 / f_unit
    int f64;                // binary64 state
    float f_L[3], f_cw[3];  // box, search cell widths
    float f_c, f_lmax, f_R; // largest coordinate, longest side, contact distance
};

// Per-instance quantities that change every step (written on the device).
struct InstDyn {
    unsigned long long vmax2_cur;   // bits of the largest |v|^2 (binary64) of the current state
    unsigned long long vmax2_next;  // accumulated by the step's move kernel
    double dt;                      // timestep of the next step (the configured one unless adaptive)
    double dt_prev;                 // timestep of the step just taken (virial pressure)
    double time;                    // simulated time since the state was set
    float dtf;                      // dt rounded to binary32
    int k[3];                       // search half-window in search cells
    int mom_e[3];                   // moment sums: fixed-point exponents of v, v^2 and W
    // filtered search (kmc_filter.cuh): frames of 2^f_shift search cells (at most all), coordinates
    // in units of 1 / f_scale (a power of two); the margins in the square of those units (f_g1,
    // f_c1, f_rt per unit of length)
    int f_shift[3];
    float f_w[3];                   // search cell widths (binary32)
    int f_image;                    // a window may hold a pair at more than half a periodic box
    float f_scale, f_dts;           // the scale, scale x timestep
    float f_g0, f_g1;               // a particle's share of F's margin: f_g0 + f_g1 |s|
    float f_c0, f_c1;               // the same of the margin of a and f
    float f_thr;                    // threshold at the contact distance
    float f_rt, f_slack;            // threshold at distance d (in those units): d^2 + f_rt d + f_slack
    float f_box;                    // widening of a home's swept box
    // pair search (kmc_pairs.cuh)
    int p_image;                    // a pair may meet at half a periodic box or more
    float p_slack;                  // rounding of a squared distance of closest approach, in the test against the closest so far
};

struct Geo {
    int dim;
    int vdim;   // velocity components: 3, or 2 (x, y only: the paper's 2-D runs)
    int n[3];
    int bc[3];
    double lo[3], hi[3], L[3], inv_dx[3];
    double rc[3];   // centre of the radial velocity moment
};

// The geometry in the state precision, a part of every kernel's parameters: its
// values come from the constant bank.  For walled dimensions the half length is
// +inf so the minimum-image shift never fires.
template <typename T>
struct GeoT {
    T lo[3], hi[3], inv[3], L[3], hL[3], rc[3];
    int n[3];
    bool wall[3];     // no periodic wrap: reflective or absorbing
    bool absorb[3];   // absorbing: a particle that ends a step outside is removed
    int vdim;
    void load(const Geo& g) {
        vdim = g.vdim;
        for (int d = 0; d < 3; ++d) {
            lo[d] = (T)g.lo[d];
            hi[d] = (T)g.hi[d];
            inv[d] = (T)g.inv_dx[d];
            L[d] = (T)g.L[d];
            wall[d] = g.bc[d] != 0;
            absorb[d] = g.bc[d] == 2;
            hL[d] = wall[d] ? (T)INFINITY : (T)0.5 * L[d];
            rc[d] = (T)g.rc[d];
            n[d] = g.n[d];
        }
    }
};

struct DevState {
    uint32_t step;        // Philox counter word 1 of the step being taken
    uint32_t error;       // kErr* bits
    uint32_t spin_cap;    // bounded waits: polls before giving up (0: kSpinCap)
    uint32_t hold_tile1;  // test of the bounded wait: scan tile hold_tile1 - 1 never publishes its
                          // status (0: none); set only through kmc_test_hold_scan
    uint32_t steps_left;  // steps still to take in the current graph-resident step loop
    uint32_t pad;
};

template <typename T>
struct Vec4;
template <>
struct Vec4<float> {
    using type = float4;
};
struct __align__(32) dvec4 {
    double x, y, z, w;
};
template <>
struct Vec4<double> {
    using type = dvec4;
};

// Pointers and sizes of one simulation, passed by value to every launcher.
template <typename T>
struct Bufs {
    using V = typename Vec4<T>::type;
    int64_t n;
    int n_inst;
    const InstDev* inst;     // [n_inst]
    InstDyn* dyn;            // [n_inst]
    DevState* st;
    Geo geo;
    GeoT<T> g;
    V* posA; V* velA;        // sorted state (search-grid key order)
    V* posB; V* velB;        // staging / unsorted end-of-step state
    unsigned long long* bkey;  // [n] partner key of A[p] (tag of the closest candidate, kNoPartner)
    uint32_t* slot_of;       // [n] by global id: sorted position in A (written by the search);
                             // the scatter reuses it for the tags of shared search cells
    uint32_t* key;           // [n] search key of B
    uint32_t* tagB;          // [n] tag of B[p], written with B (read coalesced by the scatter)
    uint32_t* slot;          // [n] rank of B[p] within its search cell
    uint32_t* count;         // [n_keys + 1] histogram (zero outside the step)
    uint32_t* start;         // [n_keys + 1] exclusive scan of count
    unsigned long long* scan_status;  // [1 + n_tiles]: ticket + tile descriptors
    uint32_t n_keys;
    uint32_t n_tiles;
    unsigned long long* acc; // [n_bins * kAccFields] moment sums, fixed point (two's complement)
    double* mom;             // raw [n_bins][8], derived [n_bins][8], radial [n_bins][2]
    double* glob;            // [n_inst * 8]
    int64_t n_bins;
    int32_t* rec_best;       // RECORD: [n] by global id
    int32_t* rec_partner;    // RECORD: [n] by global id
    int record;
    // staged search launch
    uint32_t n_stage_tiles;  // tiles over all staged instances (0: none)
    int stage_cap;           // candidate vectors a tile can stage
    int stage_rows;          // row slots of the staged start table
    int stage_stride;        // entries per row slot (max M[2] + 1, even)
    int stage_pair_cap;      // entries of the binary32 pair list
    int any_direct;          // some instance uses the direct (per-thread) search
    int any_tiled;           // some instance uses the tile search (one block per c-bin)
    int any_plain_tiled;     // some tiled instance searches on its c-bins (not pruned)
    int filtered;            // some instance is searched by the filtered search (kmc_filter.cuh)
    int paired;              // some instance is searched by lanes of homes against pairs (kmc_pairs.cuh): 1, or 3
                             // where many candidates pass
    int filter_chi;          // it also filters by criterion 1
    int filter_split;        // log2 of the warps that share a group of 32 homes
    int dsmc;                // the random-partner comparison variant instead of the PoCA search
    int radial;              // accumulate Sum v.r_hat (KMC_FLAG_RADIAL_MOMENT)
    int cbin_moments;        // every c-bin is at most kCbinRows runs of search cells: moments per c-bin
    int tile_threads;        // tile search: threads per c-bin block (a multiple of 32, 64 ... 256)
    int tile_cap;            // tile search: candidates staged in shared memory at once (even)
    int tile_split;          // tile search: blocks sharing one c-bin's window (binary32)
    int tile_prune;          // some instance uses the pruned tile search (binary32, half c-bins)
    unsigned long long* tile_tests;  // [kTestSlots] pair tests made by the pruned tile search (cumulative; may be null)
    // particle tag = (instance << id_bits) | instance-local id
    uint32_t id_bits;        // 32 when there is one instance
    uint32_t id_mask;
};

// Launchers (defined in kmc_kernels.cuh, instantiated per precision).
template <typename T>
cudaError_t launch_pack(const Bufs<T>& b, const T* pos3, const T* vel3, uint32_t* bad, cudaStream_t s);
template <typename T>
cudaError_t launch_bin_init(const Bufs<T>& b, cudaStream_t s);
template <typename T>
cudaError_t launch_search(const Bufs<T>& b, cudaStream_t s);       // staged + per-particle search
template <typename T>
cudaError_t launch_tile_search(const Bufs<T>& b, cudaStream_t s);  // one block per c-bin (tiled instances)
template <typename T>
cudaError_t launch_pairs_search(const Bufs<T>& b, cudaStream_t s);     // lanes of homes, pairs of candidates
template <typename T>
cudaError_t launch_filtered_search(const Bufs<T>& b, cudaStream_t s);  // tensor-core filter, every instance
template <typename T>
cudaError_t prepare_staged(const Bufs<T>& b);
template <typename T>
size_t stage_smem_bytes(const Bufs<T>& b);
template <typename T>
cudaError_t prepare_tile(const Bufs<T>& b);
template <typename T>
size_t tile_smem_bytes(const Bufs<T>& b);
template <typename T>
cudaError_t launch_move(const Bufs<T>& b, cudaStream_t s);
template <typename T>
cudaError_t launch_scatter(const Bufs<T>& b, cudaStream_t s);
template <typename T>
cudaError_t launch_gather_state(const Bufs<T>& b, T* pos3, T* vel3, cudaStream_t s);
template <typename T>
cudaError_t launch_cell_keys(const Bufs<T>& b, int32_t* keys, cudaStream_t s);
template <typename T>
cudaError_t launch_moments(const Bufs<T>& b, int use_virial, cudaStream_t s);
template <typename T>
cudaError_t launch_window_count(const Bufs<T>& b, unsigned long long* total, cudaStream_t s);
template <typename T>
cudaError_t launch_perm(const Bufs<T>& b, int32_t* perm, cudaStream_t s);
template <typename T>
cudaError_t launch_dsmc(const Bufs<T>& b, cudaStream_t s);     // random-partner collisions per c-bin
template <typename T>
cudaError_t launch_cbin_hist(const Bufs<T>& b, uint32_t* hist, unsigned long long* vmax2, double* sample, cudaStream_t s);

// Lengths of an instance for the filtered search (I.R2, I.w set).  A contact distance
// beyond 2^20 boxes lets every pair pass, as one of 2^20 boxes does.
inline void filter_lengths(InstDev& I, const Geo& g, bool binary64) {
    I.f64 = binary64;
    double lmax = 0.0, cmax = 0.0;
    for (int d = 0; d < g.dim; ++d) {
        lmax = fmax(lmax, g.L[d]);
        cmax = fmax(cmax, fmax(fabs(g.lo[d]), fabs(g.hi[d])));
    }
    const double unit = ldexp(1.0, -ilogb(lmax));
    I.f_unit = (float)unit;
    I.f_len = (float)ldexp(1.0, ilogb(lmax));
    for (int d = 0; d < 3; ++d) {
        I.f_L[d] = d < g.dim ? (float)(g.L[d] * unit) : 0.f;
        I.f_cw[d] = d < g.dim ? (float)(I.w[d] * unit) : 0.f;
    }
    I.f_c = (float)(cmax * unit);
    I.f_lmax = (float)(lmax * unit);
    I.f_R = (float)fmin(sqrt(I.R2) * unit, 0x1p20);
}

// Whether a binary64 instance's lengths and timestep fit the filtered search, whose
// operands and swept boxes are differences and products rounded to binary32 (their
// squares must fit too).  Otherwise it takes one thread per particle.
inline bool filter_fits(const InstDev& I, const Geo& g, double dt) {
    double lmax = 0.0;
    for (int d = 0; d < g.dim; ++d) lmax = fmax(lmax, g.L[d]);
    return lmax > 0x1p-40 && lmax < 0x1p40 && dt > 0x1p-60 && dt < 0x1p60;
}

#ifdef __CUDACC__
#define KMC_HOST_DEVICE __host__ __device__
#else
#define KMC_HOST_DEVICE
#endif
// Pieces of `size` positions, counted from position 0, that positions [q0, q1) touch.
// Positions go up to 2^31 - 2: nothing is rounded up past them.
KMC_HOST_DEVICE inline int32_t pieces_touched(int32_t q0, int32_t q1, int32_t size) {
    return q1 > q0 ? (q1 - 1) / size - q0 / size + 1 : 0;
}

// Particles the buffers of a state of n hold: whole groups of 32, so that the filtered
// search's operands of a last tile of 8, and that tile's box, lie inside them.
inline size_t buffer_rows(int64_t n) { return ((size_t)(n > 0 ? n : 1) + 31) / 32 * 32; }

// log2 of the warps that share a group of 32 homes of the filtered search: a
// small system has too few groups to fill the chip, so up to eight warps (a
// block) take one group, until about 16 warps per SM are busy.
inline int filter_split(int64_t n, int sms) {
    const int64_t groups = (n + 31) / 32;
    int s = 0;
    while (s < 3 && (groups << s) < (int64_t)sms * 16) ++s;
    return s;
}

// Counting-sort scatter of large cells (rank_cells_kernel): launches of it for a
// state of n particles over n_keys search cells.  Counting a cell's tags in the moving
// pass, and ranking them by a block, both scatter passes of 4M particles, ms, by
// particles per cell: 117 0.121 / 0.17, 169 0.139 / 0.15, 200 0.164 / 0.14, 400 0.254 / 0.12
// (64M: 40 1.40 / 2.47, 64 1.57 / 2.98).  A launch costs each cell it leaves alone 0.5 ns, so
// it is made where a mean cell is nearly large enough.
constexpr uint32_t kRankMin = 192;       // cells up to this many particles: the moving pass counts
constexpr int kRankCap = 4096;           // the first launch's largest cell (32 KiB of shared memory)
constexpr int64_t kRankMean = 160;       // mean particles per cell from which the first launch runs
constexpr int64_t kRankMeanLarge = 1024; // and from which the second runs, for cells up to kCanonMax
inline int rank_launches(int64_t n, uint32_t n_keys) {
    const int64_t mean = n_keys > 0 ? n / (int64_t)n_keys : 0;
    return mean >= kRankMeanLarge ? 2 : mean >= kRankMean ? 1 : 0;
}

// Estimated costs of the three searches of a binary32 instance in ps per particle (binary64 below),
// fitted on a GB300 to 36 states (slab tubes of 0.3M-16M particles with R from one to
// sixty c-bins, 2-D implosions and quadrants, 3-D blasts).  `cand`: candidates in
// a particle's window; `hits`: those that pass the filter; `passing`: those that meet;
// `rows`: rows of search cells in the window; `n_row`: particles in a row of cells.
// Measured / estimated, one thread per particle, filtered, pairs:
//   16M slab tube, 14 candidates    70 / 88     - / 191    161 / 178
//   4M slab, 206                   370 / 338  287 / 273    238 / 214
//   4M slab, 469                   623 / 680  232 / 222    321 / 299
//   2-D Noh, 189                   183 / 186  604 / 372    102 / 133
//   2-D quadrants, 2427              -       1665 / 1756   938 / 927
//   3-D blast, 246                 260 / 254  150 / 182    199 / 208
// One thread per particle takes longer where c-bins are split (`split`: shorter rows).
// To these come the times of a single walk, which small handles (`n_all` particles)
// take whole; us measured / estimated for tubes of 10,000-110,000 particles: 10 candidates
// 23 / 23, 93-170 / 85-120, 46-54 / 36-40; 223 candidates 115 / 119, 69 / 76, 51 / 69. A
// window that may reach around a periodic box (`wraps`) makes the pair search decide
// every pair exactly (4,900 particles, 440 candidates: 138 us, 113, 1240).
// A warp's homes test the union of their windows, 32 particles more per row, and a
// warp whose homes lie in several rows walks once per row (`runs`).  `walks`: frame blocks
// that a warp of the filtered search visits in all (walk_blocks); up to ten are in the fit
// above.  Particles spread thinly beside a dense cluster, with contact distance and
// displacement far below a cell, make hundreds: 2.1M particles, 260 candidates 19.0 ms filtered,
// 0.67 one thread per particle (without this term the filter was chosen).
struct SearchCosts {
    double ps[3];           // kSearchDirect, kSearchFilter, kSearchPairs
    bool tile = false;      // a small single run whose tile search costs less than any of them
};
inline double walk_cost(double walks, double n_all) { return walks > 10.0 ? (10.0 + 1.5e6 / n_all) * (walks - 10.0) : 0.0; }
inline SearchCosts search_costs(int dim, bool split, bool wraps, double n_all, double cand, double hits, double passing,
                                double rows, double n_row, double walks) {
    const double tests = cand + 32.0 * rows, runs = 1.0 + 32.0 / (n_row > 1.0 ? n_row : 1.0);
    SearchCosts c;
    c.ps[kSearchDirect] = dim == 2 ? 25.0 + 0.85 * cand : split ? 70.0 + 1.3 * cand : 45.0 + 0.85 * cand;
    c.ps[kSearchFilter] = (130.0 + 0.07 * cand + 6.0 * hits) * runs;
    c.ps[kSearchPairs] = (dim == 3 ? 38.0 + 0.30 * tests : 24.0 + 0.28 * tests) * runs + 3.0 * (passing < 64.0 ? passing : 64.0);
    c.ps[kSearchDirect] += (20.0 + 0.27 * cand) * 1e6 / n_all;
    c.ps[kSearchFilter] += (45.0 + 10.0 * runs + 0.3 * hits) * 1e6 / n_all + walk_cost(walks, n_all);
    c.ps[kSearchPairs] += (35.0 + 0.04 * cand) * 1e6 / n_all;
    if (wraps) c.ps[kSearchPairs] *= 20.0;
    return c;
}
// Binary64: one thread per particle or filtered, per particle of a handle of n_all.  Up to
// some 100,000 particles a search is about one wave, its time that of a particle's walk or
// of a group's runs and frame blocks; fitted to 410 states of 2,000-100,000 particles.  us per
// search, measured / estimated, one thread per particle and filtered: 2-D, 20,000 particles, 13
// candidates, 3 blocks 30 / 41, 85 / 65; 3-D, 5,600, 55, 8 blocks 95 / 112, 110 / 104; above, slab
// tubes: 1M, 11, 33 per row 1190 / 1270, 940 / 950; 1M, 67, 65 per row 4600 / 4800, 1000 / 910.
// `runs` here is the mean over the particles (few per row count fully).
inline SearchCosts search_costs64(int dim, double n_all, double cand, double n_row, double runs, double walks) {
    const double L = 1e6 / n_all;
    SearchCosts c;
    if (n_all < 1e5) {
        c.ps[kSearchDirect] = dim == 3 ? (55.0 + 0.9 * cand) * L + 80.0 + 24.0 * cand : (20.0 + 0.84 * cand) * L + 20.0 + 24.0 * cand;
        c.ps[kSearchFilter] = dim == 3 ? (76.0 + 3.0 * runs + 1.9 * walks) * L + 360.0 + 66.0 * walks
                                       : (40.0 + 3.0 * walks) * L + 320.0 * runs + 4.4 * cand;
    } else {
        c.ps[kSearchDirect] = (45.0 + 3.4 * cand) * L + 500.0 + 60.0 * cand;
        c.ps[kSearchFilter] = 75.0 * (1.0 + 32.0 / (n_row > 1.0 ? n_row : 1.0)) * L + 800.0 + walk_cost(walks, n_all);
    }
    c.ps[kSearchPairs] = c.ps[kSearchDirect] + c.ps[kSearchFilter];   // binary32 only
    return c;
}
// Frame blocks that a warp of the filtered search walks, over all its runs of homes: the
// frames as the step's constants set them (kmc_scan.cu, filter_constants), n_row homes
// per row of search cells, spread over its length.
inline double walk_blocks(const InstDev& I, const Geo& g, bool chi, double s, double n_row) {
    const int F = g.dim - 1;
    const double R = sqrt(I.R2), D = R + 2.0 * s, Re = I.sym ? R : 0.125 * R;
    double reach = 0.0;
    for (int d = 0; d <= F; ++d) reach = fmax(reach, fmin(D, 2.0 * I.s[d] * I.w[d]));
    const double width = 2.0 * ((chi ? fmin(200.0 * R, 400.0 * s) : 46.0 * sqrt(Re * Re + s * s / 16.0)) - reach - s);
    const double rows = fmax(n_row, 1e-3);
    double blocks = 1.0 + 32.0 / rows;   // runs
    for (int d = 0; d <= F; ++d) {
        int sh = 0;
        while ((1 << sh) < I.M[d] && fmin(2 << sh, I.M[d]) * I.w[d] <= width) ++sh;
        const double k = ceil((1.001 * D + 1e-5 * g.L[d]) / I.w[d]), M = (double)I.M[d];
        double cells = fmin(2.0 * k + 1.0, fmin(3 * I.s[d], I.M[d]));
        if (d == F) cells = fmin(cells + fmin(1.0, 32.0 / rows) * M, M + 1.0);
        blocks *= 1.0 + (cells - 1.0) / fmin(1 << sh, M);
    }
    return blocks;
}

// the cheapest of the searches in `allowed` (a bit each)
inline int cheapest_search(const SearchCosts& c, unsigned allowed) {
    int best = -1;
    for (int k = 0; k < 3; ++k)
        if ((allowed >> k & 1u) && (best < 0 || c.ps[k] < c.ps[best])) best = k;
    return best;
}

// precision-independent
cudaError_t launch_scan(uint32_t* count, uint32_t* start, uint32_t n_keys, uint32_t n_tiles,
                        unsigned long long* status, InstDyn* dyn, const InstDev* inst,
                        int n_inst, DevState* st, Geo geo, int bump_step, cudaStream_t s);
// gacc: [n_inst * 8] integer totals, zero between calls (the launch leaves it zero)
cudaError_t launch_finalize(const InstDev* inst, const InstDyn* dyn, int n_inst, Geo geo,
                            const unsigned long long* acc, double* mom, double* glob, unsigned long long* gacc,
                            int64_t n_bins, cudaStream_t s);

}  // namespace kmc
