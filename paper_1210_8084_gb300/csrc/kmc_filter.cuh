// kmc_filter.cuh -- closest-candidate search with a tensor-core filter.
//
// The acceptance test (criteria 1-2) of a pair with separation r0 at the start
// of the step and r1 = r0 + v_rel dt at its end under free flight implies
//
//     F = r0 . r1 < R^2 :
//
// with a = r0 . v, b = |v|^2 it asks a < 0, a + b dt > 0 and a^2 - b (|r0|^2 -
// R^2) >= 0, so |r0|^2 <= R^2 + a^2 / b and F = |r0|^2 + a dt <= R^2 + (a / b)
// (a + b dt) < R^2.  A pair whose distance of closest approach d^2 = |r0|^2 -
// a^2 / b is below the home's closest so far has F < d^2 by the same algebra, so
// that value may stand in for R^2.  F is bilinear in the two particles' (x, y),
// y = x + v dt:
//
//     F = x_i.y_i + x_j.y_j - x_i.y_j - y_i.x_j,
//
// a product whose sign one m16n8k16 tensor instruction gives for 128 pairs.  Only
// pairs with F below the threshold (a few per home where the plain search tests
// thousands) go to the exact test, so the decisions, and with them every result,
// are those of the exact test alone.
//
// Rounding.  Coordinates are taken relative to a frame (a block of search
// cells), scaled by a power of two and rounded to binary16 (the middle of a path
// to two halves); homes and candidates of a frame block share its centre.  With a
// separation component off by E, F is off by at most sqrt(3) E (|r0| + |r1|) +
// 3 E^2, and |r0| + |r1| <= 2 d + (|v_i| + |v_j|) dt for a pair that passes; the
// form with the middle of the paths likewise.  The threshold is raised by that
// bound, split into a share of each particle, by the rounding of the exact test
// itself (a pair it accepts has F <= R^2 + 45 u |r0| (|r0| + |v_rel| dt), u = 2^-24,
// below 2^-17 D^2 with D the reach R + 2 v_max dt) and by that of the product's
// sum (16 terms of 12 X^2 in all: 2^-18 of it).  kmc_scan.cu holds the constants.
//
// Bound by instruction issue (71 % of the slots, 9,900 instructions per 32 homes of the
// 16M tube).  The searches it replaced -> this one, GB300, ms per step: 3-D Sod tube,
// 512M particles 423 -> 191, 16M 14.6 -> 6.3, 21M at 20 per c-bin 25.0 -> 3.6; Sedov
// blast, 8M 15.3 -> 1.14; binary64 slab tube, 200k 2.33 -> 0.26.  Per 32 homes of the 16M
// tube: 431 tiles of 8 candidates in the window, 135 past the box check, 411 pairs
// past the filter.
#pragma once

#include "kmc_kernels.cuh"

namespace kmc {

constexpr int kFiltTile = 8;      // candidates per tile (columns of one tensor instruction)
constexpr int kFiltChunk = 4;     // tiles filtered at a time
constexpr int kFiltList = 36;     // listed tiles: 3 left of a round and 32 of the next, a multiple of 4
constexpr int kFiltQueue = 64;    // queued words of surviving pairs, one per lane and chunk (a power of two)
constexpr int kFiltChunks = 32;   // chunks whose words may be queued or in test (a power of two)
constexpr uint32_t kTilePart = 0x80000000u;   // listed tile that reaches past its row's range
constexpr uint32_t kTileOwn = 0x40000000u;    // listed tile that holds some of the homes (symmetric search)
constexpr uint32_t kTileMask = 0x0fffffffu;   // its number (below 2^28: fewer than 2^31 particles)
constexpr float kNoHit = 60000.f;             // own term of a row that has no pair: no sum falls below zero; with the
                                              // sign flipped, of one whose margin lets every pair pass

__device__ __forceinline__ uint32_t pack_half2(float a, float b) { return half2_bits(__floats2half2_rn(a, b)); }
__device__ __forceinline__ float2 unpack_half2(uint32_t u) {
    __half2 h;
    memcpy(&h, &u, sizeof(h));
    return __half22float2(h);
}
// x as two halves, high and low part
__device__ __forceinline__ uint32_t split_half2(float x) {
    const __half h = __float2half_rn(x);
    return half2_bits(__halves2half2(h, __float2half_rn(x - __half2float(h))));
}

// Coordinate of a frame's centre (half of c2 search cells from the low wall, any
// image) along dimension d.
__device__ __forceinline__ float frame_centre(const GeoT<float>& G, const InstDev&, const InstDyn& D, int d, int c2) {
    return fmaf(0.5f * (float)c2, D.f_w[d], G.lo[d]);
}
__device__ __forceinline__ double frame_centre(const GeoT<double>& G, const InstDev& I, const InstDyn&, int d, int c2) {
    return G.lo[d] + 0.5 * (double)c2 * I.w[d];
}

// A particle's path along one dimension in a frame of centre `ctr`: coordinate X and
// displacement S in the frame's units; xf and sf the same for the swept boxes.  Those
// are in binary32's coordinates, `image` lower; in binary64 from the low wall on, the
// centre at `off` (a box far from the origin would lose its digits).
struct Path1 {
    float X, S, xf, sf;
};
__device__ __forceinline__ Path1 path_in_frame(const InstDyn& D, float x, float v, float ctr, float image, float) {
    return Path1{(x - ctr) * D.f_scale, v * D.f_dts, x - image, v * D.dtf};
}
__device__ __forceinline__ Path1 path_in_frame(const InstDyn& D, double x, double v, double ctr, double, float off) {
    const float xc = (float)(x - ctr), vf = __double2float_rz(v);   // rz: a speed out of range stays finite
    return Path1{xc * D.f_scale, vf * D.f_dts, xc + off, vf * D.dtf};
}

// A particle's operands in a frame from its coordinates X and displacement S in
// the frame's units, as a candidate (columns of B) or a home (rows of A), with its
// own terms in two halves (high, low).  The product is of depth 16; lane 4 r + q of
// a warp supplies the words q (halves 2 q, 2 q + 1) and q + 4 of row or column r.
// The sum starts at zero: a home's own term is a product with ones.
//
// One filter: F = |dm|^2 - |dh|^2 with m = x + h, h = s / 2 the middle of the
// path, m in two halves (the product of the low parts is left to the margin):
//   A: 2 mh | 2 mh | 2 ml | 2 h | 1 1 | N - threshold
//   B: -mh  | -ml  | -mh  | h   | N   | 1 1
// Three filters, in x, y = x + s and s; words 0-2 hold one dimension each:
//   F: A (-y, -x) x 3 | 1 1 | N - threshold | 0    | 0 | 0,  B (x, y) x 3 | N   | 1 1 | 0   | 0 | 0
//   a: A (-s, -x) x 3 | 1 1 | 0             | Na   | 0 | 0,  B (x, s) x 3 | Na  | 0   | 1 1 | 0 | 0
//   f: A (-s, -y) x 3 | 0   | 1, Nf high    | 1, Nf low | 0 | 0,
//      B (y, s) x 3   | .   | Nf high, 1    | Nf low, 1 | 0 | .
__device__ __forceinline__ uint32_t lo_lo(uint32_t a, uint32_t b) { return __byte_perm(a, b, 0x5410); }
__device__ __forceinline__ uint32_t hi_lo(uint32_t a, uint32_t b) { return __byte_perm(a, b, 0x5432); }
constexpr uint32_t kNegHalves = 0x80008000u;   // flips the sign of both halves
constexpr uint32_t kOneOne = 0x3c003c00u;      // (1, 1)

struct PathTerms {   // one filter
    uint32_t mh01, mh2, ml01, ml2, h01, h2;
    float N;   // |m|^2 - |h|^2 of the rounded values
};
__device__ __forceinline__ PathTerms path_terms(const float X[3], const float S[3]) {
    PathTerms t;
    float m[3], N = 0.f;
#pragma unroll
    for (int d = 0; d < 3; ++d) m[d] = fmaf(0.5f, S[d], X[d]);
    t.mh01 = pack_half2(m[0], m[1]);
    t.mh2 = pack_half2(m[2], 0.f);
    const float2 a = unpack_half2(t.mh01), c = unpack_half2(t.mh2);
    t.ml01 = pack_half2(m[0] - a.x, m[1] - a.y);
    t.ml2 = pack_half2(m[2] - c.x, 0.f);
    const float2 al = unpack_half2(t.ml01), cl = unpack_half2(t.ml2);
    t.h01 = pack_half2(0.5f * S[0], 0.5f * S[1]);
    t.h2 = pack_half2(0.5f * S[2], 0.f);
    const float2 u = unpack_half2(t.h01), v = unpack_half2(t.h2);
    const float m0 = a.x + al.x, m1 = a.y + al.y, m2 = c.x + cl.x;
    N = fmaf(m2, m2, fmaf(m1, m1, m0 * m0));
    t.N = N - fmaf(v.x, v.x, fmaf(u.y, u.y, u.x * u.x));
    return t;
}
__device__ __forceinline__ uint32_t times2(uint32_t h2) {
    __half2 h;
    memcpy(&h, &h2, sizeof(h));
    return half2_bits(__hadd2(h, h));
}

struct ChiTerms {   // three filters
    uint32_t xy[3], s[3];   // (x_d, y_d); s_d in the low half
    float xy_, xs, ys;      // x.y, x.s, y.s of the rounded values
};
__device__ __forceinline__ ChiTerms chi_terms(const float X[3], const float S[3]) {
    ChiTerms t;
    t.xy_ = t.xs = t.ys = 0.f;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        t.xy[d] = pack_half2(X[d], X[d] + S[d]);
        t.s[d] = pack_half2(S[d], 0.f);
        const float2 c = unpack_half2(t.xy[d]);
        const float u = unpack_half2(t.s[d]).x;
        t.xy_ = fmaf(c.x, c.y, t.xy_);
        t.xs = fmaf(c.x, u, t.xs);
        t.ys = fmaf(c.y, u, t.ys);
    }
    return t;
}

// Candidate operands, swept boxes of 8 consecutive candidates and the sorted
// position of every particle by id.  The unsorted state's buffers are free
// during the search: the operands go to posB and velB (16 bytes per particle
// each), the boxes (the union of the tile's paths x .. x + s: lo, then hi, 32
// bytes per tile) to key.
template <typename T, int DIM, bool CHI>
__global__ void __launch_bounds__(kThreads) filter_prep_kernel(Bufs<T> b) {
    using V = typename Vec4<T>::type;
    const GeoT<T>& G = b.g;   // kernel parameter: constant bank
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const bool valid = p < b.n;
    float lo[3], hi[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        lo[d] = R<float>::inf();
        hi[d] = -R<float>::inf();
    }
    uint4 op = make_uint4(0u, 0u, 0u, 0u), op2 = op;
    V P = {}, Q = {};
    int inst = 0;
    if (valid) {
        P = b.posA[p];
        Q = b.velA[p];
        inst = tag_inst(b, R<T>::bits(P.w));
    }
    const InstDev& I = b.inst[inst];
    const InstDyn& D = b.dyn[inst];
    if (valid && I.search == kSearchFilter) {
        const uint32_t tag = R<T>::bits(P.w);
        // sorted position by id, read by the move kernel to find a partner
        b.slot_of[I.p_off + (int64_t)tag_id(b, tag)] = (uint32_t)p;
        const T x[3] = {P.x, P.y, P.z}, v[3] = {Q.x, Q.y, Q.z};
        float X[3] = {0.f, 0.f, 0.f}, S[3] = {0.f, 0.f, 0.f}, s2 = 0.f;
#pragma unroll
        for (int d = 0; d < DIM; ++d) {
            int c, g;
            cell_and_search<T>(x[d], G.lo[d], G.inv[d], G.n[d], I.s[d], c, g);
            const int sh = D.f_shift[d];
            const int c2 = (((g >> sh) * 2) << sh) + min(1 << sh, I.M[d]);
            const Path1 w = path_in_frame(D, x[d], v[d], frame_centre(G, I, D, d, c2), (T)0, 0.5f * (float)c2 * D.f_w[d]);
            X[d] = w.X;
            S[d] = w.S;
            s2 += S[d] * S[d];
            lo[d] = fminf(w.xf, w.xf + w.sf);
            hi[d] = fmaxf(w.xf, w.xf + w.sf);
        }
        const float sl = sqrtf(s2);
        const float share = fmaf(D.f_g1, sl, D.f_g0);   // this particle's share of the margin
        if constexpr (CHI) {
            const ChiTerms t = chi_terms(X, S);
            const float c = fmaf(D.f_c1, sl, D.f_c0);
            const uint32_t nf = split_half2(fminf(t.ys + c, kNoHit));
            op = make_uint4(t.xy[0], t.xy[1], t.xy[2], split_half2(t.xy_ - share));
            op2 = make_uint4(lo_lo(t.s[0], nf), lo_lo(t.s[1], nf >> 16), t.s[2], split_half2(fmaxf(t.xs - c, -kNoHit)));
        } else {
            const PathTerms t = path_terms(X, S);
            const uint32_t m01 = t.mh01 ^ kNegHalves, m2 = t.mh2 ^ kNegHalves;
            // words (0, 4 | 1, 5) and (2, 6 | 3, 7)
            op = make_uint4(m01, lo_lo(m2, t.h01), lo_lo(m2, t.ml01 ^ kNegHalves), hi_lo(t.h01, t.h2));
            op2 = make_uint4(hi_lo(t.ml01, t.ml2) ^ kNegHalves, split_half2(t.N - share), m01, kOneOne);
        }
    }
    if (p < ((b.n + kFiltTile - 1) & ~(int64_t)(kFiltTile - 1))) {
        reinterpret_cast<uint4*>(b.posB)[p] = op;
        reinterpret_cast<uint4*>(b.velB)[p] = op2;
    }
#pragma unroll
    for (int o = 1; o < kFiltTile; o <<= 1) {
#pragma unroll
        for (int d = 0; d < DIM; ++d) {
            lo[d] = fminf(lo[d], __shfl_xor_sync(kFull, lo[d], o));
            hi[d] = fmaxf(hi[d], __shfl_xor_sync(kFull, hi[d], o));
        }
    }
    if (valid && (p & (kFiltTile - 1)) == 0) {   // the tile's first particle
        float4* bx = reinterpret_cast<float4*>(b.key) + 2 * (p / kFiltTile);
        bx[0] = make_float4(lo[0], lo[1], DIM == 3 ? lo[2] : 0.f, 0.f);
        bx[1] = make_float4(hi[0], hi[1], DIM == 3 ? hi[2] : 0.f, 0.f);
    }
}

// D = A B for a 16 x 8 tile of depth 16: rows are homes, columns candidates.
__device__ __forceinline__ void filter_mma(float d[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                           uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
        : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(0.f));
}

// Unwrapped search cells of one dimension that can hold a candidate of homes in
// cells g_lo ... g_hi of c-bins c_lo ... c_hi: within k cells (at most half a
// periodic box) and, where c-bins more than one apart cannot be neighbours
// around the box, inside the neighbouring c-bins.  Within [-M, 2 M).
__device__ __forceinline__ void filter_range(int g_lo, int g_hi, int c_lo, int c_hi, int s, int M, int n, int k,
                                             bool wall, int& lo, int& hi) {
    const int kk = wall ? k : min(k, M / 2 + 1);
    lo = g_lo - kk;
    hi = g_hi + kk;
    if (wall || n >= 5) {
        lo = max(lo, (c_lo - 1) * s);
        hi = min(hi, (c_hi + 2) * s - 1);
    }
    if (wall) {
        lo = max(lo, 0);
        hi = min(hi, M - 1);
    }
}

// The frame (2^sh cells, or all M) that holds unwrapped cell t of [-M, 2 M): image, last
// unwrapped cell of the frame inside [t, hi], twice the frame's centre in cells.
__device__ __forceinline__ void filter_frame(int t, int hi, int M, int sh, int& image, int& end, int& centre2) {
    image = t < 0 ? -1 : (t >= M ? 1 : 0);
    const int o = image * M, f = (t - o) >> sh;
    end = min(hi, o + min(M, (f + 1) << sh) - 1);
    centre2 = 2 * o + ((2 * f) << sh) + min(1 << sh, M);
}

__device__ __forceinline__ bool cbins_adjacent(int a, int b, int n, bool wall) {
    const int d = abs(a - b);
    return d <= 1 || (!wall && d >= n - 1);
}

// Closest candidate so far of a warp's homes: the partner key in binary32
// (minima by atomicMin), distance and id in binary64.
template <typename T>
struct FiltBest;
template <>
struct FiltBest<float> {
    unsigned long long key[32];
    __device__ __forceinline__ void clear(int i) { key[i] = kNoPartner; }
    // a lane's passing pair: home i, distance^2 and tag of the candidate
    __device__ __forceinline__ void offer(bool pass, int i, float d2, uint32_t tag) {
        if (pass) atomicMin(&key[i], partner_key<float>(d2, tag));
    }
    // distance of the closest candidate in the frame's units
    __device__ __forceinline__ bool distance(int i, const InstDyn& D, float& d) const {
        const uint32_t o = (uint32_t)(key[i] >> 32);
        d = sqrtf(fmaxf(__uint_as_float((o & 0x80000000u) ? (o ^ 0x80000000u) : ~o), 0.f)) * D.f_scale;
        return o != 0xffffffffu;
    }
};
template <>
struct FiltBest<double> {
    double d2[32];
    uint32_t id[32];
    __device__ __forceinline__ void clear(int i) {
        d2[i] = R<double>::inf();
        id[i] = 0xffffffffu;
    }
    __device__ __forceinline__ void offer(bool pass, int i, double d, uint32_t tag) {
        for (unsigned m = __ballot_sync(kFull, pass); m; m &= m - 1) {   // one lane at a time
            if ((int)lane_id() == __ffs(m) - 1 && (d < d2[i] || (d == d2[i] && tag < id[i]))) {
                d2[i] = d;
                id[i] = tag;
            }
            __syncwarp();
        }
    }
    __device__ __forceinline__ bool distance(int i, const InstDyn& D, float& d) const {
        d = sqrtf(fmaxf((float)d2[i], 0.f)) * D.f_scale;
        return id[i] != 0xffffffffu;
    }
};

// A warp's walk of its window.  Kept in shared memory (every lane writes the same
// value): it is used once per block of the walk, and the registers it would take
// are those of the filter and the tests.
struct FiltWalk {
    int xa, xb, ya, yb, za, zb;   // the window in unwrapped search cells
    int g0, g1;                   // the row of the homes
    int tx, ty, tz;               // the current block: first unwrapped cells,
    int ex, ey, ez;               // last ones,
    int kx, ky, kz;               // image,
    int cx2, cy2, cz2;            // twice the frame's centre in cells,
    int rows, r0;                 // its rows of cells, and those looked at
    unsigned seg, pending;        // homes of this run, homes not searched yet
};

// Shared memory of a warp.
template <typename T>
struct FiltWarp {
    FiltWalk walk;
    float4 box[2];                             // swept box of the homes (lo, hi) in the block's image, widened
    typename Vec4<T>::type pos[32], vel[32];   // the homes
    uint4 op[64];                              // their rows of A in the current frame
    uint4 chunk[kFiltChunks];                  // tiles of the chunks in test
    uint4 list[kFiltList / 4];                 // listed tiles: number, kTilePart, kTileOwn
    uint2 queue[kFiltQueue];                   // surviving pairs: a lane's word of a chunk, (chunk << 5 | lane)
    unsigned char range[kFiltList];            // candidates of a kTilePart tile that belong to its row's range
    FiltBest<T> best;
};

// Search of every particle: a warp takes 32 consecutive sorted positions
// (homes) and, per run of homes of one row of search cells, walks the frame
// blocks of their window.  Per block: a lane per row finds its candidates'
// positions, the rows' tiles of 8 candidates are numbered through, and a lane per
// tile checks the tile's swept box against the homes'; the tiles that meet it are
// listed and go through the tensor filter four at a time (32 x 32 pairs).  A
// lane's surviving pairs of such a chunk are the bits of a word; words are queued
// and the pairs tested exactly, one per lane, while every lane has one.
//   sym (binary32): only candidates at higher positions, the outcome offered to
//   both keys (each pair once), threshold R^2.  Otherwise the whole window, the
//   outcome kept by the home alone and the threshold lowered to its closest
//   candidate: better where many candidates of the window pass (a contact
//   distance about as wide as the c-bins); binary64.
//   CHI: two more products give the signs of a = r0.s and f = r1.s (s = v_rel
//   dt), criterion 1 itself: worth it where the contact distance is wider than a
//   step's displacement, so that F < R^2 keeps most of the near pairs.
// 1 << split warps share a group's tiles (a small system has too few groups to
// fill the chip).
template <typename T, int DIM, bool CHI, int WARPS>
__global__ void __launch_bounds__(WARPS * 32, (sizeof(T) == 8 ? 16 : CHI ? 24 : 32) / WARPS)
    filter_search_kernel(Bufs<T> b, int split) {
    using V = typename Vec4<T>::type;
    constexpr int F = DIM - 1;
    constexpr bool kF32 = sizeof(T) == 4;
    const GeoT<T>& G = b.g;   // kernel parameter: constant bank
    __shared__ FiltWarp<T> shared_warps[WARPS];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    FiltWarp<T>& W = shared_warps[warp];
    const int64_t group = ((int64_t)blockIdx.x * WARPS + warp) >> split;
    const int sub = warp & ((1 << split) - 1);
    const int32_t p0 = (int32_t)(group * 32);   // position of the group's first home
    const float4* __restrict__ boxB = reinterpret_cast<const float4*>(b.key);
    // words (q, q + 4) of candidate lane / 4, q = lane % 4, of tile 0
    const uint2* __restrict__ op16 = reinterpret_cast<const uint2*>((lane & 2) ? b.velB : b.posB) + (lane >> 2) * 2 + (lane & 1);
    // the same with three filters: word q of the candidate in either buffer
    const uint32_t* __restrict__ opB = reinterpret_cast<const uint32_t*>(b.posB) + lane;
    const uint32_t* __restrict__ opS = reinterpret_cast<const uint32_t*>(b.velB) + lane;
    const uint32_t nmax = (uint32_t)b.n;

    FiltWalk& w = W.walk;
    uint32_t row;   // row of search cells of this lane's home
    int inst;
    {
        const int64_t p64 = group * 32 + lane;
        bool valid = p64 < b.n;
        V P = {}, Q = {};
        if (valid) {
            P = b.posA[p64];
            Q = b.velA[p64];
            valid = !absorbed(Q.w);
        }
        W.pos[lane] = P;
        W.vel[lane] = Q;
        inst = valid ? tag_inst(b, R<T>::bits(P.w)) : 0;
        const InstDev& I = b.inst[inst];
        valid = valid && I.search == kSearchFilter;
        int c, g0, g1 = 0;
        cell_and_search<T>(P.x, G.lo[0], G.inv[0], G.n[0], I.s[0], c, g0);
        if (DIM == 3) cell_and_search<T>(P.y, G.lo[1], G.inv[1], G.n[1], I.s[1], c, g1);
        row = DIM == 3 ? (uint32_t)g0 * (uint32_t)I.M[1] + (uint32_t)g1 : (uint32_t)g0;
        W.best.clear(lane);
        w.pending = __ballot_sync(kFull, valid);
    }
    __syncwarp();
    while (const unsigned pending = w.pending) {
        // the next run: homes of one instance and row, from home `first` to `last`
        const int first = __ffs(pending) - 1;
        const int seg_inst = __shfl_sync(kFull, inst, first);
        const uint32_t seg_row = __shfl_sync(kFull, row, first);
        const unsigned seg = __ballot_sync(kFull, inst == seg_inst && row == seg_row) & pending;
        const int last = 31 - __clz(seg);
        __syncwarp();
        w.pending = pending & ~seg;
        w.seg = seg;
        const InstDev& I = b.inst[seg_inst];
        const InstDyn& D = b.dyn[seg_inst];
        const bool sym = kF32 && I.sym;
        const T dt = step_dt(D, T()), R2 = inst_R2(I, T());
        unsigned wtests = 0;   // exact tests
        // rows lane / 4 + 0, 8, 16, 24: words q (per filter), words q + 4 (F and a share them, f)
        uint32_t A[CHI ? 12 : 4], N[CHI ? 8 : 4];
        float nI = 0.f;   // this lane's home: its own term less its share of the margin
        const uint32_t* ow = reinterpret_cast<const uint32_t*>(W.op);
        // the homes' own terms, with their thresholds after the tests so far
        auto put_own = [&]() {
            float thr = D.f_thr;
            if (!sym) {
                float d;   // distance of the closest candidate so far
                if (W.best.distance(lane, D, d)) thr = fminf(thr, fmaf(d * (1.f + 0x1p-19f), d, fmaf(D.f_rt, d, D.f_slack)));
            }
            // (a contact distance beyond the frames' width: within binary16's range all the same)
            const uint32_t w = split_half2(fmaxf(fminf(nI - thr, kNoHit), -kNoHit));
            __syncwarp();
            if (CHI) W.op[lane].x = w;
            else W.op[2 * lane + 1].w = w;
            __syncwarp();
#pragma unroll
            for (int k = 0; k < 4; ++k) N[k] = CHI ? ow[32 * k + lane] : ow[64 * k + 2 * lane + 1];
        };

        {
            const V P = W.pos[first], Z = W.pos[last];
            const T x[3] = {P.x, P.y, P.z}, z[3] = {Z.x, Z.y, Z.z};
            int c, ca, ga, gb, g, lo, hi;
            cell_and_search<T>(x[0], G.lo[0], G.inv[0], G.n[0], I.s[0], c, g);
            filter_range(g, g, c, c, I.s[0], I.M[0], G.n[0], D.k[0], G.wall[0], lo, hi);
            w.g0 = g;
            w.tx = w.xa = lo;
            w.xb = hi;
            w.g1 = w.ty = w.ya = w.yb = w.ey = w.ky = w.cy2 = 0;
            if (DIM == 3) {
                cell_and_search<T>(x[1], G.lo[1], G.inv[1], G.n[1], I.s[1], c, g);
                filter_range(g, g, c, c, I.s[1], I.M[1], G.n[1], D.k[1], G.wall[1], lo, hi);
                w.g1 = g;
                w.ty = w.ya = lo;
                w.yb = hi;
            }
            cell_and_search<T>(x[F], G.lo[F], G.inv[F], G.n[F], I.s[F], ca, ga);
            cell_and_search<T>(z[F], G.lo[F], G.inv[F], G.n[F], I.s[F], c, gb);
            filter_range(ga, gb, ca, c, I.s[F], I.M[F], G.n[F], D.k[F], G.wall[F], lo, hi);
            w.za = lo;
            w.zb = hi;
            // the walk steps to its first block from the one before it
            w.tz = w.ez = lo - 1;
            w.ex = w.tx - 1;
            w.rows = w.r0 = 0;
            __syncwarp();
        }
        int total = 0, t0 = 0;            // tiles of the current 32 rows, and those looked at
        int32_t q0 = 0, q1 = 0;           // this lane's row: its candidates,
        int incl = 0, first_tile = 0;     // tiles up to and with it, first tile less the tiles before it
        int listed = 0, chunks = 0;
        int qhead = 0, qn = 0;            // queued words
        uint32_t word = 0u, from = 0u;    // this lane's word in test: its pairs left, (chunk << 5 | lane)
        int busy = 0;                     // lanes that have one
        bool built = false, images = false, more = true;   // more: blocks of the window are left
        while (true) {
            bool rows_left = w.r0 < w.rows;
            if (t0 >= total && !rows_left && listed == 0 && more) {
                // the next block
                int tx = w.tx, ty = w.ty, tz = w.ez + 1;
                if (tz > w.zb) {
                    tz = w.za;
                    ty = w.ey + 1;
                    if (DIM == 2 || ty > w.yb) {
                        ty = w.ya;
                        tx = w.ex + 1;
                    }
                }
                more = tx <= w.xb;
                if (more) {
                    int kx, ky = 0, kz, ex, ey = ty, ez, c2;
                    __syncwarp();
                    filter_frame(tx, w.xb, I.M[0], D.f_shift[0], kx, ex, c2);
                    w.cx2 = c2;
                    if (DIM == 3) {
                        filter_frame(ty, w.yb, I.M[1], D.f_shift[1], ky, ey, c2);
                        w.cy2 = c2;
                    }
                    filter_frame(tz, w.zb, I.M[F], D.f_shift[F], kz, ez, c2);
                    w.cz2 = c2;
                    const int gx = ex - kx * I.M[0], gy = DIM == 3 ? ey - ky * I.M[1] : 0;   // last row
                    // lower positions: their homes test this group
                    const bool lower = sym && (gx < w.g0 || (DIM == 3 && gx == w.g0 && gy < w.g1));
                    w.tx = tx;
                    w.ty = ty;
                    w.tz = tz;
                    w.ex = ex;
                    w.ey = ey;
                    w.ez = ez;
                    w.kx = kx;
                    w.ky = ky;
                    w.kz = kz;
                    w.rows = lower ? 0 : (ex - tx + 1) * (ey - ty + 1);
                    w.r0 = 0;
                    total = t0 = 0;
                    built = false;
                    __syncwarp();
                    continue;
                }
            } else if (t0 >= total && rows_left) {
                // a lane per row: its candidates' positions and tiles
                const int gx = w.tx - w.kx * I.M[0], gy = DIM == 3 ? w.ty - w.ky * I.M[1] : 0, gz = w.tz - w.kz * I.M[F];
                const int ny = DIM == 3 ? w.ey - w.ty + 1 : 1, nz = w.ez - w.tz + 1;
                const int r = w.r0 + lane;
                q0 = q1 = 0;
                if (r < w.rows) {
                    const int ix = DIM == 3 ? r / ny : r, iy = DIM == 3 ? r - ix * ny : 0;
                    // four periodic c-bins: the one across the box is no neighbour
                    bool near = true;
                    if (G.n[0] == 4 && !G.wall[0]) near = cbins_adjacent((gx + ix) / I.s[0], w.g0 / I.s[0], 4, false);
                    if (DIM == 3 && G.n[1] == 4 && !G.wall[1])
                        near = near && cbins_adjacent((gy + iy) / I.s[1], w.g1 / I.s[1], 4, false);
                    if (near) {
                        const uint32_t key = DIM == 3 ? cell_key<3>(I, gx + ix, gy + iy, gz) : cell_key<2>(I, gx + ix, gz, 0);
                        // clamped so that a corrupted scan (flagged on the host) cannot read outside A
                        q0 = (int32_t)min(b.start[key], nmax);
                        q1 = (int32_t)min(b.start[key + (uint32_t)nz], nmax);
                        if (sym) q0 = max(q0, p0 + first + 1);
                    }
                }
                const int tile0 = q0 / kFiltTile, cnt = pieces_touched(q0, q1, kFiltTile);
                incl = cnt;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int y = __shfl_up_sync(kFull, incl, o);
                    if (lane >= o) incl += y;
                }
                first_tile = tile0 - (incl - cnt);
                total = __shfl_sync(kFull, incl, 31);
                t0 = 0;
                const int seen = w.r0 + 32;
                rows_left = seen < w.rows;
                __syncwarp();
                w.r0 = seen;
                __syncwarp();
                if (total == 0) continue;
            }
            if (t0 < total) {
                if (!built) {   // the homes in this frame
                    built = true;
                    images = images || w.kx != 0 || w.ky != 0 || w.kz != 0 || D.f_image != 0;
                    const int c2[3] = {w.cx2, DIM == 3 ? w.cy2 : w.cz2, w.cz2};
                    T ctr[3] = {(T)0, (T)0, (T)0};
#pragma unroll
                    for (int d = 0; d < DIM; ++d) ctr[d] = frame_centre(G, I, D, d, c2[d]);
                    const bool act = (w.seg >> lane) & 1u;
                    const V P = W.pos[lane], Q = W.vel[lane];
                    const T x[3] = {P.x, P.y, P.z}, v[3] = {Q.x, Q.y, Q.z};
                    float X[3] = {0.f, 0.f, 0.f}, S[3] = {0.f, 0.f, 0.f}, s2 = 0.f;
                    float lo[3] = {0.f, 0.f, 0.f}, hi[3] = {0.f, 0.f, 0.f};
                    const int kd[3] = {w.kx, DIM == 3 ? w.ky : w.kz, w.kz};
#pragma unroll
                    for (int d = 0; d < DIM; ++d) {
                        const Path1 p = path_in_frame(D, x[d], v[d], ctr[d], (T)kd[d] * G.L[d],
                                                      0.5f * (float)(c2[d] - 2 * kd[d] * I.M[d]) * D.f_w[d]);
                        X[d] = p.X;
                        S[d] = p.S;
                        s2 += S[d] * S[d];
                        // widened by the contact distance and the rounding of the exact test
                        lo[d] = act ? fminf(p.xf, p.xf + p.sf) - D.f_box : R<float>::inf();
                        hi[d] = act ? fmaxf(p.xf, p.xf + p.sf) + D.f_box : -R<float>::inf();
#pragma unroll
                        for (int o = 1; o < 32; o <<= 1) {
                            lo[d] = fminf(lo[d], __shfl_xor_sync(kFull, lo[d], o));
                            hi[d] = fmaxf(hi[d], __shfl_xor_sync(kFull, hi[d], o));
                        }
                    }
                    W.box[0] = make_float4(lo[0], lo[1], lo[2], 0.f);
                    W.box[1] = make_float4(hi[0], hi[1], hi[2], 0.f);
                    const float sl = sqrtf(s2), share = fmaf(D.f_g1, sl, D.f_g0);
                    auto rows_of = [&](uint4 w, uint32_t* a) {   // word q of rows lane / 4 + 0, 8, 16, 24
                        __syncwarp();
                        W.op[lane] = w;
                        __syncwarp();
#pragma unroll
                        for (int k = 0; k < 4; ++k) a[k] = ow[32 * k + lane];
                    };
                    // a lane without a home here, or one too far off to pair with this frame's
                    // candidates (its coordinates may overflow), has no pair
                    if constexpr (CHI) {
                        const ChiTerms t = chi_terms(X, S);
                        const float c = fmaf(D.f_c1, sl, D.f_c0);
                        const bool home = act && t.xy_ - share < kNoHit && fabsf(t.xs) + fabsf(t.ys) < kNoHit;
                        nI = home ? t.xy_ - share : R<float>::inf();
                        // (y, x), (s, x) and (s, y) with the signs flipped, then the own terms
                        uint32_t yx[3], sx[3], sy[3];
#pragma unroll
                        for (int d = 0; d < 3; ++d) {
                            yx[d] = home ? hi_lo(t.xy[d], t.xy[d]) ^ kNegHalves : 0u;
                            sx[d] = home ? lo_lo(t.s[d], t.xy[d]) ^ kNegHalves : 0u;
                            sy[d] = home ? lo_lo(t.s[d], t.xy[d] >> 16) ^ kNegHalves : 0u;
                        }
                        const uint32_t nf = home ? split_half2(fminf(t.ys + c, kNoHit)) : 0u;
                        rows_of(make_uint4(yx[0], yx[1], yx[2], kOneOne), A);
                        rows_of(make_uint4(sx[0], sx[1], sx[2], kOneOne), A + 4);
                        rows_of(make_uint4(sy[0], sy[1], sy[2], 0u), A + 8);
                        rows_of(make_uint4(lo_lo(kOneOne, nf), hi_lo(kOneOne, nf >> 16), 0u, 0u), N + 4);
                        __syncwarp();
                        W.op[lane] = make_uint4(0u, home ? split_half2(fmaxf(t.xs - c, -kNoHit)) : 0u, 0u, 0u);
                    } else {
                        const PathTerms t = path_terms(X, S);
                        const bool home = act && t.N - share < kNoHit;
                        nI = home ? t.N - share : R<float>::inf();
                        const uint32_t mh01 = times2(t.mh01), mh2 = times2(t.mh2), ml01 = times2(t.ml01),
                                       ml2 = times2(t.ml2), h01 = times2(t.h01), h2 = times2(t.h2);
                        // words (0, 4 | 1, 5) and (2, 6 | 3, 7)
                        uint4 w1 = make_uint4(mh01, lo_lo(ml2, h01), lo_lo(mh2, mh01), hi_lo(h01, h2));
                        uint4 v2 = make_uint4(hi_lo(mh01, mh2), kOneOne, ml01, 0u);
                        if (!home) {
                            w1 = make_uint4(0u, 0u, 0u, 0u);
                            v2 = make_uint4(0u, kOneOne, 0u, 0u);
                        }
                        __syncwarp();
                        W.op[2 * lane] = w1;
                        W.op[2 * lane + 1] = v2;
                        __syncwarp();
#pragma unroll
                        for (int k = 0; k < 4; ++k) A[k] = ow[64 * k + 2 * lane];
                    }
                    put_own();
                }
                // a lane per tile: the row it belongs to, then its box
                const int f = t0 + lane;
                int rr = 0;
#pragma unroll
                for (int o = 16; o > 0; o >>= 1)
                    if (__shfl_sync(kFull, incl, rr + o - 1) <= f) rr += o;
                const int tile = f + __shfl_sync(kFull, first_tile, rr & 31);
                const int32_t rq0 = __shfl_sync(kFull, q0, rr & 31), rq1 = __shfl_sync(kFull, q1, rr & 31);
                bool meet = f < total;
                if (split) meet = meet && (f & ((1 << split) - 1)) == sub;   // this warp's share
                uint32_t entry = (uint32_t)tile;
                unsigned vm = 0u;   // candidates of the tile that belong to the row's range
                if (meet) {
                    const float4 l = __ldg(boxB + 2 * (size_t)tile), u = __ldg(boxB + 2 * (size_t)tile + 1);
                    const float4 hl = W.box[0], hu = W.box[1];
                    meet = l.x <= hu.x && u.x >= hl.x && l.y <= hu.y && u.y >= hl.y;
                    if (DIM == 3) meet = meet && l.z <= hu.z && u.z >= hl.z;
                    const int a = max(rq0 - tile * kFiltTile, 0), e = min(rq1 - tile * kFiltTile, kFiltTile);
                    vm = (0xffu >> (kFiltTile - e)) & (0xffu << a);
                    if (vm != 0xffu) entry |= kTilePart;
                    if (sym && tile * kFiltTile <= p0 + 31) entry |= kTileOwn;
                }
                const unsigned mm = __ballot_sync(kFull, meet);
                if (meet) {
                    const int e = listed + __popc(mm & ((1u << lane) - 1u));
                    reinterpret_cast<uint32_t*>(W.list)[e] = entry;
                    W.range[e] = (unsigned char)vm;
                }
                listed += __popc(mm);
                t0 += 32;
                __syncwarp();
            }
            // Four listed tiles at a time: filter, queue, test.  Fewer when the
            // block ends; none, but the queue emptied, after the last block.
            const bool flush = t0 >= total && !rows_left;
            const bool final = flush && listed == 0;
            if (final && more) continue;
            if (flush && (listed & 3)) {   // the last chunk of the block: filled up with empty tiles
                if (lane >= (listed & 3) && lane < 4) {
                    const int e = (listed & ~3) + lane;
                    reinterpret_cast<uint32_t*>(W.list)[e] = (reinterpret_cast<uint32_t*>(W.list)[0] & kTileMask) | kTilePart;
                    W.range[e] = 0;
                }
                listed = (listed | 3) + 1;
                __syncwarp();
            }
            {
                int at = 0;
                while (listed - at >= kFiltChunk || final) {
                    if (!final) {
                        const uint4 e = W.list[at >> 2];
                        uint32_t t[4] = {e.x, e.y, e.z, e.w};
                        const uint32_t marks = (t[0] | t[1] | t[2] | t[3]) & (kTilePart | kTileOwn);
                        if (marks) {
#pragma unroll
                            for (int k = 0; k < 4; ++k) t[k] &= kTileMask;
                        }
                        uint32_t part[4];   // per tile: the signs of homes 0-15 and, 16 bits up, of homes 16-31
                        if constexpr (CHI) {
                            uint32_t B[4], S[4];
#pragma unroll
                            for (int k = 0; k < 4; ++k) {
                                B[k] = __ldg(opB + (size_t)t[k] * 32);
                                S[k] = __ldg(opS + (size_t)t[k] * 32);
                            }
                            const int q = lane & 3;
                            const uint32_t sel = q == 3 ? 0x7654u : 0x5410u;
                            const uint32_t one0 = q == 0 ? kOneOne : 0u, one1 = q == 1 ? kOneOne : 0u;
#pragma unroll
                            for (int k = 0; k < 4; ++k) {
                                const uint32_t wa = __byte_perm(B[k], S[k], sel), wf = hi_lo(B[k], S[k]),
                                               wn = hi_lo(S[k], kOneOne);
                                uint32_t w[2];
#pragma unroll
                                for (int o = 0; o < 2; ++o) {
                                    float d[4], da[4], df[4];
                                    filter_mma(d, A[2 * o], A[2 * o + 1], N[2 * o], N[2 * o + 1], B[k], one0);
                                    filter_mma(da, A[4 + 2 * o], A[5 + 2 * o], N[2 * o], N[2 * o + 1], wa, one1);
                                    filter_mma(df, A[8 + 2 * o], A[9 + 2 * o], N[4 + 2 * o], N[5 + 2 * o], wf, wn);
                                    w[o] = 0u;
#pragma unroll
                                    for (int r = 0; r < 4; ++r)
                                        w[o] = __funnelshift_l(__float_as_uint(d[r]) & __float_as_uint(da[r]) &
                                                                   ~__float_as_uint(df[r]), w[o], 1);
                                }
                                part[k] = w[0] + (w[1] << 16);
                            }
                        } else {
                            uint2 B[4];
#pragma unroll
                            for (int k = 0; k < 4; ++k) B[k] = __ldg(op16 + (size_t)t[k] * 16);
#pragma unroll
                            for (int k = 0; k < 4; ++k) {
                                float d[4], e2[4];
                                filter_mma(d, A[0], A[1], N[0], N[1], B[k].x, B[k].y);
                                filter_mma(e2, A[2], A[3], N[2], N[3], B[k].x, B[k].y);
                                uint32_t w0 = 0u, w1 = 0u;
#pragma unroll
                                for (int r = 0; r < 4; ++r) {
                                    w0 = __funnelshift_l(__float_as_uint(d[r]), w0, 1);
                                    w1 = __funnelshift_l(__float_as_uint(e2[r]), w1, 1);
                                }
                                part[k] = w0 + (w1 << 16);
                            }
                        }
                        // bit 4 (3 - k) + 3 - r of a half: tile k, output r
                        uint32_t hit = ((part[0] * 16u + part[1]) * 16u + part[2]) * 16u + part[3];
                        if (marks & kTilePart) {
                            const uint32_t vm = *reinterpret_cast<const uint32_t*>(W.range + at) >> (2 * (lane & 3));
                            uint32_t keep = 0u;
#pragma unroll
                            for (int k = 0; k < 4; ++k) keep = keep << 4 | (0xf5a0u >> (4 * (vm >> (8 * k) & 3u)) & 0xfu);
                            hit &= keep | keep << 16;
                        }
                        if (marks & kTileOwn) {   // each pair once: positions above the home's
#pragma unroll
                            for (int k = 0; k < 4; ++k) {
#pragma unroll
                                for (int r = 0; r < 4; ++r) {
                                    const int32_t dq = (int32_t)t[k] * kFiltTile + 2 * (lane & 3) + (r & 1) -
                                                       (p0 + (lane >> 2) + 8 * (r >> 1));
                                    if (dq <= 0) hit &= ~(1u << (4 * (3 - k) + 3 - r));
                                    if (dq <= 16) hit &= ~(0x10000u << (4 * (3 - k) + 3 - r));
                                }
                            }
                        }
                        at += kFiltChunk;
                        // the lanes' words with pairs go to the queue
                        const unsigned some = __ballot_sync(kFull, hit != 0u);
                        if (some) {
                            if (hit)
                                W.queue[(qhead + qn + __popc(some & ((1u << lane) - 1u))) & (kFiltQueue - 1)] =
                                    make_uint2(hit, (unsigned)(chunks & (kFiltChunks - 1)) << 5 | (unsigned)lane);
                            if (lane == 0) W.chunk[chunks & (kFiltChunks - 1)] = make_uint4(t[0], t[1], t[2], t[3]);
                            ++chunks;
                            qn += __popc(some);
                        }
                    }
                    // Exact tests, a pair of its word per lane, while every lane has one; while
                    // any has at the end and before a chunk's slot is used again.
                    const int least = final || (chunks & (kFiltChunks - 1)) == 0 ? 1 : 32;
                    bool tested = false;
                    while (qn + busy >= least) {
                        tested = true;
                        __syncwarp();
                        const unsigned idle = __ballot_sync(kFull, word == 0u);
                        const int mine = __popc(idle & ((1u << lane) - 1u));
                        if (word == 0u && mine < qn) {
                            const uint2 e = W.queue[(qhead + mine) & (kFiltQueue - 1)];
                            word = e.x;
                            from = e.y;
                        }
                        const int took = min(__popc(idle), qn);
                        qhead += took;
                        qn -= took;
                        wtests += (unsigned)(busy + took);
                        bool pass = false;
                        int i = 0;
                        uint32_t tj = 0u;
                        T d2 = (T)0;
                        if (word != 0u) {
                            const int bit = __ffs(word) - 1;
                            word &= word - 1u;
                            const uint32_t tk = reinterpret_cast<const uint32_t*>(W.chunk + (from >> 5))[3 - (bit >> 2 & 3)];
                            i = (bit & 16) + (int)(from >> 2 & 7u) + ((bit & 2) ? 0 : 8);
                            const int32_t q = (int32_t)(tk * kFiltTile + 2u * (from & 3u) + (~(unsigned)bit & 1u));
                            const V Pj = ldg_vec(b.posA + q), Qj = ldg_vec(b.velA + q);
                            const V Pi = W.pos[i], Qi = W.vel[i];
                            tj = R<T>::bits(Pj.w);
                            const T xi[3] = {Pi.x, Pi.y, Pi.z}, vi[3] = {Qi.x, Qi.y, Qi.z};
                            const T xj[3] = {Pj.x, Pj.y, Pj.z}, vj[3] = {Qj.x, Qj.y, Qj.z};
                            const T zero[3] = {(T)0, (T)0, (T)0};
                            if (q != p0 + i &&
                                (images ? poca_test_sh<T, DIM, true>(G, xi, vi, xj, vj, zero, dt, R2, d2)
                                        : poca_test_sh<T, DIM, false, false>(G, xi, vi, xj, vj, zero, dt, R2, d2))) {
                                // the rows of the walk hold neighbouring c-bins only; along the
                                // fast dimension they are the union over the homes
                                int ci, cj, gs;
                                cell_and_search<T>(xi[F], G.lo[F], G.inv[F], G.n[F], 1, ci, gs);
                                cell_and_search<T>(xj[F], G.lo[F], G.inv[F], G.n[F], 1, cj, gs);
                                pass = cbins_adjacent(ci, cj, G.n[F], G.wall[F]);
                                if (kF32 && sym && pass) atomicMin(&b.bkey[q], partner_key<T>(d2, R<T>::bits(Pi.w)));
                            }
                        }
                        W.best.offer(pass, i, d2, tj);
                        busy = __popc(__ballot_sync(kFull, word != 0u));
                    }
                    if (final) break;
                    if (!sym && tested) put_own();   // lower thresholds
                }
                if (final) break;
                if (at > 0 && listed > at) {   // the rest moves to the front
                    uint32_t w = 0u;
                    unsigned char v = 0;
                    if (lane < listed - at) {
                        w = reinterpret_cast<uint32_t*>(W.list)[at + lane];
                        v = W.range[at + lane];
                    }
                    __syncwarp();
                    if (lane < listed - at) {
                        reinterpret_cast<uint32_t*>(W.list)[lane] = w;
                        W.range[lane] = v;
                    }
                }
                listed -= at;
                __syncwarp();
            }
        }
        if (I.prune && wtests && lane == 0)
            atomicAdd(&b.tile_tests[blockIdx.x % kTestSlots], (unsigned long long)wtests);
    }
    if constexpr (kF32) {
        __syncwarp();
        const unsigned long long key = W.best.key[lane];
        if (key != kNoPartner) atomicMin(&b.bkey[p0 + lane], key);
    } else {
        __syncthreads();   // the warps that share a group are of one block
        if (sub == 0) {
            double bd = W.best.d2[lane];
            uint32_t bi = W.best.id[lane];
            for (int o = 1; o < (1 << split); ++o) {
                const FiltBest<T>& S = shared_warps[warp + o].best;
                if (S.d2[lane] < bd || (S.d2[lane] == bd && S.id[lane] < bi)) {
                    bd = S.d2[lane];
                    bi = S.id[lane];
                }
            }
            if (bi != 0xffffffffu) b.bkey[p0 + lane] = partner_key<T>((T)bd, bi);
        }
    }
}

template <typename T, int DIM, bool CHI>
cudaError_t launch_filtered(const Bufs<T>& b, cudaStream_t s) {
    const int64_t warps = ((b.n + 31) / 32) << b.filter_split;
    filter_prep_kernel<T, DIM, CHI><<<blocks_for((b.n + 31) & ~(int64_t)31), kThreads, 0, s>>>(b);
    // the warps that share a group are a block; a group of its own is a block of one
    // warp (a block holds its place until its slowest warp is done: 4 warps took 8-10 %
    // longer on the 3-D Sod tubes)
    if (b.filter_split == 0) filter_search_kernel<T, DIM, CHI, 1><<<(unsigned)warps, 32, 0, s>>>(b, 0);
    else if (b.filter_split < 3)
        filter_search_kernel<T, DIM, CHI, 4><<<(unsigned)((warps + 3) / 4), 128, 0, s>>>(b, b.filter_split);
    else filter_search_kernel<T, DIM, CHI, 8><<<(unsigned)(warps / 8), 256, 0, s>>>(b, 3);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_filtered_search(const Bufs<T>& b, cudaStream_t s) {
    if (b.n == 0) return cudaSuccess;
    if constexpr (sizeof(T) == 4)   // binary64 filters by criterion 1 too
        if (!b.filter_chi) return b.geo.dim == 3 ? launch_filtered<T, 3, false>(b, s) : launch_filtered<T, 2, false>(b, s);
    return b.geo.dim == 3 ? launch_filtered<T, 3, true>(b, s) : launch_filtered<T, 2, true>(b, s);
}

}  // namespace kmc
