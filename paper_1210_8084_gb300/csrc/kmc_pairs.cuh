// kmc_pairs.cuh -- closest-candidate search of middle windows (binary32): a warp
// takes 32 consecutive sorted positions, a lane per home, and walks the union of
// their windows.  64 candidates at a time are staged in shared memory as negated
// pairs; every lane tests two candidates per step (paired_signs), all lanes the same
// ones, and keeps a bit per candidate.  The pairs that pass, a few per cent, are
// queued and decided exactly by 32 lanes at a time.  Each pair once, by its lower
// position, the outcome offered to both keys: the decisions and keys of the other
// searches.
//
// Against one thread per particle, each walking its own window: no divergence, two
// tests per step, loads and staging shared by the warp, for the price of the union
// (32 candidates more per row).  Against the filtered search: no operands and no
// approximate pairs, which outnumber the true ones where particles move along with
// one another or the contact distance is wide.  Bound by the paired FP32 pipe and by
// issue (2-D: 14 paired operations of 2 cycles per step of two candidates).
//
// CLOSE: where many candidates pass (kPairsClose), a pair is also tested against the
// closest so far of either particle: its distance of closest approach is at most B
// iff a^2 >= b (r^2 - B), so B takes the place of R^2, widened by p_slack for the
// rounding of the stored distance (relative errors of a few 2^-24 of terms of
// at most D^2, D = R + 2 vmax dt).  A stale bound is a larger one.  The 64M-particle
// quadrants, 2200 candidates of which 130 would pass, took 117 ms without and 82 ms
// with it; 92 ms with the farthest of the staged candidates for all of them.  Where
// few pass it costs 10 % (5M Noh 0.50 -> 0.58 ms).
//
// Search times before (the cheaper of the other searches) and here: 5M 2-D Noh
// 0.91 -> 0.50 ms, 64M quadrants 104 -> 82, 5M slab tube with 160 candidates 1.53 ->
// 1.09, 4M Noh of 150^2 c-bins 13.9 -> 2.3.  Warps of 64 registers, 32 per SM: 24
// of 80 registers took 4-10 % longer.
#pragma once

#include "kmc_filter.cuh"

namespace kmc {

constexpr int kPairsBlocks = 32;   // per SM, of one warp each
constexpr int kPairsChunk = 64;   // candidates staged at a time

struct PairsWarp {
    float4 A[kPairsChunk / 2], B[kPairsChunk / 2], C[kPairsChunk / 2];   // staged candidates (paired_core's layout)
    uint32_t tag[kPairsChunk];
    alignas(8) float least[kPairsChunk];   // their negated bounds
    float4 pos[32], vel[32];             // the homes
    unsigned long long key[32];          // their closest candidates so far
    unsigned short queue[32 * 32 + 32];  // pairs that meet criteria 1-2: home << 6 | candidate
};

template <int DIM, bool CLOSE>
__global__ void __launch_bounds__(32, kPairsBlocks) pairs_search_kernel(Bufs<float> b) {
    constexpr int F = DIM - 1;
    const GeoT<float>& G = b.g;
    __shared__ PairsWarp W;
    const int lane = threadIdx.x;
    const int64_t p64 = (int64_t)blockIdx.x * 32 + lane;
    const int32_t p = (int32_t)p64;
    const uint32_t nmax = (uint32_t)b.n;
    bool valid = p64 < b.n;
    float4 P = make_float4(0.f, 0.f, 0.f, 0.f), Q = P;
    if (valid) {
        P = b.posA[p64];
        Q = b.velA[p64];
    }
    const uint32_t tag = __float_as_uint(P.w);
    const int inst = valid ? tag_inst(b, tag) : 0;
    valid = valid && b.inst[inst].search == kSearchPairs;
    // sorted position by id, read by the move kernel to find a partner
    if (valid) b.slot_of[b.inst[inst].p_off + (int64_t)tag_id(b, tag)] = (uint32_t)p;
    valid = valid && !absorbed(Q.w);
    const float xi[3] = {P.x, P.y, P.z}, vi[3] = {Q.x, Q.y, Q.z};
    int c[3] = {0, 0, 0}, g[3] = {0, 0, 0};
    uint32_t row;
    {
        const InstDev& I = b.inst[inst];
#pragma unroll
        for (int d = 0; d < DIM; ++d) cell_and_search<float>(xi[d], G.lo[d], G.inv[d], G.n[d], I.s[d], c[d], g[d]);
        row = DIM == 3 ? (uint32_t)g[0] * (uint32_t)I.M[1] + (uint32_t)g[1] : (uint32_t)g[0];
    }
    W.pos[lane] = P;
    W.vel[lane] = Q;
    W.key[lane] = CLOSE && valid ? __ldcg(&b.bkey[p]) : kNoPartner;
    for (unsigned pending = __ballot_sync(kFull, valid); pending;) {
        // a run of homes of one instance and row of search cells
        const int first = __ffs(pending) - 1;
        const int seg_inst = __shfl_sync(kFull, inst, first);
        const uint32_t seg_row = __shfl_sync(kFull, row, first);
        const unsigned seg = __ballot_sync(kFull, inst == seg_inst && row == seg_row) & pending;
        pending &= ~seg;
        const int last = 31 - __clz(seg);
        const bool act = (seg >> lane) & 1u;
        const InstDev& I = b.inst[seg_inst];
        const InstDyn& D = b.dyn[seg_inst];
        const float dt = D.dtf, R2 = I.R2f;
        PairHome ph = pair_home(xi, vi, dt, R2);
        if (!act) ph.x0 = make_float2(__int_as_float(0x7fc00000), __int_as_float(0x7fc00000));   // no pair
        // the window in unwrapped search cells
        int lo[3] = {0, 0, 0}, hi[3] = {0, 0, 0};
#pragma unroll
        for (int d = 0; d < DIM; ++d) {
            const int ga = __shfl_sync(kFull, g[d], first), gb = __shfl_sync(kFull, g[d], last);
            const int ca = __shfl_sync(kFull, c[d], first), cb = __shfl_sync(kFull, c[d], last);
            filter_range(ga, gb, ca, cb, I.s[d], I.M[d], G.n[d], D.k[d], G.wall[d], lo[d], hi[d]);
        }
        const int g0 = __shfl_sync(kFull, g[0], first), g1 = __shfl_sync(kFull, g[1], first);
        const int ny = DIM == 3 ? hi[1] - lo[1] + 1 : 1;
        const int z0 = lo[F] < 0 ? -1 : 0, z1 = hi[F] >= I.M[F] ? 1 : 0, nz = z1 - z0 + 1;   // images of the fast dimension
        const int rows = (hi[0] - lo[0] + 1) * ny * nz;
        for (int r0 = 0; r0 < rows; r0 += 32) {
            // a lane per row and image: its candidates' positions and image
            const int r = r0 + lane;
            int32_t q0 = 0, q1 = 0;
            unsigned code = 0u;
            if (r < rows) {
                const int kz = z0 + r % nz, xy = r / nz;
                const int tx = lo[0] + (DIM == 3 ? xy / ny : xy), ty = DIM == 3 ? lo[1] + xy % ny : 0;
                const int kx = tx < 0 ? -1 : tx >= I.M[0] ? 1 : 0, ky = DIM == 3 ? (ty < 0 ? -1 : ty >= I.M[1] ? 1 : 0) : 0;
                const int gx = tx - kx * I.M[0], gy = DIM == 3 ? ty - ky * I.M[1] : 0;
                const int za = max(lo[F], kz * I.M[F]) - kz * I.M[F], zb = min(hi[F], (kz + 1) * I.M[F] - 1) - kz * I.M[F];
                // four periodic c-bins: the one across the box is no neighbour
                bool near = true;
                if (G.n[0] == 4 && !G.wall[0]) near = cbins_adjacent(gx / I.s[0], g0 / I.s[0], 4, false);
                if (DIM == 3 && G.n[1] == 4 && !G.wall[1]) near = near && cbins_adjacent(gy / I.s[1], g1 / I.s[1], 4, false);
                if (near) {
                    const uint32_t key = DIM == 3 ? cell_key<3>(I, gx, gy, za) : cell_key<2>(I, gx, za, 0);
                    // clamped so that a corrupted scan (flagged on the host) cannot read outside A
                    q0 = max((int32_t)min(b.start[key], nmax), (int32_t)(blockIdx.x * 32) + first + 1);
                    q1 = (int32_t)min(b.start[key + (uint32_t)(zb - za + 1)], nmax);
                    code = (unsigned)(kx + 1) | (unsigned)(ky + 1) << 2 | (unsigned)(kz + 1) << 4;
                }
            }
            for (unsigned some = __ballot_sync(kFull, q1 > q0); some; some &= some - 1) {
                const int o = __ffs(some) - 1;
                const int32_t a0 = __shfl_sync(kFull, q0, o), a1 = __shfl_sync(kFull, q1, o);
                const unsigned cd = __shfl_sync(kFull, code, o);
                // separation x_i - x_j - image: the shift of x_i - x_j
                const float sh[3] = {(float)(1 - (int)(cd & 3u)) * G.L[0],
                                     DIM == 3 ? (float)(1 - (int)(cd >> 2 & 3u)) * G.L[1] : (float)(1 - (int)(cd >> 4 & 3u)) * G.L[1],
                                     DIM == 3 ? (float)(1 - (int)(cd >> 4 & 3u)) * G.L[2] : 0.f};
                const bool shifted = sh[0] != 0.f || sh[1] != 0.f || sh[2] != 0.f;
                // counted down: positions go up to 2^31 - 2, and a step past a1 could pass 2^31
                uint32_t next = (uint32_t)a0;
                for (int32_t left = a1 - a0; left > 0; left -= kPairsChunk, next += kPairsChunk) {
                    const int32_t base = (int32_t)next;
                    const int n = min(kPairsChunk, left);
                    __syncwarp();
                    // a pair farther than both of its particles' closest so far is no pair
                    // (a stale value is a larger one): negated bounds on its distance^2
                    auto bound = [&](uint32_t u) {
                        const float d2 = __uint_as_float((u & 0x80000000u) ? (u ^ 0x80000000u) : ~u);
                        return u == 0xffffffffu ? -R2 : fmaxf(-R2, -(d2 + D.p_slack));
                    };
                    float mB = 0.f;
                    if constexpr (CLOSE) mB = bound((uint32_t)(W.key[lane] >> 32));
#pragma unroll
                    for (int o = 0; o < kPairsChunk; o += 32) {
                        float least = 0.f;
                        float4 Pj = make_float4(0.f, 0.f, 0.f, 0.f), Qj = Pj;
                        Pj.x = __int_as_float(0x7fc00000);   // a pad fails every test
                        if (o + lane < n) {
                            Pj = ldg_vec(b.posA + base + o + lane);
                            Qj = ldg_vec(b.velA + base + o + lane);
                            if constexpr (CLOSE) least = bound((uint32_t)(__ldcg(&b.bkey[base + o + lane]) >> 32));
                        }
                        float* a = reinterpret_cast<float*>(W.A + ((o + lane) >> 1)) + (lane & 1);
                        float* bz = reinterpret_cast<float*>(W.B + ((o + lane) >> 1)) + (lane & 1);
                        float* cc = reinterpret_cast<float*>(W.C + ((o + lane) >> 1)) + (lane & 1);
                        a[0] = -Pj.x;
                        a[2] = -Pj.y;
                        bz[0] = -Pj.z;
                        bz[2] = -Qj.x;
                        cc[0] = -Qj.y;
                        cc[2] = -Qj.z;
                        W.tag[o + lane] = __float_as_uint(Pj.w);
                        if constexpr (CLOSE) W.least[o + lane] = least;
                    }
                    __syncwarp();
                    int queued = 0;
                    // the first `count` queued pairs, one per lane: the exact decision, criterion 3
                    auto drain = [&](int at, int count) {
                        if (lane < count) {
                            const int w = W.queue[at + lane], i = w >> 6, e = w & 63;
                            const float* A = reinterpret_cast<const float*>(W.A + (e >> 1)) + (e & 1);
                            const float* B = reinterpret_cast<const float*>(W.B + (e >> 1)) + (e & 1);
                            const float* C = reinterpret_cast<const float*>(W.C + (e >> 1)) + (e & 1);
                            const float4 Pi = W.pos[i], Qi = W.vel[i];
                            const float hx[3] = {Pi.x, Pi.y, Pi.z}, hv[3] = {Qi.x, Qi.y, Qi.z};
                            const float xj[3] = {-A[0], -A[2], -B[0]}, vj[3] = {-B[2], -C[0], -C[2]};
                            float d2;
                            const bool met = D.p_image ? poca_test_sh<float, DIM, true>(G, hx, hv, xj, vj, sh, dt, R2, d2)
                                                       : poca_test_sh<float, DIM, false>(G, hx, hv, xj, vj, sh, dt, R2, d2);
                            if (met) {
                                // the rows hold neighbouring c-bins; along the fast dimension they
                                // are the union over the homes
                                int ci, cj, gs;
                                cell_and_search<float>(hx[F], G.lo[F], G.inv[F], G.n[F], 1, ci, gs);
                                cell_and_search<float>(xj[F], G.lo[F], G.inv[F], G.n[F], 1, cj, gs);
                                if (cbins_adjacent(ci, cj, G.n[F], G.wall[F])) {
                                    const unsigned long long ki = partner_key<float>(d2, W.tag[e]),
                                                             kj = partner_key<float>(d2, __float_as_uint(Pi.w));
                                    if (ki < W.key[i]) atomicMin(&W.key[i], ki);
                                    // farther than its closest so far: not offered.  A bound of R^2 rules
                                    // nothing out: the rounded d^2 of a pair that meets may lie above it
                                    if (!CLOSE || W.least[e] <= -R2 || -d2 >= W.least[e])
                                        atomicMin(&b.bkey[base + e], kj);
                                }
                            }
                        }
                    };
#pragma unroll 1
                    for (int o = 0; o < n; o += 32) {
                        // criteria 1-2 of every lane's home against 32 candidates: candidate o + e at bit 31 - e
                        unsigned m = 0u;
                        const int pairs = (min(32, n - o) + 1) >> 1;
                        if (D.p_image) m = act ? kFull << (32 - 2 * pairs) : 0u;   // images within one row: every pair's own
                        else {
                            auto test = [&](auto has_shift) {
                                const PairShift ps = pair_shift(sh);
#pragma unroll 4
                                for (int k = 0; k < pairs; ++k) {
                                    float2 rr, a, bb;
                                    if constexpr (CLOSE) {
                                        const float2 t = *reinterpret_cast<const float2*>(W.least + o + 2 * k);
                                        ph.mR2 = make_float2(fminf(mB, t.x), fminf(mB, t.y));
                                    }
                                    const uint2 w = paired_signs<DIM, decltype(has_shift)::value>(
                                        ph, ps, W.A[(o >> 1) + k], W.B[(o >> 1) + k], W.C[(o >> 1) + k], rr, a, bb);
                                    m = __funnelshift_l(w.x, m, 1);
                                    m = __funnelshift_l(w.y, m, 1);
                                }
                                m <<= 32 - 2 * pairs;
                            };
                            if (shifted) test(std::true_type{});
                            else test(std::false_type{});
                        }
                        const int below = p + 1 - base - o;   // candidates at or below the home's position
                        if (below > 0) m = below < 32 ? m & (kFull >> below) : 0u;
                        // queue them, a run of entries per lane
                        const int mine = __popc(m);
                        int at = mine;
#pragma unroll
                        for (int k = 1; k < 32; k <<= 1) {
                            const int x = __shfl_up_sync(kFull, at, k);
                            if (lane >= k) at += x;
                        }
                        const int total = __shfl_sync(kFull, at, 31);
                        at += queued - mine;
                        while (m) {
                            const int e = __clz(m);
                            m &= ~(0x80000000u >> e);
                            W.queue[at++] = (unsigned short)(lane << 6 | (o + e));
                        }
                        queued += total;
                        __syncwarp();
                        int done = 0;
                        const bool all = o + 32 >= n;
                        while (queued - done >= 32 || (all && queued > done)) {
                            drain(done, min(32, queued - done));
                            done += 32;
                        }
                        if (!all) {   // fewer than 32 are left: to the front
                            unsigned short w = 0;
                            if (lane < queued - done) w = W.queue[done + lane];
                            __syncwarp();
                            if (lane < queued - done) W.queue[lane] = w;
                            queued -= done;
                        }
                    }
                }
            }
        }
    }
    __syncwarp();
    const unsigned long long best = W.key[lane];
    if (best != kNoPartner) atomicMin(&b.bkey[p], best);
}

template <typename T>
cudaError_t launch_pairs_search(const Bufs<T>& b, cudaStream_t s) {
    if constexpr (sizeof(T) == 4) {
        if (b.n == 0) return cudaSuccess;
        const unsigned blocks = (unsigned)((b.n + 31) / 32);
        if (b.paired & 2) {
            if (b.geo.dim == 3) pairs_search_kernel<3, true><<<blocks, 32, 0, s>>>(b);
            else pairs_search_kernel<2, true><<<blocks, 32, 0, s>>>(b);
        } else {
            if (b.geo.dim == 3) pairs_search_kernel<3, false><<<blocks, 32, 0, s>>>(b);
            else pairs_search_kernel<2, false><<<blocks, 32, 0, s>>>(b);
        }
        return cudaGetLastError();
    } else {
        (void)b;
        (void)s;
        return cudaSuccess;   // binary32 only
    }
}

}  // namespace kmc
