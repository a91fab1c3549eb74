// kmc_scan.cu -- single-pass exclusive scan of the search-key histogram
// (decoupled look-back) and the moment finalisation kernels.
//
// The scan turns count[k] (particles per search cell) into start[k], the first
// sorted position of cell k, and clears count for the next step.  Tiles are
// claimed with an atomic ticket, so every predecessor of a tile has already
// started when the tile looks back; each wait is bounded (kSpinCap) and sets
// kErrScanTimeout instead of hanging.
//
// The block holding tile 0 also rolls the per-instance step bookkeeping: the
// largest speed of the new state becomes current and the search half-window
// k_d = ceil(D' / w_d) with D' = 1.001 (R + 2 v_max dt) + 1e-5 L_d is derived
// from it.  Any pair that passes the acceptance test is closer than
// R + |v_rel| t_poca <= R + 2 v_max dt at the start of the step, so the window
// never drops a candidate of the 3^D c-bin neighbourhood.  The same block sets
// the fixed-point exponents of the moment sums from the largest speed.
#include <math.h>

#include "kmc_internal.h"

namespace kmc {

namespace {

constexpr unsigned long long kFlagAgg = 1ull << 32;
constexpr unsigned long long kFlagInc = 2ull << 32;

__device__ __forceinline__ unsigned long long load_status(const unsigned long long* p) {
    return *reinterpret_cast<const volatile unsigned long long*>(p);
}

// Largest e (within [-120, 120]) with m 2^e < 2^62: a sum of terms bounded by
// m in total stays inside a signed 64-bit integer with a factor 2 to spare.
__device__ __forceinline__ int fixed_exponent(double m) {
    if (!(m > 0.0) || !isfinite(m)) return 0;
    const int e = 61 - ilogb(m);
    return e < -120 ? -120 : (e > 120 ? 120 : e);
}

// Frames, units and margins of the filtered search (derivation at the head of
// kmc_filter.cuh) for a largest displacement s = v_max dt; the reach is
// D = R + 2 s.  The frames are as wide as keeps the rounding margin of an
// ordinary pair to about a tenth of what decides it: R^2 + |v_rel|^2 dt^2 / 4
// with one filter (R counts little where the threshold falls to the closest
// candidate so far: R / 8), R and |v_rel| dt with three.  Every bound below holds
// for any width.
// Computed in binary32 (one thread per instance, in the way of the step; binary64
// took 7 us): every bound carries a factor of 1 + 2^-10, far above its rounding.  Lengths
// are in units of f_len, or of s where that is longer, so nothing leaves the range.
__device__ void filter_constants(InstDyn& dy, const InstDev& in, const Geo& geo, double displacement) {
    const float up = 1.f + 0x1p-10f, r3 = 1.7320508f * up;
    float s = (float)fmin(displacement * (double)in.f_unit, 0x1p100) * (1.f + 0x1p-20f);
    const float z = s > 1.f ? __int_as_float((127 - ilogbf(s)) << 23) : 1.f;
    s *= z;
    const float Rc = in.f_R * z * (1.f + 0x1p-20f), R2 = Rc * Rc * (1.f + 0x1p-20f), Re = in.sym ? Rc : 0.125f * Rc;
    const float D = (Rc + 2.f * s) * (1.f + 0x1p-20f), cmax = in.f_c * z, lmax = in.f_lmax * z;
    float w[3], reach = 0.f;   // reach: largest separation of neighbouring c-bins, at most D
    int image = 0;
    for (int d = 0; d < geo.dim; ++d) {
        w[d] = in.f_cw[d] * z;
        reach = fmaxf(reach, fminf(D, 2.f * (float)in.s[d] * w[d]));
        if (geo.bc[d] == KMC_BC_PERIODIC && (geo.n[d] < 5 || D >= 0.499f * z * in.f_L[d])) image = 1;
    }
    const float aim = in.chi ? fminf(200.f * Rc, 400.f * s) : 46.f * sqrtf(Re * Re + s * s / 16.f);
    const float width = 2.f * (aim - reach - s);
    float half = 0.f;
    for (int d = 0; d < 3; ++d) {
        int sh = 0;
        dy.f_w[d] = 0.f;
        if (d < geo.dim) {
            while ((1 << sh) < in.M[d] && (float)min(2 << sh, in.M[d]) * w[d] <= width) ++sh;
            half = fmaxf(half, 0.5f * (float)min(1 << sh, in.M[d]) * w[d]);
            dy.f_w[d] = (float)in.w[d];
        }
        dy.f_shift[d] = sh;
    }
    // largest coordinate of a candidate in its frame and of a home that may pair with it
    const float X = (half + reach + s) * up;
    const float sc = __int_as_float((127 + 4 - ilogbf(X)) << 23), sc2 = sc * sc;   // X sc in [16, 32)
    // rounding of the coordinates and frame centres; binary64 rounds to binary32 after it has
    // taken the difference from the centre (the boxes' coordinates: and added the centre's)
    const float far = in.f64 ? 0x1p-50f * (cmax + lmax) : 0x1p-20f * (cmax + lmax);
    const float e32 = far + 0x1p-20f * (in.f64 ? X + s : s), tiny = 0x1p-23f / sc;
    float slack = 0x1p-17f * D * D + 0x1p-18f * 12.f * X * X;
    float E;   // error of a separation component that |r0| + |r1| (three filters) or |dm| (one) multiplies
    if (in.chi) {
        E = (0x1p-10f * X + e32 + tiny) * up;
        const float Es = (0x1p-10f * s + 0x1p-20f * s + tiny) * up;   // of the displacements
        dy.f_g0 = 1.5f * up * E * E * sc2;
        dy.f_g1 = r3 * E * sc;
        // criterion 1: a and f are off by at most sqrt(3) (E |s_rel| + Es |r|) + 3 E Es, |r| <= R + |s_i| + |s_j|
        dy.f_c1 = r3 * (E + Es) * sc;
        dy.f_c0 = ((0.5f * r3 * Rc * Es + 1.5f * E * Es) * up + (0x1p-19f * D + 0x1p-18f * 12.f * X) * s) * sc2;
    } else {
        E = (0x1p-21f * X + e32 + tiny) * up;
        const float Eh = (0x1p-11f * s + 0x1p-20f * s + tiny) * up;   // of half displacements
        slack += 0x1p-19f * X * X;   // the products of the low parts
        dy.f_g0 = 1.5f * up * (E * E + Eh * Eh) * sc2;
        dy.f_g1 = r3 * (E + Eh) * sc;
        dy.f_c0 = dy.f_c1 = 0.f;
    }
    dy.f_image = image;
    dy.f_scale = sc * z * in.f_unit;
    dy.f_dts = dy.f_scale * dy.dtf;
    dy.f_rt = 2.f * r3 * E * sc;
    dy.f_slack = slack * up * sc2;
    dy.f_thr = (R2 + 2.f * r3 * E * Rc + slack * up) * sc2;
    dy.f_box = (Rc * up + 0x1p-9f * D + 4.f * far + (in.f64 ? 0x1p-18f * lmax : 0.f)) / z * in.f_len;
    // speeds or timesteps out of binary32's range (binary64 states set later): every pair passes
    if (!(displacement < 0x1p100 * in.f_len && dy.dt > 0x1p-100 && dy.dt < 0x1p100)) {
        dy.f_scale = dy.f_dts = dy.f_g0 = dy.f_g1 = dy.f_c1 = dy.f_rt = 0.f;
        dy.f_c0 = dy.f_thr = dy.f_slack = 1.f;
        dy.f_box = __int_as_float(0x7f800000);
    }
}

__device__ void step_bookkeeping(InstDyn* dyn, const InstDev* inst, int n_inst, DevState* st, const Geo& geo,
                                 int bump) {
    for (int i = threadIdx.x; i < n_inst; i += blockDim.x) {
        const unsigned long long nx = dyn[i].vmax2_next;
        dyn[i].vmax2_cur = nx;
        dyn[i].vmax2_next = 0ull;
        const double vmax = sqrt(__longlong_as_double((long long)nx));
        // timestep of the next step: the configured one, or dx_min / v_max(t)
        // (adaptive; the previous one while every particle is at rest)
        const double prev = dyn[i].dt;
        double dt = inst[i].dt;
        if (inst[i].adaptive) dt = vmax > 0.0 ? inst[i].dx_min / vmax : (prev > 0.0 ? prev : inst[i].dt);
        if (bump) {
            dyn[i].dt_prev = prev;
            dyn[i].time += prev;
        } else {   // state set: no step taken yet
            dyn[i].dt_prev = dt;
        }
        dyn[i].dt = dt;
        dyn[i].dtf = (float)dt;
        const double D = sqrt(inst[i].R2) + 2.0 * vmax * dt;
        for (int d = 0; d < 3; ++d) {
            const double Dp = D * 1.001 + 1e-5 * geo.L[d];
            const double r = Dp / inst[i].w[d];
            int k = inst[i].M[d];
            if (r < (double)inst[i].M[d]) k = (int)ceil(r);
            dyn[i].k[d] = k < 1 ? 1 : k;
        }
        // Moment sums (fixed point): over the instance's n particles |v_d| <= v_max,
        // v_d^2 <= v_max^2, and a collided particle's |W| = |r_ij(t_poca) . dv| <=
        // R (1 + sqrt 2) v_max (the pair's PoCA distance is at most R, and the
        // pair's energy bounds the pre-collision speed by sqrt 2 v_max); the
        // factors 1 + 1e-6 and 4 cover the rounding of |v|^2 and of W.
        const double nn = (double)(inst[i].n > 0 ? inst[i].n : 1);
        const double vm = vmax * (1.0 + 1e-6);
        dyn[i].mom_e[0] = vm > 0.0 ? fixed_exponent(nn * vm) : 120;
        dyn[i].mom_e[1] = vm > 0.0 ? fixed_exponent(nn * vm * vm) : 120;
        const double wm = nn * 4.0 * sqrt(inst[i].R2) * vm;
        dyn[i].mom_e[2] = wm > 0.0 ? fixed_exponent(wm) : 120;
        dyn[i].p_image = 0;
        for (int d = 0; d < geo.dim; ++d)
            if (geo.bc[d] == KMC_BC_PERIODIC && D * 1.001 >= 0.499 * geo.L[d]) dyn[i].p_image = 1;
        dyn[i].p_slack = (float)(0x1p-19 * D * D);
        if (inst[i].search == kSearchFilter) filter_constants(dyn[i], inst[i], geo, vmax * dt);
    }
    if (threadIdx.x == 0 && bump) st->step += 1u;
}

__global__ void __launch_bounds__(kScanThreads) scan_kernel(uint32_t* __restrict__ count,
                                                            uint32_t* __restrict__ start,
                                                            unsigned long long* status, InstDyn* dyn,
                                                            const InstDev* inst, int n_inst, DevState* st,
                                                            Geo geo, int bump) {
    __shared__ uint32_t s_tile;
    __shared__ uint32_t s_warp[kScanThreads / 32];
    __shared__ uint32_t s_prefix;
    if (threadIdx.x == 0) s_tile = (uint32_t)atomicAdd(&status[0], 1ull);
    __syncthreads();
    const uint32_t tile = s_tile;
    if (tile == 0) step_bookkeeping(dyn, inst, n_inst, st, geo, bump);
    // the test of the bounded wait lowers the cap and holds back one tile's status
    const uint32_t cap = st->spin_cap ? st->spin_cap : kSpinCap;
    const bool publish = st->hold_tile1 != tile + 1u;

    const unsigned lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    const size_t base = (size_t)tile * kScanTile + (size_t)threadIdx.x * kScanItems;
    uint32_t it[kScanItems];
    const uint4* src = reinterpret_cast<const uint4*>(count + base);
#pragma unroll
    for (int q = 0; q < kScanItems / 4; ++q) {
        const uint4 v = src[q];
        it[4 * q + 0] = v.x; it[4 * q + 1] = v.y; it[4 * q + 2] = v.z; it[4 * q + 3] = v.w;
    }
    uint32_t total = 0;
#pragma unroll
    for (int i = 0; i < kScanItems; ++i) {
        const uint32_t c = it[i];
        it[i] = total;          // exclusive within the thread
        total += c;
    }
    // block-wide exclusive scan of the thread totals
    uint32_t inc = total;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
        if ((int)lane >= o) inc += y;
    }
    if (lane == 31) s_warp[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        uint32_t w = lane < kScanThreads / 32 ? s_warp[lane] : 0u;
        uint32_t wi = w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, wi, o);
            if ((int)lane >= o) wi += y;
        }
        const uint32_t aggregate = __shfl_sync(0xffffffffu, wi, kScanThreads / 32 - 1);
        if (lane < kScanThreads / 32) s_warp[lane] = wi - w;  // exclusive warp offsets
        // decoupled look-back
        uint32_t prefix = 0;
        if (tile == 0) {
            if (lane == 0 && publish) atomicExch(&status[1], kFlagInc | (unsigned long long)aggregate);
        } else {
            if (lane == 0 && publish) atomicExch(&status[1 + tile], kFlagAgg | (unsigned long long)aggregate);
            long long pred = (long long)tile - 1;
            bool done = false;
            while (!done) {
                const long long t = pred - (long long)lane;
                unsigned long long sv = kFlagInc;
                if (t >= 0) {
                    uint32_t spins = 0;
                    for (;;) {
                        sv = load_status(&status[1 + t]);
                        if ((sv >> 32) != 0ull) break;
                        if (++spins > cap) {
                            atomicOr(&st->error, kErrScanTimeout);
                            sv = kFlagInc;
                            break;
                        }
                        if (spins > 16) __nanosleep(64);
                    }
                }
                const uint32_t flag = (uint32_t)(sv >> 32);
                const uint32_t val = (uint32_t)sv;
                const unsigned incl = __ballot_sync(0xffffffffu, flag == 2u);
                uint32_t contrib;
                if (incl) {
                    const int first = __ffs(incl) - 1;
                    contrib = ((int)lane <= first) ? val : 0u;
                    done = true;
                } else {
                    contrib = val;
                    pred -= 32;
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) contrib += __shfl_xor_sync(0xffffffffu, contrib, o);
                prefix += contrib;
            }
            if (lane == 0 && publish)
                atomicExch(&status[1 + tile], kFlagInc | (unsigned long long)(prefix + aggregate));
        }
        if (lane == 0) s_prefix = prefix;
    }
    __syncthreads();
    const uint32_t off = s_prefix + s_warp[warp] + (inc - total);
    uint4* dst = reinterpret_cast<uint4*>(start + base);
    uint4* clr = reinterpret_cast<uint4*>(count + base);
#pragma unroll
    for (int q = 0; q < kScanItems / 4; ++q) {
        dst[q] = make_uint4(off + it[4 * q], off + it[4 * q + 1], off + it[4 * q + 2], off + it[4 * q + 3]);
        clr[q] = make_uint4(0u, 0u, 0u, 0u);
    }
}

// Fixed-point sum -> binary64 (exact below 2^53, correctly rounded above).  The
// scaling by 2^-e, |e| <= 120, is an addition to the exponent: a non-zero sum
// lies in [1, 2^63).  (ldexp took a dozen binary64 operations, which run at 1/64 of
// the binary32 rate.)
__device__ __forceinline__ double unfix(unsigned long long a, int e) {
    const double x = (double)(long long)a;
    return x == 0.0 ? 0.0 : __longlong_as_double(__double_as_longlong(x) - ((long long)e << 52));
}

// a / b, correctly rounded, from the correctly rounded reciprocal r of an integer b
// below 2^32 (a count, or 3), for quotients away from the ends of the range, as here.
// a r is within 2^-52 of the quotient, the step on its residual then within 2^-104 before
// the last rounding.  That rounds as the quotient does, because no quotient comes as near
// to the middle m of two neighbours: |a - b m| is not zero (a would need 54 bits) and a multiple
// of m's last place, 2^-54 m or more, so |a / b - m| is at least 2^-86 m.
__device__ __forceinline__ double div_rcp(double a, double b, double r) {
    const double q = a * r;
    return fma(fma(-q, b, a), r, q);
}

// Derived per-c-bin moments (Eqs. vel_b, stress, 18, 19 with the readings
// u = Sum v / N, v_rms^2 = <|v - u|^2>, T = v_rms^2 / 3, p = n T + virial),
// and the per-instance integer totals of the fixed-point sums (exact, so the
// order of the atomics does not matter): a block whose bins belong to one
// instance adds once per total.  Bound by the binary64 operations; rows of the
// result leave through shared memory as whole runs.  1,000,000 c-bins, GB300: 0.329 ms
// with a division per quotient, ldexp, row-strided stores and seven atomics per
// warp -> 0.111 ms.
constexpr int kFinThreads = 128;
__global__ void __launch_bounds__(kFinThreads) finalize_bins_kernel(const InstDev* __restrict__ inst,
                                                                    const InstDyn* __restrict__ dyn, Geo geo,
                                                                    const unsigned long long* __restrict__ acc,
                                                                    double* __restrict__ mom, unsigned long long* gacc,
                                                                    int64_t n_bins, int64_t bins_per_inst, double Vc) {
    constexpr int kWarps = kFinThreads / 32;
    __shared__ double out[kFinThreads][17];              // a row of 8 raw and 8 derived (17: no bank conflicts)
    __shared__ unsigned long long part[kWarps][7];
    const int64_t first = (int64_t)blockIdx.x * kFinThreads, bidx = first + threadIdx.x;
    const bool valid = bidx < n_bins;
    const int i = valid ? (int)(bidx / bins_per_inst) : 0;
    const bool one = first / bins_per_inst == min(first + kFinThreads - 1, n_bins - 1) / bins_per_inst;   // block-uniform
    unsigned long long t[7] = {0, 0, 0, 0, 0, 0, 0};
    if (valid) {
        const InstDyn& D = dyn[i];
        unsigned long long ai[kAccFields];
        const ulonglong2* a2 = reinterpret_cast<const ulonglong2*>(acc + bidx * kAccFields);   // 80 bytes: aligned
#pragma unroll
        for (int k = 0; k < kAccFields / 2; ++k) {
            const ulonglong2 v = a2[k];
            ai[2 * k] = v.x;
            ai[2 * k + 1] = v.y;
        }
        t[0] = ai[0];
        t[1] = ai[4] + ai[5] + ai[6];
        t[2] = ai[1];
        t[3] = ai[2];
        t[4] = ai[3];
        t[5] = ai[7];
        t[6] = ai[8];
        double* o = out[threadIdx.x];
        double r[8];
        r[0] = (double)(long long)ai[0];
        for (int k = 1; k <= 3; ++k) r[k] = unfix(ai[k], D.mom_e[0]);
        for (int k = 4; k <= 6; ++k) r[k] = unfix(ai[k], D.mom_e[1]);
        r[7] = unfix(ai[7], D.mom_e[2]);
        for (int k = 0; k < 8; ++k) o[k] = r[k];
        const double N = r[0];
        double vr = 0.0;
        const double svr = unfix(ai[9], D.mom_e[0]);
        if (N <= 0.0) {
            for (int k = 8; k < 16; ++k) o[k] = 0.0;
        } else {
            const double dt = D.dt_prev;   // the step whose collisions W sums
            const double rN = __drcp_rn(N);
            const double ux = div_rcp(r[1], N, rN), uy = div_rcp(r[2], N, rN), uz = div_rcp(r[3], N, rN);
            const double c2 = div_rcp(r[4] + r[5] + r[6], N, rN) - (ux * ux + uy * uy + uz * uz);
            // f velocity degrees of freedom
            const double T = geo.vdim == 2 ? 0.5 * c2 : div_rcp(c2, 3.0, 1.0 / 3.0);
            const double nd = N / Vc;
            const double pkin = nd * T;
            const double pvir = r[7] == 0.0 ? 0.0 : r[7] / (2.0 * geo.dim * Vc * dt);
            o[8] = nd; o[9] = ux; o[10] = uy; o[11] = uz;
            o[12] = T; o[13] = pkin; o[14] = pvir; o[15] = pkin + pvir;
            if (svr != 0.0) vr = div_rcp(svr, N, rN);   // Eq. vel_r
        }
        *reinterpret_cast<double2*>(mom + 16 * n_bins + 2 * bidx) = make_double2(svr, vr);
    }
#pragma unroll
    for (int k = 0; k < 7; ++k) {
        if (one) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) t[k] += __shfl_xor_sync(0xffffffffu, t[k], o);
            if ((threadIdx.x & 31u) == 0) part[threadIdx.x >> 5][k] = t[k];
        } else if (valid && t[k]) {
            atomicAdd(gacc + (size_t)i * 8 + k, t[k]);
        }
    }
    __syncthreads();
    if (one && threadIdx.x < 7) {
        unsigned long long s = 0;
        for (int w = 0; w < kWarps; ++w) s += part[w][threadIdx.x];
        if (s) atomicAdd(gacc + (size_t)(first / bins_per_inst) * 8 + threadIdx.x, s);
    }
    const int words = 8 * (int)min((int64_t)kFinThreads, n_bins - first);
    for (int w = threadIdx.x; w < words; w += kFinThreads) {
        mom[8 * first + w] = out[w >> 3][w & 7];
        mom[8 * (n_bins + first) + w] = out[w >> 3][8 + (w & 7)];
    }
}

// Per-instance totals (N, energy, momentum, virial, pairs) from the integer
// totals, converted once; the totals are cleared for the next reduction.
__global__ void finalize_glob_kernel(const InstDyn* __restrict__ dyn, unsigned long long* gacc,
                                     double* __restrict__ glob, int n_inst) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n_inst) return;
    const InstDyn& D = dyn[i];
    unsigned long long* t = gacc + (size_t)i * 8;
    double* g = glob + (int64_t)i * 8;
    g[0] = (double)(long long)t[0];
    g[1] = 0.5 * unfix(t[1], D.mom_e[1]);
    g[2] = unfix(t[2], D.mom_e[0]);
    g[3] = unfix(t[3], D.mom_e[0]);
    g[4] = unfix(t[4], D.mom_e[0]);
    g[5] = unfix(t[5], D.mom_e[2]);
    g[6] = 0.5 * (double)(long long)t[6];  // collided particles / 2 = pairs
    g[7] = 0.0;
    for (int k = 0; k < 8; ++k) t[k] = 0ull;
}

}  // namespace

cudaError_t launch_scan(uint32_t* count, uint32_t* start, uint32_t n_keys, uint32_t n_tiles,
                        unsigned long long* status, InstDyn* dyn, const InstDev* inst, int n_inst,
                        DevState* st, Geo geo, int bump_step, cudaStream_t s) {
    (void)n_keys;
    cudaError_t e = cudaMemsetAsync(status, 0, sizeof(unsigned long long) * (1 + (size_t)n_tiles), s);
    if (e != cudaSuccess) return e;
    scan_kernel<<<n_tiles, kScanThreads, 0, s>>>(count, start, status, dyn, inst, n_inst, st, geo, bump_step);
    return cudaGetLastError();
}

cudaError_t launch_finalize(const InstDev* inst, const InstDyn* dyn, int n_inst, Geo geo,
                            const unsigned long long* acc, double* mom, double* glob, unsigned long long* gacc,
                            int64_t n_bins, cudaStream_t s) {
    if (n_bins == 0 || n_inst == 0) return cudaSuccess;
    const int64_t per = n_bins / n_inst;
    double Vc = 1.0;
    for (int d = 0; d < geo.dim; ++d) Vc *= geo.L[d] / (double)geo.n[d];
    finalize_bins_kernel<<<(unsigned)((n_bins + kFinThreads - 1) / kFinThreads), kFinThreads, 0, s>>>(
        inst, dyn, geo, acc, mom, gacc, n_bins, per, Vc);
    finalize_glob_kernel<<<(n_inst + 127) / 128, 128, 0, s>>>(dyn, gacc, glob, n_inst);
    return cudaGetLastError();
}

}  // namespace kmc
