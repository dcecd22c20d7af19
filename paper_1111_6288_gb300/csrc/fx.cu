// The recurrences of the FP64 operators on the integer pipes (fx_arith.h, fx_site.h), on links that launch_fx_survey
// finds fit for it.
//
// Every step of the polynomial Q P(Q^2) (Sec. 2) in FP64 is one application of H_w.  The FP64 stencil
// (dslash_kernel<double>) keeps this GPU's FP64 pipe 91 % busy at 2 multiply-adds per clock and SM, so
// it cannot get faster there.  Here the vectors of a recurrence are site-scaled 57-bit integers, the
// link products are 32 x 32 + 64-bit multiply-adds (64 per clock and SM), and only the conversions at
// the ends of a recurrence touch FP64.  Per application the result is closer to the exact one than
// FP64's (relative error 2e-17 against 1.1e-16 on random fields, 5e-17 against 2e-16 at the worst site).
#include <algorithm>
#include <atomic>
#include <cmath>
#include <type_traits>

#include "fx_site.h"
#include "ovl_internal.h"

namespace ovl {
namespace {

using fx::i64;

constexpr int FX_THREADS = 128;
// Stages of a warp's ring and blocks per SM: 2 and 4 (128 registers, 43 KB a block) against 3 and 3 (168
// registers): 257 and 268 us a launch at 24^3 x 48, 51.5 and 51.9 us at 16^3 x 32, equal at 8^3 x 16 x 12;
// four stages, two or five blocks are 5-15 % slower.
constexpr int kStages = 2;
constexpr int kBlocksPerSm = 4;
// Launches of at most this many blocks of 16 sites go to fx_split_kernel: three on each of the 152 SMs, all it
// has registers for.  Two lanes a site against eight: 6.6 / 5.1 us on 4^4 (16 blocks), 7.4 / 6.5 on 8^3 x 12,
// 7.6 / 6.6 on 9^3 x 10 (456 blocks), 7.3 / 8.7 on 8^3 x 16 (512 blocks); the derivative 10.3 / 7.7 us on 4^3 x 8,
// 11.4 / 9.3 on 9^3 x 10, 11.4 / 12.7 on 8^3 x 16.
constexpr int kSplitBlocks = 3 * 152;
constexpr int kSpinInt4 = 6 * 32;             // a lane's six components of a spinor
constexpr int kStageInt4 = kSpinInt4 + 9 * 16;  // and the links of the warp's 16 sites
constexpr int kWarpBytes = kStages * kStageInt4 * 16;

// 16 bytes, global -> shared, in the background.
__device__ __forceinline__ void copy_async16(void* dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void copy_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Two lanes of a warp per (site, right-hand side): lanes 0-15 hold row 0 and lanes 16-31 row 1 of 16
// consecutive sites.  What a lane needs comes in twelve steps: the neighbour and the link of each hop,
// then its components of psi and of the three epilogue vectors.  Each warp copies the next step into
// shared memory while it computes (the two lanes of a site share the copy of its link).
//
// Bound by the integer pipes and the register reads behind them (per lane and site about 700 32 x 32 +
// 64-bit multiply-adds of 2600 instructions), beyond L2 also by the links (576 B a site, read 1.4 times).
// Measured, mean of the two launches of a Clenshaw step against dslash_kernel<double>: 48.5 against 231 us
// at 16^3 x 32, 36.7 against 180 us for 12 systems of 8^3 x 16, 6.6 against 35 us on 4^4.  (With four limb
// products a complex product and 51 us at 16^3 x 32, one thread a site instead of two lanes took 66 us and
// operands loaded straight into registers 65 us.)
template <bool EPI, bool DUAL>
__global__ void __launch_bounds__(FX_THREADS, kBlocksPerSm) fx_dslash_kernel(const __grid_constant__ fx::Args a, int nrhs) {
    extern __shared__ int4 ring[];
    const int V = a.V;
    const int lane = threadIdx.x & 31, f = lane >> 4;
    const int site = blockIdx.x * (blockDim.x / 2) + (threadIdx.x >> 5) * 16 + (lane & 15);
    const int rhs = blockIdx.y * blockDim.y + threadIdx.y;
    const bool active = site < V && rhs < nrhs;
    const int s = min(site, V - 1), r = min(rhs, nrhs - 1);
    const i64 off = (i64)r * fx::rhs_bytes(V);
    const char* in = a.in + off;
    int4* const stages = ring + ((threadIdx.y * blockDim.x + threadIdx.x) >> 5) * (kStages * kStageInt4);
    fx::Half H;
    fx::half_setup(a, s, r, f, H);
    const char* const ux = fx::links_of_dir(a, r, 0);
    const i64 lb = fx::link_bytes(V);
    auto slot = [&](int k) { return stages + (k % kStages) * kStageInt4; };
    auto copy_spin = [&](int k, const int4* pa, const int4* pb) {
        int4* d = slot(k) + lane;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            copy_async16(d + c * 32, pa + c * fx::kTile);
            copy_async16(d + (3 + c) * 32, pb + c * fx::kTile);
        }
    };
    auto issue = [&](auto kc) {
        constexpr int k = decltype(kc)::value;
        if constexpr (k < 8) {
            constexpr int mu = fx::dir_of(k);
            const int4* p = fx::at(in, H.nb[k]);
            copy_spin(k, p + 3 * fx::kTile * f, p + fx::partner(mu, f) * fx::kTile);
            const int4* u = fx::link_at(mu == 0 ? ux : a.U + mu * lb, k % 2 == 0 ? s : H.nb[k]);
            int4* d = slot(k) + kSpinInt4 + (lane & 15);
            // lane 0 of a site copies entries 0 to 4, lane 1 the others
#pragma unroll
            for (int q = 0; q < 4; ++q) copy_async16(d + (5 * f + q) * 16, u + (5 * f + q) * fx::kTile);
            if (f == 0) copy_async16(d + 4 * 16, u + 4 * fx::kTile);
        } else {
            const char* v = k == 8 ? in : nullptr;
            if constexpr (EPI) {
                if (k == 9 && a.v1) v = a.v1 + off;
                if (k == 10 && a.v2) v = a.v2 + off;
                if (k == 11 && a.v3) v = a.v3 + off;
            }
            if (v) copy_spin(k, fx::at(v, s) + 3 * fx::kTile * f, fx::at(v, s) + (6 + 3 * f) * fx::kTile);
        }
        copy_commit();
    };
    constexpr int kSteps = EPI ? 12 : 9;
    // waits for step k, after which step k + kStages - 1 is on its way into the slot of step k - 1
    auto ready = [&](auto kc) {
        constexpr int k = decltype(kc)::value;
        __syncwarp();  // the other lanes are done with step k - 1
        if constexpr (k + kStages - 1 < kSteps) {
            issue(std::integral_constant<int, k + kStages - 1>{});
            copy_wait<kStages - 1>();
        } else {
            copy_wait<kSteps - 1 - k>();
        }
        __syncwarp();  // and every lane's copies of step k have landed
    };
    issue(std::integral_constant<int, 0>{});
    static_assert(kStages == 2, "one step is issued ahead of the loop");
    int e1 = 0, e2 = 0, e3 = 0;
    if constexpr (EPI) {
        if (a.v1) e1 = *fx::exponent_at(a.v1 + off, s);
        if (a.v2) e2 = *fx::exponent_at(a.v2 + off, s);
        if (a.v3) e3 = *fx::exponent_at(a.v3 + off, s);
    }
    auto pair_or = [&](uint64_t o) { return o | __shfl_xor_sync(0xffffffffu, o, 16); };
    {
        i64 fu[6], fl[6], bu[6], bl[6];
#pragma unroll
        for (int k = 0; k < 6; ++k) fu[k] = fl[k] = bu[k] = bl[k] = 0;
        auto step = [&](auto kc) {
            constexpr int k = decltype(kc)::value;
            ready(kc);
            const int4* d = slot(k);
            fx::half_hop<k, DUAL, 32, 16>(H, d + lane, d + 3 * 32 + lane, d + kSpinInt4 + (lane & 15), fu, fl, bu, bl);
        };
        step(std::integral_constant<int, 0>{});
        step(std::integral_constant<int, 1>{});
        step(std::integral_constant<int, 2>{});
        step(std::integral_constant<int, 3>{});
        step(std::integral_constant<int, 4>{});
        step(std::integral_constant<int, 5>{});
        step(std::integral_constant<int, 6>{});
        step(std::integral_constant<int, 7>{});
        if constexpr (DUAL) {
            int ed = fx::dual_split(H, fu, fl, bu, bl);
            ed = fx::deriv_scale(H, fu, fl, pair_or(fx::or_bits(fu, fl)), ed);
            ed = fx::normalise(fu, fl, pair_or(fx::or_bits(fu, fl)), ed);
            if (active) {
                int4* o = fx::at(a.out2 + off, s);
                fx::store_spin(o, f, fu);
                fx::store_spin(o, 3 - f, fl);
                if (f == 0) *fx::exponent_at(a.out2 + off, s) = H.bad_x ? fx::kNanExp : ed;
            }
        }
    }
#pragma unroll
    for (int k = 0; k < 6; ++k) H.own[k] += __shfl_xor_sync(0xffffffffu, H.oth[k], 16);
    int4 u[3], l[3];
    auto fetch = [&](auto kc) {
        ready(kc);
        const int4* d = slot(decltype(kc)::value) + lane;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            u[c] = d[c * 32];
            l[c] = d[(3 + c) * 32];
        }
    };
    fetch(std::integral_constant<int, 8>{});
    fx::mass_term(a, H, u, l);
    int E = H.eref - 1;
    bool bad = H.eref > fx::kNanTest;
    if constexpr (EPI) {
        const int ej = E + a.c0e;
        E = ej;
        if (a.v1) E = max(E, fx::term_exp(e1, a.c1));
        if (a.v2) E = max(E, fx::term_exp(e2, a.c2));
        if (a.v3) E = max(E, fx::term_exp(e3, a.c3));
        bad = bad || e1 > fx::kNanTest || e2 > fx::kNanTest || e3 > fx::kNanTest;
        const int d = fx::align_shift(E, ej);
        const i64 half = fx::half_of(d);
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            H.up[k] = fx::shifted(H.up[k], d, half);
            H.own[k] = fx::shifted(H.own[k], d, half);
        }
        auto term = [&](auto kc, bool there, int e, const fx::Coef& c) {
            fetch(kc);
            if (!there) return;
            fx::add_term(H.up, u, e, c, E);
            fx::add_term(H.own, l, e, c, E);
        };
        term(std::integral_constant<int, 9>{}, a.v1 != nullptr, e1, a.c1);
        term(std::integral_constant<int, 10>{}, a.v2 != nullptr, e2, a.c2);
        term(std::integral_constant<int, 11>{}, a.v3 != nullptr, e3, a.c3);
    }
    E = fx::normalise(H.up, H.own, pair_or(fx::or_bits(H.up, H.own)), E);
    if (active) {
        int4* o = fx::at(a.out + off, s);
        fx::store_spin(o, f, H.up);
        fx::store_spin(o, 2 + f, H.own);
        if (f == 0) *fx::exponent_at(a.out + off, s) = bad ? fx::kNanExp : E;
    }
}

// The same on few sites, eight lanes a site: there a launch takes as long as one warp's instructions, one
// every four to five cycles, whatever the memory does (a ring that holds every step took 6.1 us on 4^4 instead
// of 6.4).  4^4: 6.6 -> 5.1 us.  A block has 16 sites; each of its four warps does the two hops of one direction,
// operands loaded straight into registers, and the sums meet in shared memory, where each thread takes three of a site's 24
// numbers through the epilogue.  The sums are integers, so the bits are those of fx_dslash_kernel.
template <bool EPI, bool DUAL>
__global__ void __launch_bounds__(128) fx_split_kernel(const __grid_constant__ fx::Args a) {
    __shared__ i64 sums[4][24][17];
    __shared__ int eref_of[16], e0_of[16];
    const int V = a.V, warp = threadIdx.x >> 5, lane = threadIdx.x & 31, f = lane >> 4;
    const int first = blockIdx.x * 16, r = blockIdx.y;
    const i64 off = (i64)r * fx::rhs_bytes(V);
    const char* in = a.in + off;
    // numbers 3 t .. 3 t + 2 of site first + j
    const int j = threadIdx.x >> 3, t = threadIdx.x & 7, sj = min(first + j, V - 1);
    auto number = [&](const char* v, int q) {
        const int k = 3 * t + q;
        return (const int2*)(fx::at(v, sj) + (k >> 1) * fx::kTile) + (k & 1);
    };
    int2 x[3], x1[3], x2[3], x3[3];
    int e1 = 0, e2 = 0, e3 = 0;
    auto fetch = [&](const char* v, int2(&d)[3]) {
#pragma unroll
        for (int q = 0; q < 3; ++q) d[q] = v ? *number(v + off, q) : make_int2(0, 0);
        return v ? *fx::exponent_at(v + off, sj) : 0;
    };
    fetch(a.in, x);
    if constexpr (EPI) {
        e1 = fetch(a.v1, x1);
        e2 = fetch(a.v2, x2);
        e3 = fetch(a.v3, x3);
    }
    fx::Half H;
    const int s = min(first + (lane & 15), V - 1);
    fx::half_setup(a, s, r, f, H);
    if (threadIdx.x < 16) {
        eref_of[threadIdx.x] = H.eref;
        e0_of[threadIdx.x] = H.e0;
    }
    i64 fu[6], fl[6], bu[6], bl[6];
#pragma unroll
    for (int k = 0; k < 6; ++k) fu[k] = fl[k] = bu[k] = bl[k] = 0;
    auto both = [&](auto kc) {
        constexpr int k = decltype(kc)::value, mu = fx::dir_of(k);
        const char* u = mu == 0 ? fx::links_of_dir(a, r, 0) : a.U + mu * fx::link_bytes(V);
        const int4* p = fx::at(in, H.nb[k]);
        const int4* m = fx::at(in, H.nb[k + 1]);
        fx::half_hop<k, DUAL, fx::kTile, fx::kTile>(H, p + 3 * fx::kTile * f, p + fx::partner(mu, f) * fx::kTile,
                                                    fx::link_at(u, s), fu, fl, bu, bl);
        fx::half_hop<k + 1, DUAL, fx::kTile, fx::kTile>(H, m + 3 * fx::kTile * f, m + fx::partner(mu, f) * fx::kTile,
                                                        fx::link_at(u, H.nb[k + 1]), fu, fl, bu, bl);
        if constexpr (DUAL && mu == 0) {
            auto pair_or = [&](uint64_t o) { return o | __shfl_xor_sync(0xffffffffu, o, 16); };
            int ed = fx::dual_split(H, fu, fl, bu, bl);
            ed = fx::deriv_scale(H, fu, fl, pair_or(fx::or_bits(fu, fl)), ed);
            ed = fx::normalise(fu, fl, pair_or(fx::or_bits(fu, fl)), ed);
            if (first + (lane & 15) < V) {
                int4* o = fx::at(a.out2 + off, s);
                fx::store_spin(o, f, fu);
                fx::store_spin(o, 3 - f, fl);
                if (f == 0) *fx::exponent_at(a.out2 + off, s) = H.bad_x ? fx::kNanExp : ed;
            }
        }
        const i64 neg = k == 0 ? -(i64)f : 0;  // the y hops' lower spin; the z hops' has its sign already
#pragma unroll
        for (int q = 0; q < 6; ++q) {
            sums[k / 2][6 * f + q][lane & 15] = H.up[q];
            sums[k / 2][6 * (mu < 2 ? 3 - f : 2 + f) + q][lane & 15] = mu < 2 ? (H.oth[q] ^ neg) - neg : H.own[q];
        }
    };
    if (warp == 0) both(std::integral_constant<int, 0>{});
    else if (warp == 1) both(std::integral_constant<int, 2>{});
    else if (warp == 2) both(std::integral_constant<int, 4>{});
    else both(std::integral_constant<int, 6>{});
    __syncthreads();
    const int eref = eref_of[j];
    bool bad = eref > fx::kNanTest;
    i64 v[3];
    {
        const fx::Coef D = a.scale->diag;
        const int d = fx::align_shift(eref, e0_of[j] + D.e);
        const i64 half = fx::half_of(d);
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            const int k = 3 * t + q;
            const i64 sum = (sums[0][k][j] + sums[1][k][j]) + (sums[2][k][j] + sums[3][k][j]);
            fx::Sum m = fx::start(half);
            fx::mac(m, D.m, fx::Num{x[q].x, x[q].y});
            const i64 mass = fx::value(m) >> d;
            v[q] = t < 4 ? mass - sum : sum - mass;
        }
    }
    int E = eref - 1;
    if constexpr (EPI) {
        const int ej = E + a.c0e;
        E = ej;
        if (a.v1) E = max(E, fx::term_exp(e1, a.c1));
        if (a.v2) E = max(E, fx::term_exp(e2, a.c2));
        if (a.v3) E = max(E, fx::term_exp(e3, a.c3));
        bad = bad || e1 > fx::kNanTest || e2 > fx::kNanTest || e3 > fx::kNanTest;
        const int d = fx::align_shift(E, ej);
        const i64 half = fx::half_of(d);
#pragma unroll
        for (int q = 0; q < 3; ++q) v[q] = fx::shifted(v[q], d, half);
        if (a.v1) fx::add_term(v, x1, e1, a.c1, E);
        if (a.v2) fx::add_term(v, x2, e2, a.c2, E);
        if (a.v3) fx::add_term(v, x3, e3, a.c3, E);
    }
    uint64_t o = 0;
#pragma unroll
    for (int q = 0; q < 3; ++q) o |= (uint64_t)(v[q] ^ (v[q] >> 63));
#pragma unroll
    for (int m = 1; m < 8; m *= 2) o |= __shfl_xor_sync(0xffffffffu, o, m);
    E = fx::normalise(v, o, E);
    if (first + j < V) {
        char* out = a.out + off;
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            const fx::Num z = fx::split(v[q]);
            *const_cast<int2*>(number(out, q)) = make_int2(z.hi, z.lo);
        }
        if (t == 0) *fx::exponent_at(out, sj) = bad ? fx::kNanExp : E;
    }
}

// max over the links of the largest squared row or column norm, as the bits of a double (positive
// doubles order like their bits; a NaN orders above all of them)
__global__ void fx_link_norm_k(const double2* __restrict__ U, int V, unsigned long long* __restrict__ out) {
    unsigned long long best = 0;
    for (i64 idx = (i64)blockIdx.x * blockDim.x + threadIdx.x; idx < 4LL * V; idx += (i64)gridDim.x * blockDim.x) {
        const int mu = (int)(idx / V), s = (int)(idx % V);
        const double2* u = U + (i64)mu * 9 * V + s;
        double row[3] = {0, 0, 0}, col[3] = {0, 0, 0};
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            const double2 z = u[(i64)k * V];
            const double q = z.x * z.x + z.y * z.y;
            row[k / 3] += q;
            col[k % 3] += q;
        }
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            // the sign bit of a NaN is cleared so that it orders above infinity
            const unsigned long long x = (unsigned long long)__double_as_longlong(row[i]) & 0x7fffffffffffffffULL;
            const unsigned long long y = (unsigned long long)__double_as_longlong(col[i]) & 0x7fffffffffffffffULL;
            best = x > best ? x : best;
            best = y > best ? y : best;
        }
    }
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long v = __shfl_down_sync(0xffffffffu, best, o);
        best = v > best ? v : best;
    }
    if ((threadIdx.x & 31) == 0) atomicMax(out, best);
}

// Smallest of the warp's values, given as bits of doubles that are not negative.
__device__ __forceinline__ unsigned long long warp_min(unsigned long long v) {
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long w = __shfl_down_sync(0xffffffffu, v, o);
        v = w < v ? w : v;
    }
    return v;
}

// out[1], out[2] of launch_fx_survey (out[0] is fx_link_norm_k's): a thread per site, the links of its eight hops
__global__ void __launch_bounds__(128) fx_survey_k(const double2* __restrict__ U, Geom g, unsigned long long* __restrict__ out) {
    unsigned long long least = ~0ULL, mixed = ~0ULL;
    const int V = g.V;
    for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < V; s += gridDim.x * blockDim.x) {
        double share[3][3] = {};
        double norm = INFINITY;
        int rest = s, stride = 1;
        for (int mu = 0; mu < 4; ++mu) {
            const int L = g.L[mu], x = rest % L;
            rest /= L;
            const bool open = g.bcf[mu] == 0.0;
            for (int back = 0; back < 2; ++back) {
                if (open && x == (back ? 0 : L - 1)) continue;
                const int site = back ? (x == 0 ? s + (L - 1) * stride : s - stride) : s;
                const double2* u = U + (i64)mu * 9 * V + site;
                double row[3] = {0, 0, 0}, col[3] = {0, 0, 0};
#pragma unroll
                for (int k = 0; k < 9; ++k) {
                    const double2 z = u[(i64)k * V];
                    const double q = z.x * z.x + z.y * z.y, m = fmax(fabs(z.x), fabs(z.y));
                    row[k / 3] += q;
                    col[k % 3] += q;
                    // forward: entry (a, b) brings b to a; backward, U^+: b = row, a = column
                    if (back) share[k % 3][k / 3] += m;
                    else share[k / 3][k % 3] += m;
                }
#pragma unroll
                for (int i = 0; i < 3; ++i) norm = fmin(norm, fmin(row[i], col[i]));
            }
            stride *= L;
        }
        const double a = fmin(fmin(share[0][1], share[1][0]), fmin(share[0][2], share[2][0]));
        const double m = fmin(a, fmin(share[1][2], share[2][1]));
        least = min(least, (unsigned long long)__double_as_longlong(norm));
        mixed = min(mixed, (unsigned long long)__double_as_longlong(m));
    }
    least = warp_min(least);
    mixed = warp_min(mixed);
    if ((threadIdx.x & 31) == 0) {
        atomicMin(out + 1, least);
        atomicMin(out + 2, mixed);
    }
}

// a 2^k to the nearest integer, a = hi + lo
__device__ __forceinline__ i64 to_int(double hi, double lo, int k) {
    return __double2ll_rn(scalbn(hi, k)) + __double2ll_rn(scalbn(lo, k));
}

// le: g U is stored divided by 2^le, so that no row or column norm exceeds 1.05 (and the largest is above
// 0.52); the mass coefficient 2 (4 + m0) g = d_hi + d_lo in the units of the hops where it is below 7.5.
__global__ void fx_scale_k(fx::Scale* __restrict__ sc, double g, double d_hi, double d_lo) {
    const double q = __longlong_as_double((long long)sc->norm_bits);
    int le = 0;
    if (!(q < INFINITY)) {
        le = fx::kNanExp;
    } else if (q > 0.0) {
        const double n = sqrt(q) * g * (1.0 / 1.05);
        le = ilogb(n);
        if (scalbn(n, -le) > 1.0) ++le;
    }
    fx::Coef c{{0, 0}, 0, 0};
    if (le <= fx::kNanTest && d_hi != 0.0) {
        int k = ilogb(d_hi) + 1 - (fx::kBits + 2);  // units in which it stays below 2^58
        if (le - fx::kBits >= k - 3 && fabs(scalbn(d_hi, -le)) < 7.5) k = le - fx::kBits;
        c.m = fx::split(to_int(d_hi, d_lo, -k));
        c.e = k + fx::kBits;
    }
    sc->le = le;
    sc->diag = c;
}

// The link entry times g = g_hi + g_lo as an integer in units of 2^(le - 56).
__device__ __forceinline__ fx::Num fx_entry(double x, double g_hi, double g_lo, int le) {
    const double p = x * g_hi;
    return fx::split(to_int(p, fma(x, g_hi, -p) + x * g_lo, fx::kBits - le));
}
__device__ __forceinline__ int4 fx_link(double re, double im, double g_hi, double g_lo, int le) {
    if (le > fx::kNanTest) return make_int4(0, 0, 0, 0);
    const fx::Num a = fx_entry(re, g_hi, g_lo, le), b = fx_entry(im, g_hi, g_lo, le);
    return make_int4(a.hi, a.lo, b.hi, b.lo);
}

// FP64 links [4][9][V] -> [4] tiled; one thread per site and direction (blockIdx.y)
__global__ void fx_pack_links_k(const double2* __restrict__ U, char* __restrict__ out, int V, double g_hi, double g_lo,
                                const fx::Scale* __restrict__ sc) {
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= V) return;
    const int le = sc->le;
    int4* o = fx::link_at(out + blockIdx.y * fx::link_bytes(V), s);
    const double2* u = U + (i64)blockIdx.y * 9 * V + s;
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        const double2 z = u[(i64)k * V];
        o[k * fx::kTile] = fx_link(z.x, z.y, g_hi, g_lo, le);
    }
}

// x links times exp(i phase[q] t); one thread per site and phase
__global__ void fx_xlinks_k(const double2* __restrict__ U, char* __restrict__ out, int V, int slice,
                            const double* __restrict__ phases, double g_hi, double g_lo,
                            const fx::Scale* __restrict__ sc) {
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= V) return;
    double sn, cs;
    sincos(phases[blockIdx.y] * (double)(s / slice), &sn, &cs);
    const int le = sc->le;
    int4* o = fx::link_at(out + blockIdx.y * fx::link_bytes(V), s);
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        const double2 z = U[(i64)k * V + s];
        o[k * fx::kTile] = fx_link(z.x * cs - z.y * sn, z.x * sn + z.y * cs, g_hi, g_lo, le);
    }
}

// FP64 spinors (12 planes of double2) times factor -> fixed point (factor 0: zeros, whatever they are)
__global__ void __launch_bounds__(128) fx_from_f64_k(const double2* __restrict__ in, char* __restrict__ out, int V,
                                                     double factor) {
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= V) return;
    const double2* q = in + (i64)blockIdx.y * 12 * V + s;
    double2 p[12];
    unsigned long long top = 0;
#pragma unroll
    for (int k = 0; k < 12; ++k) {
        p[k] = q[(i64)k * V];
        p[k].x = factor == 0.0 ? 0.0 : p[k].x * factor;
        p[k].y = factor == 0.0 ? 0.0 : p[k].y * factor;
        const unsigned long long x = (unsigned long long)__double_as_longlong(p[k].x) & 0x7fffffffffffffffULL;
        const unsigned long long y = (unsigned long long)__double_as_longlong(p[k].y) & 0x7fffffffffffffffULL;
        top = x > top ? x : top;
        top = y > top ? y : top;
    }
    i64 J[4][6];
    int e;
    if (top == 0 || top >= 0x7ff0000000000000ULL) {
#pragma unroll
        for (int k = 0; k < 24; ++k) J[k / 6][k % 6] = 0;
        e = top == 0 ? fx::kZeroExp : fx::kNanExp;
    } else {
        e = ilogb(__longlong_as_double((long long)top)) + 1 - fx::kBits;
#pragma unroll
        for (int k = 0; k < 12; ++k) {
            J[k / 3][2 * (k % 3)] = __double2ll_rn(scalbn(p[k].x, -e));
            J[k / 3][2 * (k % 3) + 1] = __double2ll_rn(scalbn(p[k].y, -e));
        }
    }
    char* o = out + (i64)blockIdx.y * fx::rhs_bytes(V);
#pragma unroll
    for (int spin = 0; spin < 4; ++spin) fx::store_spin(fx::at(o, s), spin, J[spin]);
    *fx::exponent_at(o, s) = e;
}

__global__ void __launch_bounds__(128) fx_to_f64_k(const char* __restrict__ in, double2* __restrict__ out, int V,
                                                   double factor) {
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= V) return;
    const char* b = in + (i64)blockIdx.y * fx::rhs_bytes(V);
    const int e = *fx::exponent_at(b, s);
    double2* o = out + (i64)blockIdx.y * 12 * V + s;
#pragma unroll
    for (int k = 0; k < 12; ++k) {
        double2 z;
        if (e > fx::kNanTest) {
            z.x = z.y = __longlong_as_double(0x7ff8000000000000LL);
        } else {
            const int4 v = fx::at(b, s)[k * fx::kTile];
            z.x = scalbn(factor * (double)(((i64)v.x << fx::kLimb) + v.y), e);
            z.y = scalbn(factor * (double)(((i64)v.z << fx::kLimb) + v.w), e);
        }
        o[(i64)k * V] = z;
    }
}

// A coefficient of zero has an exponent below every other, so that its term sets no unit for the sum.
fx::Coef make_coef(double c) {
    fx::Coef o{{0, 0}, 0, 0};
    if (c == 1.0 || c == -1.0) o.unit = (int)c;
    int k = 0;
    const double f = std::frexp(c, &k);  // c = f 2^k, 1/2 <= |f| < 1
    o.m = fx::split(std::llrint(std::ldexp(f, fx::kBits + 2)));
    o.e = c == 0.0 ? -(1 << 22) : k - 2;
    return o;
}

}  // namespace

size_t fx_rhs_bytes(int V) { return (size_t)fx::rhs_bytes(V); }
constexpr size_t kScaleBytes = 64;
static_assert(sizeof(fx::Scale) <= kScaleBytes, "Scale");
size_t fx_link_bytes(int V) { return (size_t)(4 * fx::link_bytes(V)) + kScaleBytes; }
size_t fx_xlink_bytes(int V) { return (size_t)fx::link_bytes(V); }

namespace {
fx::Scale* scale_of(const void* links, int V) { return (fx::Scale*)((char*)links + 4 * fx::link_bytes(V)); }

// g = sqrt(a) as hi + lo
void root_hi_lo(double a, double* hi, double* lo) {
    *hi = std::sqrt(a);
    *lo = std::fma(-*hi, *hi, a) / (2.0 * *hi);
}
}  // namespace

namespace {
// The kernel's shared memory is above the default limit: raised once per device.
template <bool EPI, bool DUAL>
void fx_launch(const fx::Args& a, dim3 grid, dim3 block, int nrhs, cudaStream_t s) {
    static std::atomic<unsigned long long> raised{0};
    int dev = 0;
    cudaGetDevice(&dev);
    const unsigned long long bit = 1ULL << (dev & 63);
    if (dev > 63 || !(raised.load(std::memory_order_relaxed) & bit)) {
        cudaFuncSetAttribute(fx_dslash_kernel<EPI, DUAL>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             FX_THREADS / 32 * kWarpBytes);
        raised.fetch_or(bit, std::memory_order_relaxed);
    }
    const size_t smem = (size_t)(block.x * block.y / 32) * kWarpBytes;
    fx_dslash_kernel<EPI, DUAL><<<grid, block, smem, s>>>(a, nrhs);
}
}  // namespace

void launch_fx_survey(const Geom& g, const void* U64, void* out, cudaStream_t s) {
    unsigned long long* o = (unsigned long long*)out;
    cudaMemsetAsync(o, 0, 8, s);
    cudaMemsetAsync(o + 1, 0x7f, 16, s);  // 1e306, above every norm that counts
    fx_link_norm_k<<<(int)std::min<i64>((4LL * g.V + 255) / 256, 152 * 8), 256, 0, s>>>((const double2*)U64, g.V, o);
    fx_survey_k<<<std::min((g.V + 127) / 128, 152 * 8), 128, 0, s>>>((const double2*)U64, g, o);
    count_launch(2);
}

void launch_fx_links(const Geom& g, double m0, double scale2, const void* U64, void* dst, cudaStream_t s) {
    fx::Scale* sc = scale_of(dst, g.V);
    double hi, lo;
    root_hi_lo(scale2, &hi, &lo);
    const double d = 2.0 * (4.0 + m0), d_hi = d * hi, d_lo = std::fma(d, hi, -d_hi) + d * lo;
    cudaMemsetAsync(sc, 0, sizeof(fx::Scale), s);
    fx_link_norm_k<<<(int)std::min<i64>((4LL * g.V + 255) / 256, 152 * 8), 256, 0, s>>>((const double2*)U64, g.V,
                                                                                       &sc->norm_bits);
    fx_scale_k<<<1, 1, 0, s>>>(sc, hi, d_hi, d_lo);
    fx_pack_links_k<<<dim3((g.V + 127) / 128, 4), 128, 0, s>>>((const double2*)U64, (char*)dst, g.V, hi, lo, sc);
    count_launch(3);
}

void launch_fx_xlinks(const Geom& g, double scale2, const void* U64, const void* links, void* dst,
                      const double* d_phases, int nphase, cudaStream_t s) {
    double hi, lo;
    root_hi_lo(scale2, &hi, &lo);
    fx_xlinks_k<<<dim3((g.V + 127) / 128, nphase), 128, 0, s>>>((const double2*)U64, (char*)dst, g.V,
                                                               g.L[0] * g.L[1] * g.L[2], d_phases, hi, lo,
                                                               scale_of(links, g.V));
    count_launch();
}

void launch_fx_from_f64(const void* in, void* out, int V, int nrhs, double factor, cudaStream_t s) {
    fx_from_f64_k<<<dim3((V + 127) / 128, nrhs), 128, 0, s>>>((const double2*)in, (char*)out, V, factor);
    count_launch();
}

void launch_fx_to_f64(const void* in, void* out, int V, int nrhs, double factor, cudaStream_t s) {
    fx_to_f64_k<<<dim3((V + 127) / 128, nrhs), 128, 0, s>>>((const char*)in, (double2*)out, V, factor);
    count_launch();
}

namespace {
bool fx_split(int V, int nrhs) { return (i64)((V + 15) / 16) * nrhs <= kSplitBlocks; }
int fx_threads(int V, int nrhs) {
    int threads = FX_THREADS;
    while (threads > 32 && 2LL * V * nrhs < 152LL * 2 * threads) threads /= 2;
    return threads;
}
}  // namespace

int fx_block_rhs(int V, int nrhs) { return fx_split(V, nrhs) ? 1 : fx_threads(V, nrhs) / 32; }

void launch_fx_dslash(const Geom& g, const FxLinks& U, const void* in, void* out, void* out_deriv, int nrhs,
                      const FxEpilogue& e, cudaStream_t s, int shape) {
    fx::Args a;
    a.U = (const char*)U.links;
    a.Ux = (const char*)U.xlinks;
    a.xidx = U.xidx;
    a.scale = scale_of(U.links, g.V);
    a.in = (const char*)in;
    a.out = (char*)out;
    a.out2 = (char*)out_deriv;
    a.v1 = (const char*)e.v1;
    a.v2 = (const char*)e.v2;
    a.v3 = (const char*)e.v3;
    a.c0e = e.half ? -1 : 0;
    a.c1 = make_coef(e.c1);
    a.c2 = make_coef(e.c2);
    a.c3 = make_coef(e.c3);
    int st = 1;
    for (int mu = 0; mu < 4; ++mu) {
        a.L[mu] = g.L[mu];
        a.stride[mu] = st;
        a.dirichlet[mu] = g.bcf[mu] == 0.0;
        st *= g.L[mu];
    }
    for (int k = 0; k < 3; ++k) a.div[k] = fx::make_div((uint32_t)g.L[k]);
    a.V = g.V;
    const bool epi = e.v1 || e.v2 || e.v3 || e.half;
    if (fx_split(g.V, nrhs)) {
        const dim3 grid((g.V + 15) / 16, nrhs);
        if (out_deriv) {
            if (epi) fx_split_kernel<true, true><<<grid, 128, 0, s>>>(a);
            else fx_split_kernel<false, true><<<grid, 128, 0, s>>>(a);
        } else {
            if (epi) fx_split_kernel<true, false><<<grid, 128, 0, s>>>(a);
            else fx_split_kernel<false, false><<<grid, 128, 0, s>>>(a);
        }
        count_launch();
        return;
    }
    const int threads = fx_threads(g.V, nrhs);
    int by = (shape & kShapeRhsMask) > 0 ? (shape & kShapeRhsMask) : 4;
    by = std::min(by, fx_block_rhs(g.V, nrhs));
    while (by > 1 && by > nrhs) by >>= 1;
    const int bx = threads / by, sites = bx / 2;
    const dim3 block(bx, by), grid((g.V + sites - 1) / sites, (nrhs + by - 1) / by);
    if (out_deriv) {
        if (epi) fx_launch<true, true>(a, grid, block, nrhs, s);
        else fx_launch<false, true>(a, grid, block, nrhs, s);
    } else {
        if (epi) fx_launch<true, false>(a, grid, block, nrhs, s);
        else fx_launch<false, false>(a, grid, block, nrhs, s);
    }
    count_launch();
}

}  // namespace ovl
