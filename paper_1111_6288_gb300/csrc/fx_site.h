// Half a site of the fixed-point Wilson operator (fx_arith.h): g H_w, H_w = gamma5 D_w of Sec. 2 on
// site-scaled integers, with the epilogue of the recurrences.  Host and device code.
//
// A hop (1 -+ gamma_mu) U psi acts on two half-spinor rows h_0, h_1 that never mix: row f takes spin f
// of the neighbour and spin 2 + f (z and t) or 3 - f (x and y), and its product goes back to the same
// two spins.  Two lanes share a site, lane f doing row f of all eight hops; at the end lane f owns
// spins f and 2 + f, and the sums of the other lane's lower spin are exchanged.  Half a site per lane
// needs half the accumulators, so twice the warps are resident, and a lattice of few sites spreads
// over twice the lanes.
//
// Layout: tiles of 32 consecutive sites, so that everything a lane reads of one site lies at constant
// offsets from one address.  Vector, one right-hand side (rhs_bytes(V) bytes): per tile [12][32] int4,
// component k = 3 spin + colour as (re.hi, re.lo, im.hi, im.lo), then [32] int exponents.  Links: [4]
// directions of per tile [9][32] int4, entry 3 a + b of g U_mu(n) 2^-le, the antiperiodic boundary
// signs folded in; g is the scale that turns alpha H_w^2 of a recurrence into (g H_w)^2, so that a step
// multiplies its operator by nothing.
#pragma once

#include <vector_types.h>

#include "fx_arith.h"

namespace ovl {
namespace fx {

constexpr int kTile = 32;
constexpr int kTileBytes = (12 * 16 + 4) * kTile;   // of a vector
constexpr int kLinkTileBytes = 9 * 16 * kTile;
FX_FN i64 tiles(i64 V) { return (V + kTile - 1) / kTile; }
FX_FN i64 rhs_bytes(i64 V) { return tiles(V) * kTileBytes; }
FX_FN i64 link_bytes(i64 V) { return tiles(V) * kLinkTileBytes; }  // one direction
// component 0 of site s of a vector; component k follows k * kTile int4 later
FX_FN const int4* at(const char* v, int s) {
    return (const int4*)(v + (i64)(s >> 5) * kTileBytes) + (s & 31);
}
FX_FN int4* at(char* v, int s) { return (int4*)(v + (i64)(s >> 5) * kTileBytes) + (s & 31); }
FX_FN const int* exponent_at(const char* v, int s) {
    return (const int*)(v + (i64)(s >> 5) * kTileBytes + 12 * 16 * kTile) + (s & 31);
}
FX_FN int* exponent_at(char* v, int s) { return (int*)(v + (i64)(s >> 5) * kTileBytes + 12 * 16 * kTile) + (s & 31); }
// entry 0 of the link at site s of one direction
FX_FN const int4* link_at(const char* u, int s) {
    return (const int4*)(u + (i64)(s >> 5) * kLinkTileBytes) + (s & 31);
}
FX_FN int4* link_at(char* u, int s) { return (int4*)(u + (i64)(s >> 5) * kLinkTileBytes) + (s & 31); }

// n / d for 0 <= n < 2^31 by a multiplication.
struct Div {
    uint32_t mul, shift;
};
inline Div make_div(uint32_t d) {
    Div o{0, 0};
    while ((1ull << o.shift) < d) ++o.shift;
    o.mul = (uint32_t)(((1ull << 32) * ((1ull << o.shift) - d)) / d + 1);
    return o;
}
FX_FN int quotient(int n, Div d) {
#ifdef __CUDA_ARCH__
    return (int)((__umulhi((uint32_t)n, d.mul) + (uint32_t)n) >> d.shift);
#else
    return (int)(((uint32_t)(((uint64_t)(uint32_t)n * d.mul) >> 32) + (uint32_t)n) >> d.shift);
#endif
}

// What goes with a set of links, kept in device memory beside them.
struct Scale {
    unsigned long long norm_bits;  // largest squared row or column norm of the links, as a double's bits
    int le;
    Coef diag;                     // 2 (4 + m0) g
};

struct Args {
    const char* U;
    const char* Ux;          // per phase, one direction of x links times exp(i phase t)
    const int* xidx;         // device [nrhs]: phase of each system's x links (-1: U's), or null
    const Scale* scale;
    const char* in;
    char* out;
    char* out2;              // DUAL: g times the phi-derivative of H_w applied to in
    const char* v1;
    const char* v2;
    const char* v3;
    int c0e;                 // out = 2^c0e g H_w in + c1 v1 + c2 v2 + c3 v3
    Coef c1, c2, c3;
    int L[4];
    int stride[4];
    int dirichlet[4];
    Div div[3];              // by L[0], L[1], L[2]
    int V;
};

FX_FN Cplx as_cplx(int4 v) { return {{v.x, v.y}, {v.z, v.w}}; }
FX_FN int4 ld(const int4* p) {
#ifdef __CUDA_ARCH__
    return __ldg(p);
#else
    return *p;
#endif
}
FX_FN int ld(const int* p) {
#ifdef __CUDA_ARCH__
    return __ldg(p);
#else
    return *p;
#endif
}

// 2x2 block G of gamma_mu = [[0, G], [G^+, 0]]: diagonal (z, t) or anti-diagonal (x, y); row 0's entry
// is i^A, row 1's is i^A or, where FLIP, -i^A.
template <int MU> struct Gam;
template <> struct Gam<0> { static constexpr bool diag = false, flip = false; static constexpr int A = 3; };
template <> struct Gam<1> { static constexpr bool diag = false, flip = true; static constexpr int A = 2; };
template <> struct Gam<2> { static constexpr bool diag = true, flip = true; static constexpr int A = 3; };
template <> struct Gam<3> { static constexpr bool diag = true, flip = false; static constexpr int A = 0; };

// a + b or, where m = -1 (all ones; k = 1), a - b: one logic operation and one three-input addition
FX_FN Num add_sign(Num a, Num b, int m, int k) { return {a.hi + (b.hi ^ m) + k, a.lo + (b.lo ^ m) + k}; }
// a + i^CODE b, or a - i^CODE b where flip = 1
template <int CODE>
FX_FN Cplx add_unit_flip(Cplx a, Cplx b, int flip) {
    constexpr int c = ((CODE % 4) + 4) % 4;
    const int m = -flip, n = flip - 1, k = 1 - flip;  // n, k: the opposite sign
    if constexpr (c == 0) return {add_sign(a.re, b.re, m, flip), add_sign(a.im, b.im, m, flip)};
    else if constexpr (c == 1) return {add_sign(a.re, b.im, n, k), add_sign(a.im, b.re, m, flip)};
    else if constexpr (c == 2) return {add_sign(a.re, b.re, n, k), add_sign(a.im, b.im, n, k)};
    else return {add_sign(a.re, b.im, m, flip), add_sign(a.im, b.re, n, k)};
}

// (re, im) += i^CODE (wr, wi)
template <int CODE>
FX_FN void add_rot(i64& re, i64& im, i64 wr, i64 wi) {
    constexpr int c = ((CODE % 4) + 4) % 4;
    if constexpr (c == 0) { re += wr; im += wi; }
    else if constexpr (c == 1) { re -= wi; im += wr; }
    else if constexpr (c == 2) { re -= wr; im -= wi; }
    else { re += wi; im -= wr; }
}

// First component of the lower spin that row f of a hop in direction mu reads.
FX_FN int partner(int mu, int f) { return mu >= 2 ? 6 + 3 * f : 9 - 3 * f; }

// Row f of one hop in direction MU: up (spin f) += w, lo += i^code w with the code of row 0 (for row 1
// the caller negates lo where the block flips).  forward: (1 - gamma) U(n) psi(n + mu), backward:
// (1 + gamma) U(n - mu)^+ psi(n - mu).  pa, pb: the neighbour's spin f and its partner (components SP
// apart), u: the link's entries (SU apart), e: the exponent of the products (kZeroExp leaves nothing of
// them, whatever is loaded); sums in units of 2^eref.
template <int MU, bool FWD, int SP, int SU>
FX_FN void hop(int f, const int4* pa, const int4* pb, const int4* u, int e, int eref, i64 (&up)[6], i64 (&lo)[6]) {
    using G = Gam<MU>;
    constexpr int S = FWD ? 2 : 0;
    // (zr +- i zi)(hr + i hi) in three products instead of four:
    //   hr (zr +- zi) -+ zi (hr + hi)  and  hr (zr +- zi) + zr (hi - hr)
    // The limbs of the sums are not carried (|hi| <= 2^30, |lo| <= 2^29) and nothing is dropped but lo lo', whose
    // sum is the same either way: the bits are those of four products, with 81 multiply-adds a hop instead of
    // 108 (and 24 more additions): 51.5 -> 48.5 us a launch at 16^3 x 32, 258 -> 239 us at 24^3 x 48.
    Num r[3], p[3], q[3];  // hr, -+(hr + hi), hi - hr
    FX_UNROLL
    for (int c = 0; c < 3; ++c) {
        const Cplx a = as_cplx(pa[c * SP]), b = as_cplx(pb[c * SP]);
        Cplx h;
        if constexpr (G::flip) h = add_unit_flip<G::A + S>(a, b, f);
        else h = add_unit<G::A + S>(a, b);
        r[c] = h.re;
        p[c] = FWD ? neg(add(h.re, h.im)) : add(h.re, h.im);
        q[c] = sub(h.im, h.re);
    }
    const int d = align_shift(eref, e);
    const i64 rnd = half_of(d);
    FX_UNROLL
    for (int i = 0; i < 3; ++i) {
        Cplx z[3];
        Sum re = start(rnd);
        FX_UNROLL
        for (int j = 0; j < 3; ++j) {
            z[j] = as_cplx(u[(FWD ? 3 * i + j : 3 * j + i) * SU]);
            mac(re, FWD ? add(z[j].re, z[j].im) : sub(z[j].re, z[j].im), r[j]);
        }
        Sum im = re;
        FX_UNROLL
        for (int j = 0; j < 3; ++j) {
            mac(re, z[j].im, p[j]);
            mac(im, z[j].re, q[j]);
        }
        const i64 wr = value(re) >> d, wi = value(im) >> d;
        up[2 * i] += wr;
        up[2 * i + 1] += wi;
        add_rot<4 - G::A + S>(lo[2 * i], lo[2 * i + 1], wr, wi);
    }
}

// Largest bits of a lane's 12 numbers (0 and -1 have none).
FX_FN uint64_t or_bits(const i64 (&a)[6], const i64 (&b)[6]) {
    uint64_t o = 0;
    FX_UNROLL
    for (int k = 0; k < 6; ++k) o |= (uint64_t)(a[k] ^ (a[k] >> 63)) | (uint64_t)(b[k] ^ (b[k] >> 63));
    return o;
}

// Bring the numbers (units of 2^e) to |m| <= 2^56, o the or_bits of the whole site; returns the new
// exponent (kZeroExp where nothing is left).
FX_FN int normalise(i64 (&a)[6], i64 (&b)[6], uint64_t o, int e) {
    const int sh = bit_length(o) - kBits;
    if (o == 0) {
        FX_UNROLL
        for (int k = 0; k < 6; ++k) a[k] = b[k] = 0;
        return kZeroExp;
    }
    if (sh > 0) {
        const i64 half = half_of(sh);
        FX_UNROLL
        for (int k = 0; k < 6; ++k) {
            a[k] = shifted(a[k], sh, half);
            b[k] = shifted(b[k], sh, half);
        }
    } else if (sh < 0) {
        FX_UNROLL
        for (int k = 0; k < 6; ++k) {
            a[k] = (i64)((uint64_t)a[k] << -sh);
            b[k] = (i64)((uint64_t)b[k] << -sh);
        }
    }
    return e + sh;
}

// The same for three of a site's numbers (0 and -1 are nothing here too).
FX_FN int normalise(i64 (&a)[3], uint64_t o, int e) {
    const int sh = o == 0 ? 1 : bit_length(o) - kBits;  // a shift by one bit makes 0 of both
    FX_UNROLL
    for (int k = 0; k < 3; ++k) a[k] = sh > 0 ? shifted(a[k], sh, half_of(sh)) : (i64)((uint64_t)a[k] << -sh);
    return o == 0 ? kZeroExp : e + sh;
}

// Three components from `spin` of the site whose component 0 is at b.
FX_FN void store_spin(int4* b, int spin, const i64 (&a)[6]) {
    FX_UNROLL
    for (int c = 0; c < 3; ++c) {
        const Num re = split(a[2 * c]), im = split(a[2 * c + 1]);
        int4 v;
        v.x = re.hi;
        v.y = re.lo;
        v.z = im.hi;
        v.w = im.lo;
        b[(3 * spin + c) * kTile] = v;
    }
}

// Exponent of coefficient x number of exponent e, and the smallest unit it is kept in.
FX_FN int term_exp(int e, const Coef& c) { return c.unit ? e - 2 : e + c.e; }

// a += c v in units of 2^E (v: three components, exponent e).
FX_FN void add_term(i64 (&a)[6], const int4 (&v)[3], int e, const Coef& c, int E) {
    const int d = align_shift(E, term_exp(e, c));
    const i64 half = half_of(d);
    FX_UNROLL
    for (int k = 0; k < 3; ++k) {
        const Cplx z = as_cplx(v[k]);
        if (c.unit) {
            const i64 r = ((i64)z.re.hi << (kLimb + 2)) + ((i64)z.re.lo << 2);
            const i64 i = ((i64)z.im.hi << (kLimb + 2)) + ((i64)z.im.lo << 2);
            a[2 * k] += shifted(c.unit > 0 ? r : -r, d, half);
            a[2 * k + 1] += shifted(c.unit > 0 ? i : -i, d, half);
        } else {
            Sum r = start(half), i = start(half);
            mac(r, c.m, z.re);
            mac(i, c.m, z.im);
            a[2 * k] += value(r) >> d;
            a[2 * k + 1] += value(i) >> d;
        }
    }
}

// The same for three numbers v of one exponent.
FX_FN void add_term(i64 (&a)[3], const int2 (&v)[3], int e, const Coef& c, int E) {
    const int d = align_shift(E, term_exp(e, c));
    const i64 half = half_of(d);
    FX_UNROLL
    for (int k = 0; k < 3; ++k) {
        if (c.unit) {
            const i64 r = ((i64)v[k].x << (kLimb + 2)) + ((i64)v[k].y << 2);
            a[k] += shifted(c.unit > 0 ? r : -r, d, half);
        } else {
            Sum s = start(half);
            mac(s, c.m, Num{v[k].x, v[k].y});
            a[k] += value(s) >> d;
        }
    }
}

// One lane's half of a site.  Hops are taken in the order y, z, t, x, forward before backward:
// hop k goes in direction dir_of(k) to site nb[k].
struct Half {
    int f, x3, e0, eref;  // eref above kNanTest: the site or a neighbour holds a NaN
    bool bad_x;           // an x neighbour does (the derivative has no other hops)
    int nb[8], ex[8];
    i64 up[6], own[6], oth[6];  // spin f, spin 2 + f, the other lane's lower spin
};
FX_FN constexpr int dir_of(int k) { return (k / 2 + 1) & 3; }

FX_FN void half_setup(const Args& a, int s, int r, int f, Half& H) {
    const char* in = a.in + (i64)r * rhs_bytes(a.V);
    const int le = ld(&a.scale->le);
    H.f = f;
    int x[4];
    const int q0 = quotient(s, a.div[0]), q1 = quotient(q0, a.div[1]);
    x[0] = s - q0 * a.L[0];
    x[1] = q0 - q1 * a.L[1];
    x[3] = quotient(q1, a.div[2]);
    x[2] = q1 - x[3] * a.L[2];
    H.x3 = x[3];
    H.e0 = ld(exponent_at(in, s));
    int eref = H.e0 + ld(&a.scale->diag.e);
    FX_UNROLL
    for (int k = 0; k < 8; k += 2) {
        const int mu = dir_of(k), st = a.stride[mu], w = (a.L[mu] - 1) * st;
        const bool top = x[mu] == a.L[mu] - 1, bottom = x[mu] == 0;
        H.nb[k] = top ? s - w : s + st;
        H.nb[k + 1] = bottom ? s + w : s - st;
        const int ef = ld(exponent_at(in, H.nb[k])), eb = ld(exponent_at(in, H.nb[k + 1]));
        H.ex[k] = (top && a.dirichlet[mu] ? kZeroExp : ef) + le;
        H.ex[k + 1] = (bottom && a.dirichlet[mu] ? kZeroExp : eb) + le;
        eref = H.ex[k] > eref ? H.ex[k] : eref;
        eref = H.ex[k + 1] > eref ? H.ex[k + 1] : eref;
    }
    H.eref = eref;
    H.bad_x = H.ex[6] > kNanTest || H.ex[7] > kNanTest;
    FX_UNROLL
    for (int k = 0; k < 6; ++k) H.up[k] = H.own[k] = H.oth[k] = 0;
}

// The x links of right-hand side r, and those of direction mu.
FX_FN const char* links_of_dir(const Args& a, int r, int mu) {
    const i64 lb = link_bytes(a.V);
    if (mu == 0 && a.xidx) {
        const int xi = a.xidx[r];
        if (xi >= 0) return a.Ux + (i64)xi * lb;
    }
    return a.U + mu * lb;
}

// Hop K with its operands at pa, pb and u.  The y hops go into oth and the z hops into own while these
// hold nothing else: row 1's entries of the two blocks carry a minus sign, applied once behind them.
// DUAL: the x hops go into (fu, fl) and (bu, bl), in units of 2^(the larger of their exponents), so that
// the derivative keeps its precision where the other neighbours are larger.
template <int K, bool DUAL, int SP, int SU>
FX_FN void half_hop(Half& H, const int4* pa, const int4* pb, const int4* u, i64 (&fu)[6], i64 (&fl)[6], i64 (&bu)[6],
                    i64 (&bl)[6]) {
    constexpr int MU = dir_of(K);
    constexpr bool FWD = K % 2 == 0;
    if constexpr (MU == 0 && DUAL) {
        const int xref = H.ex[6] > H.ex[7] ? H.ex[6] : H.ex[7];
        if constexpr (FWD) hop<MU, FWD, SP, SU>(H.f, pa, pb, u, H.ex[K], xref, fu, fl);
        else hop<MU, FWD, SP, SU>(H.f, pa, pb, u, H.ex[K], xref, bu, bl);
    } else if constexpr (MU < 2) {
        hop<MU, FWD, SP, SU>(H.f, pa, pb, u, H.ex[K], H.eref, H.up, H.oth);
    } else {
        hop<MU, FWD, SP, SU>(H.f, pa, pb, u, H.ex[K], H.eref, H.up, H.own);
    }
    if constexpr (K == 3) {
        const i64 m = -(i64)H.f;  // 0 or all ones
        FX_UNROLL
        for (int k = 0; k < 6; ++k) {
            H.oth[k] = (H.oth[k] ^ m) - m;
            H.own[k] = (H.own[k] ^ m) - m;
        }
    }
}

// The x hops of DUAL: F + B into the sums, F - B (spins f and 3 - f) left in fu, fl; returns its exponent.
FX_FN int dual_split(Half& H, i64 (&fu)[6], i64 (&fl)[6], const i64 (&bu)[6], const i64 (&bl)[6]) {
    const int xref = H.ex[6] > H.ex[7] ? H.ex[6] : H.ex[7];
    const int d = align_shift(H.eref, xref);
    const i64 half = half_of(d);
    FX_UNROLL
    for (int k = 0; k < 6; ++k) {
        H.up[k] += shifted(fu[k] + bu[k], d, half);
        H.oth[k] += shifted(fl[k] + bl[k], d, half);
        fu[k] -= bu[k];
        fl[k] -= bl[k];
    }
    return xref;
}

// gamma5 (-1/2) (i t) (F - B) of the x hops, o the or_bits of dup and doth over the site.  First the
// numbers become t (re, im) -> t (im, -re) on the upper spins, in units of 2^e; then, o again, stored.
FX_FN int deriv_scale(const Half& H, i64 (&dup)[6], i64 (&doth)[6], uint64_t o, int e) {
    e = normalise(dup, doth, o, e);
    const int tb = bit_length((uint64_t)H.x3);
    const Num tm{H.x3 << (kLimb - tb), 0};  // x3 2^-tb in units of 2^-56, below 1
    FX_UNROLL
    for (int c = 0; c < 3; ++c) {
        Sum ur = start(0), ui = start(0), lr = start(0), li = start(0);
        mac(ur, tm, split(dup[2 * c]));
        mac(ui, tm, split(dup[2 * c + 1]));
        mac(lr, tm, split(doth[2 * c]));
        mac(li, tm, split(doth[2 * c + 1]));
        dup[2 * c] = value(ui);
        dup[2 * c + 1] = -value(ur);
        doth[2 * c] = -value(li);
        doth[2 * c + 1] = value(lr);
    }
    return e + tb - 1;
}

// After the exchange (own holds the whole lower spin): up, own <- +-(2 (4 + m0) g psi - sum), twice
// g H_w in, units 2^eref.  psi: the lane's six components.
FX_FN void mass_term(const Args& a, Half& H, const int4 (&pu)[3], const int4 (&pl)[3]) {
    const Coef D = a.scale->diag;
    const int d = align_shift(H.eref, H.e0 + D.e);
    const i64 half = half_of(d);
    FX_UNROLL
    for (int c = 0; c < 3; ++c) {
        const Cplx u = as_cplx(pu[c]), l = as_cplx(pl[c]);
        Sum ur = start(half), ui = start(half), lr = start(half), li = start(half);
        mac(ur, D.m, u.re);
        mac(ui, D.m, u.im);
        mac(lr, D.m, l.re);
        mac(li, D.m, l.im);
        H.up[2 * c] = (value(ur) >> d) - H.up[2 * c];
        H.up[2 * c + 1] = (value(ui) >> d) - H.up[2 * c + 1];
        H.own[2 * c] -= value(lr) >> d;
        H.own[2 * c + 1] -= value(li) >> d;
    }
}

}  // namespace fx
}  // namespace ovl
