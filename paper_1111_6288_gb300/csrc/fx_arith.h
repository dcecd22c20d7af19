// Site-scaled fixed-point numbers: 64-bit-grade arithmetic on the integer pipes.
//
// A real number of a spinor is m 2^e with one exponent e per site and an integer m held as two
// signed limbs, m = hi 2^28 + lo (|lo| <= 2^27).  The largest |m| of a site lies in [2^55, 2^56], so a
// vector is kept to 2^-56 of its site's largest number where FP64 keeps each number to 2^-53 of
// itself.  Links are integers of the same form in units of 2^-56.  A product keeps the limb products
//   hi hi' + (hi lo' + lo hi') 2^-28                      (in units of 2^-56 of the unit product)
// and drops lo lo' 2^-56, at most 1/4 unit.  Every limb product is one 32 x 32 + 64-bit multiply-add.
//
// Why: on this GPU one SM does 2 FP64 multiply-adds per clock (3.9 per ns measured) and 64 of these
// integer ones (120 per ns), so three of them replace one FP64 multiply-add at a tenth of its cost.
//
// The same source compiles for the host, where the tests of the arithmetic run.
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define FX_FN __host__ __device__ __forceinline__
#define FX_UNROLL _Pragma("unroll")
#else
#define FX_FN inline
#define FX_UNROLL
#endif

namespace ovl {
namespace fx {

typedef long long i64;

constexpr int kBits = 56;             // |m| <= 2^56
constexpr int kLimb = 28;             // bits of the low limb
constexpr int kZeroExp = -(1 << 24);  // exponent of a site of zeros
constexpr int kNanExp = 1 << 24;      // exponent of a site holding a NaN or an infinity
constexpr int kNanTest = 1 << 23;     // exponents above this mark such a site

struct Num {
    int hi, lo;
};
struct Cplx {
    Num re, im;
};

FX_FN Num add(Num a, Num b) { return {a.hi + b.hi, a.lo + b.lo}; }
FX_FN Num sub(Num a, Num b) { return {a.hi - b.hi, a.lo - b.lo}; }
FX_FN Num neg(Num a) { return {-a.hi, -a.lo}; }

// m -> limbs, |m| <= 2^56 (up to 2^58 for numbers that are only multiplied by a coefficient).
FX_FN Num split(i64 m) {
    const int lo = (int)((uint32_t)m << (32 - kLimb)) >> (32 - kLimb);
    const int hi = (int)((m + (1LL << (kLimb - 1))) >> kLimb);
    return {hi, lo};
}

// a + i^CODE b for complex numbers (CODE = 0..3: 1, i, -1, -i).
template <int CODE>
FX_FN Cplx add_unit(Cplx a, Cplx b) {
    constexpr int c = ((CODE % 4) + 4) % 4;
    if constexpr (c == 0) return {add(a.re, b.re), add(a.im, b.im)};
    else if constexpr (c == 1) return {sub(a.re, b.im), add(a.im, b.re)};
    else if constexpr (c == 2) return {sub(a.re, b.re), sub(a.im, b.im)};
    else return {add(a.re, b.im), sub(a.im, b.re)};
}

// Sum of products as (sum of hi hi', sum of the crossed limb products).
struct Sum {
    i64 h, c;
};
FX_FN void mac(Sum& s, Num a, Num b) {
    s.h += (i64)a.hi * b.hi;
    s.c += (i64)a.hi * b.lo;
    s.c += (i64)a.lo * b.hi;
}
// An empty sum, to be read by value() and shifted right: `round` is that shift's rounding constant, and the
// crossed part has its own.
FX_FN Sum start(i64 round) { return {round, 1LL << (kLimb - 1)}; }
FX_FN i64 value(Sum s) { return s.h + (s.c >> kLimb); }

// Rounding constant of a right shift by d (0 <= d <= 63).
FX_FN i64 half_of(int d) { return (i64)((1ULL << d) >> 1); }

// v 2^-d to the nearest integer (halves up).
FX_FN i64 shifted(i64 v, int d, i64 half) { return (v + half) >> d; }

FX_FN int align_shift(int eref, int e) {
    const int d = eref - e;
    return d < 63 ? d : 63;
}

// Number of bits of |v| (0 for 0) from the or of v ^ (v >> 63) over a set.
FX_FN int bit_length(uint64_t v) {
#ifdef __CUDA_ARCH__
    return 64 - __clzll((long long)v);
#else
    return v ? 64 - __builtin_clzll(v) : 0;
#endif
}

// A real coefficient: value (hi 2^28 + lo) 2^(e - 56), |hi 2^28 + lo| < 2^59.  unit: +1 or -1 where
// the coefficient is exactly that (no multiplication), else 0.  Finite coefficients only.
struct Coef {
    Num m;
    int e;
    int unit;
};

}  // namespace fx
}  // namespace ovl
