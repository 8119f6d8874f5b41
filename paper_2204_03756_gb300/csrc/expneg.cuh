// expneg.cuh -- the binary64 pair terms of Eq. 4 in 64-bit integer arithmetic:
// K = exp(-a d2) with a = 1 / (2 h^2), the row sum of K, the weight
// 2 K / (r_i + r_j) and the sum of the fluxes.
//
// GB300's binary64 unit takes a warp instruction per 16 to 20 clocks an SM, in
// which the SM issues 64 others, so a 64 x 64-bit product from 32-bit
// multiply-adds (about ten instructions) costs a sixth of a binary64
// operation, and carries more digits.
//
// Positions come as fixed-point images X = round(x 2^S) mod 2^64 (x_image),
// with S such that the cutoff psi is in (2^61, 2^62]: the difference of two
// neighbours' images, as int64, is their distance along the axis to 2^-61 psi,
// wherever the box lies (the upper bits, equal up to a borrow, drop out).
//
// The exponential follows P. T. P. Tang, "Table-driven implementation of the
// exponential function in IEEE floating-point arithmetic", ACM TOMS 15(2),
// 1989, in fixed point but for its last multiplication:
//   T = a d2 256 log2(e) = k + f, k an integer, 0 <= f < 1,
//   exp(-a d2) = 2^-(k >> 8) * 2^(-(k & 255) / 256) * exp(-c f), c = ln 2 / 256,
// exp(-c f) its Taylor series through (c f)^5 (the first omitted term is below
// 2^-60).  That multiplication by the table's 2^(-j / 256) is a binary64 one:
// it rounds and normalises K, which took 29 integer instructions, and the
// binary64 unit has the time (one operation a pair).  The error of K is three
// roundings (2^-53 each) and T's; with binary64 operations throughout it was 14
// such units at lambda = 3, from the rounding of d2.  Valid for a d2 <= 400.1
// (lambda <= 20 with the band margin); the host bounds lambda.
#pragma once
#include <cmath>
#include <cstdint>

#if defined(__CUDACC__)
#define MTPT_HD __host__ __device__ __forceinline__
#else
#define MTPT_HD inline
#endif

namespace mtpt {

constexpr int kExpTable = 256;

// Constants of one realisation's kernel (kernel_consts).
struct KernelConsts {
    int x_shift;        // S
    int f_bits;         // fraction bits of T, in [33, 60]
    uint64_t a_fix;     // T = high 64 bits of d2h a_fix, d2h = d2 2^(2 S - 64)
};

// Leading zeros of v != 0.
MTPT_HD int clz64(uint64_t v) {
#if defined(__CUDA_ARCH__)
    return __clzll((long long)v);
#else
    return __builtin_clzll(v);
#endif
}
MTPT_HD uint64_t bits_of(double x) {
#if defined(__CUDA_ARCH__)
    return uint64_t(__double_as_longlong(x));
#else
    uint64_t b;
    __builtin_memcpy(&b, &x, 8);
    return b;
#endif
}
MTPT_HD double double_of(uint64_t b) {
#if defined(__CUDA_ARCH__)
    return __longlong_as_double((long long)b);
#else
    double x;
    __builtin_memcpy(&x, &b, 8);
    return x;
#endif
}

// 32 x 32 -> 64-bit product, and the high 64 bits of 64 x 64 without the low
// words' product (at most 3 below the exact ones).
MTPT_HD uint64_t mul_wide(uint32_t a, uint32_t b) { return uint64_t(a) * b; }
MTPT_HD uint64_t mul_hi(uint64_t a, uint64_t b) {
    const uint32_t ah = uint32_t(a >> 32), al = uint32_t(a), bh = uint32_t(b >> 32), bl = uint32_t(b);
    return mul_wide(ah, bh) + (mul_wide(ah, bl) >> 32) + (mul_wide(al, bh) >> 32);
}
MTPT_HD uint64_t square_hi(uint64_t a) {
    const uint32_t ah = uint32_t(a >> 32), al = uint32_t(a);
    return mul_wide(ah, ah) + (mul_wide(ah, al) >> 31);
}
MTPT_HD uint32_t mul_hi32(uint32_t a, uint32_t b) { return uint32_t(mul_wide(a, b) >> 32); }

// The binary64 value w 2^(e - 63) of a 64-bit mantissa with its top bit set,
// rounded to nearest (a carry runs into the exponent field), for a normal
// result.
MTPT_HD double from_mantissa(uint64_t w, int e) {
    return double_of((uint64_t(e + 1022) << 52) + (w >> 11) + ((w >> 10) & 1u));
}

// v 2^e for a normal result, 0 for v = 0.
MTPT_HD double scaled(uint64_t v, int e) {
    const int z = clz64(v | 1u);
    return v == 0u ? 0.0 : from_mantissa(v << z, e + 63 - z);
}

// X = round(x 2^S) mod 2^64 (0 for subnormals, infinities and NaN, which no
// accepted pair has beyond its own zero).
MTPT_HD uint64_t x_image(double x, int shift) {
    const uint64_t b = bits_of(x);
    const int e = int(b >> 52) & 0x7ff;
    const int s = e - 1075 + shift;
    const uint64_t m = (b & 0xfffffffffffffull) | 0x10000000000000ull;
    uint64_t v;
    if (s >= 0) v = s < 64 ? m << s : 0u;
    else v = s > -55 ? (m + (1ull << (-s - 1))) >> -s : 0u;
    if (e == 0 || e == 0x7ff) v = 0u;
    return (b >> 63) ? 0u - v : v;
}

// |x_i - x_j| of one axis in units of 2^-S, and its square in units of
// 2^(64 - 2 S).
MTPT_HD uint64_t axis_distance(uint64_t xi, uint64_t xj) {
    const uint64_t d = xi - xj;
    return (d >> 63) ? 0u - d : d;
}
MTPT_HD uint64_t axis_square(uint64_t xi, uint64_t xj) { return square_hi(axis_distance(xi, xj)); }

// exp(-a d2) from d2h = d2 2^(2 S - 64).
MTPT_HD double gauss_fixed(uint64_t d2h, const double* __restrict__ table, const KernelConsts& c) {
    const uint64_t t = mul_hi(d2h, c.a_fix);
    const uint32_t k = uint32_t(t >> 32) >> (c.f_bits - 32);
    const uint64_t f = t << (64 - c.f_bits);
    const uint32_t fh = uint32_t(f >> 32);
    // exp(-c f) = 1 - f (c1 - f (c2 - f (c3 - f (c4 - f c5)))), c_m = c^m / m!;
    // c3..c5 in units of 2^-60, c1 and c2 of 2^-64
    uint32_t p = 0x276557u - mul_hi32(fh, 0x576u);
    p = 0xe35846b8u - mul_hi32(fh, p);
    const uint64_t p2 = 0x3d7f7bff058bull - (mul_wide(fh, p) >> 28);
    const uint64_t p1 = 0xb17217f7d1cf7aull - mul_hi(f, p2);
    // 1 - f p1 in (0.997, 1] as a binary64 value: below 1, 52 bits under the
    // leading one of 2^-1; at 1 the sum carries into the exponent
    const uint64_t below = mul_hi(f, p1) >> 11;
    const double e = double_of(0x3ff0000000000000ull - below);
    const double v = table[k & (kExpTable - 1)] * e;
    return double_of(bits_of(v) - (uint64_t(k >> 8) << 52));
}

// K <= 1 in units of 2^-62 (the row sums').
MTPT_HD uint64_t unit_of(double K) {
    const uint64_t b = bits_of(K);
    const uint32_t n = 1023u - uint32_t(b >> 52);
    return (((b & 0xfffffffffffffull) | 0x10000000000000ull) << 10) >> (n < 63u ? n : 63u);
}

// The weight 2 K / (ra + rb) for a positive normal K and 1 <= ra, rb < 2^60, as
// q 2^x, q in [2^59, 2^62): the quotient of the 64-bit mantissas from a
// binary32 reciprocal seed, one Newton-Raphson step in 32 bits and one
// residual correction of the quotient in 64 (relative error below 2^-54).
struct FixedWeight {
    uint64_t q;
    int x;
    MTPT_HD double value() const { return scaled(q, x); }
};
struct Reciprocal {
    uint32_t y;                  // 2^93 / d, d = (ra + rb) 2^(1085 - e) in [2^62, 2^64)
    int64_t e1;                  // 2^61 (1 - d y / 2^93)
    int e;
    MTPT_HD Reciprocal(double ra, double rb) {
        const uint64_t ab = bits_of(ra), bb = bits_of(rb);
        const uint64_t frac = 0xfffffffffffffull, one = 0x10000000000000ull;
        const int ea = int(ab >> 52), eb = int(bb >> 52);
        e = ea > eb ? ea : eb;
        const uint64_t d = ((((ab & frac) | one) << 10) >> (e - ea)) +
                           ((((bb & frac) | one) << 10) >> (e - eb));
        const uint32_t dh = uint32_t(d >> 32), dl = uint32_t(d);
#if defined(__CUDA_ARCH__)
        float s;
        asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(s) : "f"(__uint2float_rn(dh)));
        y = __float2uint_rz(s * 2305843009213693952.0f);                // 2^61; [2^29, 2^31]
#else
        y = uint32_t(2305843009213693952.0f / float(dh));
#endif
        const int64_t e0 = int64_t((1ull << 61) - mul_wide(dh, y));     // |e0| < 2^40
        y += uint32_t((int64_t(int32_t(e0 >> 19)) * int64_t(y)) >> 42);
        e1 = int64_t((1ull << 61) - mul_wide(dh, y) - (mul_wide(dl, y) >> 32));   // < 2^34
    }
    // m / (ra + rb) for m = mk 2^(ek - 1085), mk in [2^62, 2^63), as q 2^x
    MTPT_HD FixedWeight times(uint64_t mk, int ek) const {
        const uint64_t q0 = mul_wide(uint32_t(mk >> 32), y) + (mul_wide(uint32_t(mk), y) >> 32);
        return {q0 + uint64_t((int64_t(int32_t(e1 >> 3)) * int64_t(q0 >> 31)) >> 27), ek - e - 61};
    }
    // 2 K / (ra + rb) and 1 / (ra + rb)
    MTPT_HD FixedWeight weight(double K) const {
        const uint64_t kb = bits_of(K);
        return times(((kb & 0xfffffffffffffull) | 0x10000000000000ull) << 10, int(kb >> 52) + 1);
    }
    MTPT_HD FixedWeight inverse() const { return times(1ull << 62, 1023); }
};
MTPT_HD FixedWeight weight_fixed(double K, double ra, double rb) {
    return Reciprocal(ra, rb).weight(K);
}

// A sum of terms W dm over a particle's neighbours, dm a difference of masses, or of
// plain binary64 terms: 64-bit integers in units of 2^x, with x from the term of the
// largest exponent so far, raised when the sum grows past 61 bits.  A unit is at most
// 2^-54 of the largest term or 2^-57 of the largest partial sum so far, and every
// term and every change of unit costs less than one (a binary64 addition: 2^-53 of
// the partial sum).  Terms are cut toward zero.  TOWARD_ZERO cuts the sum so too at a
// change of unit, and it changes sign exactly when every dm does: what particles
// give and take is cut alike, and the total mass stays as with binary64 sums (cut
// downwards it drifted by 1e-19 of itself a step).  That takes 1.5 % of a run's time
// and 3 % of the adjoint sweep's, whose sums are cut downwards.  Terms that are not
// finite make the sum what binary64 additions would.
template <bool TOWARD_ZERO>
struct IntegerSum {
    int64_t acc = 0;
    int x = -100000;             // the sum is acc 2^x
    double special = 0.0;
    // W dm (or, without w, dm itself)
    MTPT_HD void add(double dm, const FixedWeight* w) {
        const uint64_t b = bits_of(dm);
        const int e = int(b >> 52) & 0x7ff;
        if (e == 0x7ff) {
            special += dm;
            return;
        }
        const uint64_t m = (b & 0xfffffffffffffull) | (e ? 0x10000000000000ull : 0u);
        // dm = m 2^(e - 1075), subnormals with e = 1; the term is g 2^y, g < 2^58
        uint64_t g = w ? mul_hi(m << 10, w->q) >> 3 : m << 5;
        const int y = (e ? e : 1) - 1075 + (w ? -10 + 64 + 3 + w->x : -5);
        const int up = y - x;
        if (up > 0) {
            cut(up < 63 ? up : 63);
            x = y;
        } else {
            g >>= up > -63 ? -up : 63;
        }
        acc += (b >> 63) ? -int64_t(g) : int64_t(g);
        if (uint64_t(acc + ((1ll << 61) - 1)) > (1ull << 62) - 2u) {    // |acc| >= 2^61
            cut(4);
            x += 4;
        }
    }
    // acc / 2^k, 0 < k < 64
    MTPT_HD void cut(int k) {
        if (TOWARD_ZERO) acc += int64_t(uint64_t(acc >> 63) >> (64 - k));
        acc >>= k;
    }
    MTPT_HD void add(double dm, const FixedWeight& w) { add(dm, &w); }
    MTPT_HD void add(double term) { add(term, nullptr); }
    MTPT_HD double value() const {
        if (!(special == 0.0)) return special;
        if (acc == 0) return 0.0;
        const uint64_t mag = acc < 0 ? 0u - uint64_t(acc) : uint64_t(acc);
        const int z = clz64(mag), e = 63 - z + x;
        const double v = (e > -1000 && e < 1000) ? from_mantissa(mag << z, e)
                                                 : scalbn(from_mantissa(mag << z, 0), e);
        return acc < 0 ? -v : v;
    }
};

using FluxSum64 = IntegerSum<true>;      // a particle's flux
using AdjSum64 = IntegerSum<false>;      // the adjoint's sums

// Row sum 1 + sum K in units of 2^-62, exact in 96 bits.
struct RowSum {
    uint64_t lo = 1ull << 62;
    uint32_t hi = 0;
    MTPT_HD void add(uint64_t unit) {
        lo += unit;
        hi += lo < unit ? 1u : 0u;
    }
    MTPT_HD double value() const {
        uint64_t w = lo;
        int top = 63;               // bit that w's top bit stands for
        if (hi) {
            const int z = clz64(hi) - 32;
            w = (uint64_t(hi) << (32 + z)) | (lo >> (32 - z));
            top = 95 - z;
        } else {
            const int z = clz64(lo);
            w <<= z;
            top -= z;
        }
        return from_mantissa(w, top - 62);
    }
};

// --- host: constants, in integers so that every machine gets the same ones ------

// The kernel's constants for a = 1 / (2 h^2) and cutoff psi.
inline KernelConsts kernel_consts(double a, double psi) {
    KernelConsts c{0, 60, 0};
    if (!(a > 0.0) || !(psi > 0.0)) return c;
    int e = 0;
    std::frexp(psi * (1.0 + 0x1p-20), &e);       // psi (1 + slack) < 2^e
    c.x_shift = 62 - e;
    // a 256 log2(e) 2^(f + 128 - 2 S), with the largest f <= 60 that keeps it
    // below 2^64; log2(e) in units of 2^-63
    int ea = 0;
    const uint64_t am = uint64_t(std::ldexp(std::frexp(a, &ea), 53));
    const unsigned __int128 prod = (unsigned __int128)am * 0xb8aa3b295c17f0bcull;
    const int top = (prod >> 116) ? 117 : 116;   // its bits
    const int drop = top - 64;
    const uint64_t fix = uint64_t(prod >> drop);
    // prod 2^(ea - 53 - 63 + 8 + f + 128 - 2 S) = fix 2^0
    c.f_bits = -drop - (ea - 53 - 63 + 8 + 128 - 2 * c.x_shift);
    c.a_fix = fix;
    if (c.f_bits > 60) {
        const int more = c.f_bits - 60;
        c.a_fix = more < 64 ? fix >> more : 0u;
        c.f_bits = 60;
    }
    return c;
}

// 2^(-j / 256), j in [0, 256), from 63-bit integers: products of the eight square
// roots 2^(-1/2), 2^(-1/4), ..., each the integer root of the one before.
inline void fill_exp_table(double* table) {
    uint64_t root[8];
    unsigned __int128 v = (unsigned __int128)1 << 127;   // 1/2 in units of 2^-128
    for (int k = 0; k < 8; ++k) {
        uint64_t r = 0;
        for (int b = 63; b >= 0; --b) {
            const uint64_t t = r | (1ull << b);
            if ((unsigned __int128)t * t <= v) r = t;
        }
        root[k] = r;                                     // 2^(-1 / 2^(k + 1)), 2^-64
        v = (unsigned __int128)r << 64;
    }
    for (int j = 0; j < kExpTable; ++j) {
        // the product of the roots of j's bits, with 127 fraction bits
        unsigned __int128 p = (unsigned __int128)1 << 127;
        for (int k = 0; k < 8; ++k) {
            if (!((j >> (7 - k)) & 1)) continue;
            const uint64_t ph = uint64_t(p >> 64), pl = uint64_t(p);
            p = (unsigned __int128)ph * root[k] + (((unsigned __int128)pl * root[k]) >> 64);
        }
        table[j] = std::ldexp(double(uint64_t((p + ((unsigned __int128)1 << 63)) >> 64)), -63);
    }
}

}  // namespace mtpt
