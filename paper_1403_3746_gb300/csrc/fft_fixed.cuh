// 64-bit fixed-point arithmetic for the float64 line transforms (Sec. 2.3 / Eq. (3)).
//
// GB300 issues 2 float64 operations per clock and SM, but 128 32-bit integer additions and 64
// 32-bit multiply-adds (measured: add.s64 64 per clock and SM, mul.wide.s32 60, fma.f64 2.0). A
// complex butterfly addition is four integer instructions instead of two float64 ones that take
// 32 times their slots, so the float64 lines are transformed as 64-bit integers that share one
// exponent per real line (block floating point).
//
// Scaling of a complex line of N = 2^LOG2N points, which is two real lines. Let 2^e bound the
// magnitude of a real line's numbers (from their exponents; each of the two has its own). Point x
// enters as trunc((x - c) 2^(B - e)). c is the line's mean, taken out where that leaves more bits:
// every multiplier is zero at index 0, so a constant never reaches the result. Every radix-16 pass
// that has outer twiddles ends (forward) or begins (inverse) with a factor 1/4, which the high half of
// the product with a root scaled to 2^62 gives for free. B is the largest value (line_bits) for
// which no sum can reach 2^63: a pass multiplies the largest
// modulus by at most the points it has summed, and no sum of points passes the sum of all moduli.
//
// The spectrum is shifted up before it meets the multiplier, as far as its largest entry with a
// non-zero multiplier allows, and the products again, until their summed magnitudes fill 2^63: the
// mean and the low indices, whose multipliers are small, would otherwise leave the rest few bits. (Up
// to 256 points the sum of the points themselves is enough, and cheaper.)
// Where the sum is larger than that without a shift, no sum overflows all the same: the products'
// 2-norm is at most N^(1/2) / 4^(T + 1) times the line's (T twiddled passes, the factor 1/4 of the
// product), and a sum of P of them at most sqrt(P) times that (Cauchy-Schwarz); line_bits keeps it
// below 2^63 through the inverse passes.
//
// Rounding: each product is rounded to the nearest integer up to a quarter unit, inputs are cut off
// once at 2^(e - B) (B = 54 .. 61). Root-mean-square error of a first derivative against __float128
// sums, relative to that of the float64 transform by the same radix-16 passes, 4 .. 4096 points: 0.3 to
// 0.8 for zero-mean noise, 0.0 to 0.5 for smooth and interface profiles and for noise about a mean, 0.3
// to 0.8 for single points, 0.1 to 1.05 for sharp two-level lines (the most at 4096 points); 1.4 for a
// 4096-point line of few-bit values constant but for one point, whose sums float64 holds exactly. Lines
// of 4 points, whose differences of close values float64 takes exactly: 0.4 to 1.
//
// Measured against the float64 transforms (1024^2): column pass 1225 -> 254 us per launch of 17
// fields, flux pass 330 -> 83; float64 step 8.31 -> 2.44 ms with the node loops and launch shapes.
// The passes wait for instructions and on latency, both integer pipes about half busy at 16 warps per
// SM. The two exponents, the mean, the sums and the two shifts are 3 to 6% of a step (1024^2 2.31 -> 2.44
// ms, 128 x 256 180 -> 191 us, 64^2 unchanged); without them the errors were 2 to 14 times float64's for
// sharp levels close to one another, up to 25 times for single points on a constant, from 512 points
// on, lines of 4 points constant to 10^-8 kept 9 digits of their derivative, and a line 10^-9 times its
// partner 8.
#pragma once
#include <cuda_runtime.h>
#include <math.h>

namespace lbm {
namespace fixed {

template <typename R> struct is_fixed {
    static constexpr bool value = false;
};
template <> struct is_fixed<long long> {
    static constexpr bool value = true;
};

// Second factors (roots, multipliers) are stored as balanced halves: low 32 bits as a signed
// integer bl in [-2^31, 2^31), high 32 bits bh with b = bh 2^32 + bl, |b| <= 2^63 - 2^31.
__host__ __device__ __forceinline__ long long balance(long long b) {
    return (long long)(((unsigned long long)(b + 0x80000000LL) & 0xffffffff00000000ULL) |
                       ((unsigned long long)b & 0xffffffffULL));
}
__host__ __device__ __forceinline__ int lo32(long long a) { return (int)(unsigned)(unsigned long long)a; }
__host__ __device__ __forceinline__ int hi32(long long a) { return (int)(a >> 32); }
// high half of a in balanced halves
__host__ __device__ __forceinline__ int bal_hi(long long a) {
    return hi32(a) + (int)((unsigned)lo32(a) >> 31);
}

// a b / 2^64 to the nearest integer (error at most 3/4: the low halves' product is left out),
// a as balanced halves (ah, al), b as (bh, bl); |a| <= 2^62.5. The middle products carry a bias of
// 2^63 (taken off again with the high product), so that their high word is unsigned and enters
// with a plain carry: three wide multiply-adds and two additions.
constexpr unsigned long long kMidBias = 0x8000000080000000ULL;  // 2^63, and 2^31 to round
constexpr unsigned long long kHighBias = 0ULL - 0x80000000ULL;
// a b + c with 32-bit signed factors, written as PTX's signed wide multiply-add: with products of
// 64-bit factors the column pass executed 49% more instructions (ncu's counter) and took 656 us per
// 1024^2 step instead of 484
__host__ __device__ __forceinline__ unsigned long long madw(int a, int b, unsigned long long c) {
#ifdef __CUDA_ARCH__
    unsigned long long r;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
    return r;
#else
    return (unsigned long long)((long long)a * b) + c;
#endif
}
__host__ __device__ __forceinline__ long long mulhi(int ah, int al, int bh, int bl) {
    const unsigned long long m = madw(al, bh, madw(ah, bl, kMidBias));
    return (long long)(madw(ah, bh, kHighBias) + (m >> 32));
}
// (a b + c d) / 2^64 with one rounding: the sum of the middle products stays below 2^63 for
// (a, c) of modulus up to 2^62.5 and (b, d) of modulus 2^62
__host__ __device__ __forceinline__ long long mulhi2(int ah, int al, int bh, int bl, int ch, int cl, int dh, int dl) {
    const unsigned long long m = madw(cl, dh, madw(ch, dl, madw(al, bh, madw(ah, bl, kMidBias))));
    return (long long)(madw(ch, dh, madw(ah, bh, kHighBias)) + (m >> 32));
}
__host__ __device__ __forceinline__ long long mulhi(long long a, long long b_balanced) {
    return mulhi(bal_hi(a), lo32(a), hi32(b_balanced), lo32(b_balanced));
}

__host__ __device__ __forceinline__ longlong2 mk2(long long x, long long y) {
    longlong2 c;
    c.x = x;
    c.y = y;
    return c;
}
// a / 4, rounded
__host__ __device__ __forceinline__ longlong2 quarter(longlong2 a) { return mk2((a.x + 2) >> 2, (a.y + 2) >> 2); }

// a w / 4 and a conj(w) / 4, w scaled to 2^62 in balanced halves
__host__ __device__ __forceinline__ longlong2 mul4(longlong2 a, longlong2 w) {
    const int xh = bal_hi(a.x), xl = lo32(a.x), yh = bal_hi(a.y), yl = lo32(a.y);
    const int ch = hi32(w.x), cl = lo32(w.x), sh = hi32(w.y), sl = lo32(w.y);
    return mk2(mulhi2(xh, xl, ch, cl, yh, yl, -sh, -sl), mulhi2(xh, xl, sh, sl, yh, yl, ch, cl));
}
__host__ __device__ __forceinline__ longlong2 mulc4(longlong2 a, longlong2 w) {
    const int xh = bal_hi(a.x), xl = lo32(a.x), yh = bal_hi(a.y), yl = lo32(a.y);
    const int ch = hi32(w.x), cl = lo32(w.x), sh = hi32(w.y), sl = lo32(w.y);
    return mk2(mulhi2(xh, xl, ch, cl, yh, yl, sh, sl), mulhi2(yh, yl, ch, cl, xh, xl, -sh, -sl));
}

// Constants of the 16-point transform, scaled to 2^64 (all below 1/2): tan(pi/16), sin(pi/8),
// 1 - sqrt(1/2)
constexpr unsigned long long kTan = 0x32EBEBC0AA62B00FULL;
constexpr unsigned long long kSin = 0x61F78A9ABAA58B47ULL;
constexpr unsigned long long kOneMinusSqrtHalf = 0x4AFB0CCC06219B7CULL;

// a (constant c / 2^64)
template <unsigned long long C> __host__ __device__ __forceinline__ long long scale_const(long long a) {
    constexpr int bl = (int)(unsigned)(C & 0xffffffffULL);
    constexpr int bh = (int)((C + 0x80000000ULL) >> 32);
    return mulhi(bal_hi(a), lo32(a), bh, bl);
}
// rotation by -pi/8 (NEG) or +pi/8 as three shears (lifting steps): three products instead of four
template <bool NEG> __host__ __device__ __forceinline__ longlong2 rot_pi8(longlong2 a) {
    const long long d = scale_const<kTan>(a.y);
    const long long x = NEG ? a.x + d : a.x - d;
    const long long g = scale_const<kSin>(x);
    const long long y = NEG ? a.y - g : a.y + g;
    const long long h = scale_const<kTan>(y);
    return mk2(NEG ? x + h : x - h, y);
}
__host__ __device__ __forceinline__ long long sqrt_half(long long a) {
    return a - scale_const<kOneMinusSqrtHalf>(a);
}
// a w16^M, unscaled (w16 = exp(-2 pi i / 16), the conjugate if INV)
template <bool INV, int M> __host__ __device__ __forceinline__ longlong2 w16(longlong2 a) {
    static_assert(M == 1 || M == 2 || M == 3 || M == 4 || M == 6 || M == 9, "roots of the 16-point transform");
    // multiplication by w16^4 = -i (forward), +i (inverse)
    auto quarter_turn = [](longlong2 z) { return INV ? mk2(-z.y, z.x) : mk2(z.y, -z.x); };
    if constexpr (M == 1) return rot_pi8<!INV>(a);
    if constexpr (M == 2) {
        return INV ? mk2(sqrt_half(a.x - a.y), sqrt_half(a.x + a.y)) : mk2(sqrt_half(a.x + a.y), sqrt_half(a.y - a.x));
    }
    if constexpr (M == 3) return quarter_turn(rot_pi8<INV>(a));
    if constexpr (M == 4) return quarter_turn(a);
    if constexpr (M == 6) {
        const long long s = sqrt_half(a.x + a.y), d = sqrt_half(a.y - a.x);
        return INV ? mk2(-s, -d) : mk2(d, -s);
    }
    if constexpr (M == 9) {
        const longlong2 r = rot_pi8<!INV>(a);
        return mk2(-r.x, -r.y);
    }
}

// ---- line scaling ------------------------------------------------------------------------
constexpr int kGrid = 61;  // points are cut off at 2^-61 of the line's bound or coarser, before the mean is taken off
// bits of any line of 2^LOG2N points, LOG2N <= 6 (see line_bits, with l1 = l2 + LOG2N / 2 = LOG2N + 1/2)
template <int LOG2N> constexpr int kShortBits = LOG2N < 4 ? 62 - LOG2N : 58;
// Bits B of the input points of a line of more, at least 30. m, l2: log2, relative to 2^e, of bounds of the largest real number and of
// the 2-norm (the root of the sum of all squares). l1: of the sum of all |Re| + |Im|, or 1/2 less than
// of N^(1/2) times the 2-norm.
template <int LOG2N> __host__ __device__ __forceinline__ int line_bits(float m, float l1, float l2) {
    float best = kGrid;
    // forward: sums of 2^g points have moduli of at most 2^(m + 1/2 + g), and of at most 2^l1 or
    // 2^(l1 + 1/2). They may reach 2^62.5, but the sum Re + Im of a quarter of a pass is formed too:
    // it has a quarter of the first bound, half of the third, but sqrt(2) times the second.
    int g = 0, twiddled = 0, left = LOG2N;
    if constexpr (LOG2N >= 4) {
#pragma unroll
        for (int p = 0; p < LOG2N / 4; ++p) {
            g += 4;
            best = fminf(best, 62.f + 2 * twiddled - fminf(m + g, l1));
            left -= 4;
            if (left > 0) ++twiddled;
        }
    }
    if (left > 0) best = fminf(best, 62.f + 2 * twiddled - fminf(m + g + left, l1));
    // inverse: the 2-norm of the products times sqrt(P) 4^-t after passes over P points, t of them
    // twiddled, in half bits
    int points = LOG2N & 3, t = 0, growth = points;
    if constexpr (LOG2N >= 4) {
#pragma unroll
        for (int p = LOG2N / 4 - 1; p >= 0; --p) {
            if (LOG2N - 4 - 4 * p > 0) ++t;
            points += 4;
            growth = growth > points - 4 * t ? growth : points - 4 * t;
        }
    }
    best = fminf(best, 62.9f - 0.5f * (LOG2N - 4 * twiddled - 4 + growth) - l2);
    return (int)fmaxf(best, 30.f);  // (NaN lines: any value)
}

// exponent fields below this (2^-959) count as zero, a line of such values transforms to zero
constexpr int kMinExp = 64;

// x 2^(B - e), truncated, B <= kGrid, from the bits of the double x; e = emax - 1022 (emax: the largest
// exponent field of the line, kMinExp <= emax <= 2046), top = emax + kGrid - B
__host__ __device__ __forceinline__ long long from_double(unsigned long long x, int top) {
    const int hi = (int)(x >> 32);
    int d = top - (int)(((unsigned)hi >> 20) & 0x7ffu);
    d = d < 63 ? d : 63;
    const unsigned long long mant =
        ((unsigned long long)(((unsigned)hi & 0xfffffu) | 0x100000u) << 32) | (x & 0xffffffffULL);
    const long long v = (long long)((mant << (kGrid - 53)) >> d);
    return hi < 0 ? -v : v;
}
// x 2^-e as a float from the high word of its bits, truncated; off = (emax - 126) 2^20, least the larger
// of it and 2^20 - 1. 0 for zeros and below the float's normal range.
__host__ __device__ __forceinline__ float relative(unsigned hi, int off, int least) {
    const int h = (int)(hi & 0x7fffffffu);
    const unsigned b = (h > least ? (unsigned)(h - off) << 3 : 0u) | (hi & 0x80000000u);
#ifdef __CUDA_ARCH__
    return __uint_as_float(b);
#else
    float f;
    __builtin_memcpy(&f, &b, 4);
    return f;
#endif
}

__host__ __device__ __forceinline__ int clz64(unsigned long long m) {
#ifdef __CUDA_ARCH__
    return __clzll((long long)m);
#else
    return m ? __builtin_clzll(m) : 64;
#endif
}
// bits of the double y 2^ex, rounded to nearest, -960 <= ex <= 950 (no overflow or underflow)
__host__ __device__ __forceinline__ unsigned long long to_double(long long y, int ex) {
    const unsigned long long m = y < 0 ? 0ULL - (unsigned long long)y : (unsigned long long)y;
    const int lz = clz64(m);
    const unsigned long long v = (((m << lz) >> 1) + 0x200) >> 10;  // in [2^52, 2^53]
    const unsigned hi = (unsigned)(v >> 32) + ((unsigned)(ex + 1023 + 62 - lz) << 20);
    const unsigned long long r = ((unsigned long long)(hi | ((unsigned)(y >> 32) & 0x80000000u)) << 32) | (v & 0xffffffffULL);
    return m ? r : 0ULL;
}

// Sum of 16 floats (their bits) as the bits of a double: exact but for what lies below 2^-58 of the
// largest (less than one rounding of a float64 sum), then rounded once. False, and no sum, where the
// largest is below 2^-63, infinite or NaN.
__host__ __device__ __forceinline__ bool sum16(const unsigned f[16], unsigned long long &bits) {
    unsigned top = 0;
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        const unsigned a = f[i] & 0x7fffffffu;
        top = a > top ? a : top;
    }
    const int et = (int)(top >> 23);  // every |f| < 2^(et - 126)
    long long sum = 0;                // unit 2^(et - 185): 16 values below 2^59
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        const int sh = (int)((f[i] >> 23) & 0xffu) - et + 35;
        const unsigned m = (f[i] & 0x7fffffu) | 0x800000u;
        const unsigned long long v = sh >= 0 ? (unsigned long long)m << (sh & 63) : (unsigned long long)(m >> (-sh < 31 ? -sh : 31));
        sum += (int)f[i] < 0 ? -(long long)v : (long long)v;
    }
    bits = to_double(sum, et - 185);
    return et >= 64 && et < 255;
}

// A real factor c = m 2^ex as a fixed-point number m 2^62 (|m| in [1/2, 1)) in balanced halves
struct Factor {
    long long m;
    int ex;
};
__host__ __device__ __forceinline__ Factor factor(unsigned long long bits) {
    Factor f;
    const int E = (int)((bits >> 52) & 0x7ff);
    const long long v = (long long)(((bits & 0xfffffffffffffULL) | 0x10000000000000ULL) << 9);  // [2^61, 2^62)
    f.m = E == 0 ? 0 : balance((long long)bits < 0 ? -v : v);
    f.ex = E - 1022;
    return f;
}

}  // namespace fixed
}  // namespace lbm
