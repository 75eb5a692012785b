// Spectral line operators: what the passes call to differentiate a line. Line<float> is the
// float32 transform of fft_reg.cuh; Line<double> runs the same passes in 64-bit fixed point
// (fft_fixed.cuh): the line's common exponent and mean from reductions over its threads, integer
// points between forward() and inverse(), and float64 values again after it. The spectrum between the
// two is opaque to the caller (it may be kept with storeF and read back with loadF); Scale carries
// the line's exponent along with it. Calls go in the order forward, multiply, inverse; a spectrum that
// is read back goes through multiply and inverse again.
#pragma once
#include "fft_reg.cuh"

namespace lbm {

// twiddles and derivative multipliers of one axis (digit-reversed order, see fft_reg.cuh)
template <typename R> struct Axis {
    const typename cplx<R>::T *tw;  // exp(-2 pi i k/N), k < N
    const R *k1;                    // k_eff(m(p)) / N, 0 at Nyquist
    const R *k2;                    // -k_eff(m(p))^2 / N, 0 at Nyquist
    int log2n;
};
// float64 path: the same as fixed-point numbers in balanced halves (fft_fixed.cuh): roots scaled
// to 2^62, multipliers to 2^62 of 2^p1 and 2^p2
template <> struct Axis<double> {
    const longlong2 *tw;
    const long long *k1, *k2;
    int log2n;
    int p1, p2;
};

namespace reg {

// What the float64 lines' reductions have room for: a line whose threads spread over 8 warps, and a
// column tile of 16 lines (rows of 256 bytes); the launchers take no more.
constexpr int kLineWarps = 8, kTileLines = 16;
template <typename R> constexpr bool tile_fits(int lines, int threads) {
    return sizeof(R) == 4 || (lines <= kTileLines && threads <= 32 * kLineWarps);
}

// st: distance between the threads of consecutive t (1: a line's threads are consecutive, the row
// passes; L: the L lines of a column tile are interleaved, line index fastest)
template <typename R, int LOG2N, bool PK, int CS = 1> struct Line : LineFFT<R, LOG2N, PK, CS> {
    using B = LineFFT<R, LOG2N, PK, CS>;
    using typename B::CT;
    struct Scale {};
    template <class SYNC> static __device__ __forceinline__ Scale forward(CT v[B::E], CT *buf, int t, const Axis<R> &ax, int) {
        B::template forward<SYNC>(v, buf, t, ax.tw);
        return Scale{};
    }
    template <class SYNC> static __device__ __forceinline__ void multiply(CT v[B::E], int t, int order, R c, const Axis<R> &ax, Scale &, int) {
        B::multiply(v, t, order, c, ax.k1, ax.k2);
    }
    template <class SYNC> static __device__ __forceinline__ void inverse(CT v[B::E], CT *buf, int t, const Axis<R> &ax, Scale) {
        B::template inverse<SYNC>(v, buf, t, ax.tw);
    }
    // barriers only, of forward, and of multiply and inverse (see LineFFT)
    template <class SYNC> static __device__ __forceinline__ void idle_forward(int) { B::template idle_forward<SYNC>(); }
    template <class SYNC> static __device__ __forceinline__ void idle_inverse(int) { B::template idle_inverse<SYNC>(); }
};

template <int LOG2N, bool PK, int CS> struct Line<double, LOG2N, PK, CS> : LineFFT<long long, LOG2N, false, CS> {
    using B = LineFFT<long long, LOG2N, false, CS>;
    typedef double2 CT;
    static constexpr int E = B::E, G = B::G, GL = B::GL, T = B::TWIDDLED;
    // the real and the imaginary parts, which are two real lines, are integers times 2^ex and 2^ey; all of
    // them NaN, or all zero, where these lie near kNan and kZero
    struct Scale {
        int ex, ey;
    };
    static constexpr int kNan = 1 << 20, kZero = -(1 << 20);

    static __device__ __forceinline__ void get(longlong2 u[E], const CT v[E]) {
#pragma unroll
        for (int e = 0; e < E; ++e) u[e] = fixed::mk2(__double_as_longlong(v[e].x), __double_as_longlong(v[e].y));
    }
    static __device__ __forceinline__ void put(CT v[E], const longlong2 u[E]) {
#pragma unroll
        for (int e = 0; e < E; ++e) v[e] = make_double2(__longlong_as_double(u[e].x), __longlong_as_double(u[e].y));
    }
    static __device__ __forceinline__ void storeF(const CT v[E], CT *buf, int t) {
        longlong2 u[E];
        get(u, v);
        B::storeF(u, reinterpret_cast<longlong2 *>(buf), t);
    }
    static __device__ __forceinline__ void loadF(CT v[E], const CT *buf, int t) {
        longlong2 u[E];
        B::loadF(u, reinterpret_cast<const longlong2 *>(buf), t);
        put(v, u);
    }
    static __device__ __forceinline__ void store_natural(const CT v[E], CT *buf, int t) {
        longlong2 u[E];
        get(u, v);
        B::store_natural(u, reinterpret_cast<longlong2 *>(buf), t);
    }

    // Lines of up to 64 points take as many bits as the largest magnitude allows and keep their mean: their
    // errors are at most the float64 transform's as it is, and their passes wait for instructions (64^2
    // float64 step 155 us, 167 with the general form).
    static constexpr bool kShort = LOG2N <= 6;

    static __device__ __forceinline__ long long shl(long long a, int n) { return (long long)((unsigned long long)a << n); }

    // Reduces w[0 .. W-1] over the line's threads with op(k, a, b), a commutative operation for each
    // word k whose neutral element is 0. The tree pairs the bits of t from the lowest up whatever st is, so the
    // result does not depend on the tile shape even where op rounds (float sums). Where a line's
    // threads span warps it takes one CTA barrier and words [SLOT, SLOT + W) of the scratch: a call
    // that may run while another thread still reads the last one's words takes others.
    static constexpr int kSlots = 6;
    template <class SYNC, int SLOT, int W, class OP> static __device__ __forceinline__ void reduce(unsigned (&w)[W], int st, OP op) {
        static_assert(SLOT + W <= kSlots, "scratch words");
        if constexpr (G == 1) return;
        const int tid = threadIdx.x, lane = tid & 31;
        const int n = GL * st;  // threads over which the line's threads spread (spans_warps: more than a warp's)
        const unsigned mask = n >= 32 ? 0xffffffffu : ((1u << n) - 1u) << (lane & ~(n - 1));
        for (int off = st; off < 32 && off < n; off <<= 1)
#pragma unroll
            for (int k = 0; k < W; ++k) w[k] = op(k, w[k], __shfl_xor_sync(mask, w[k], off));
        if (spans_warps(st)) {
            // one entry per warp and line
            unsigned(*part)[kPart] = scratch();
            const int nw = n >> 5, wp = tid >> 5, l = tid & (st - 1);
            if (lane < st) {
#pragma unroll
                for (int k = 0; k < W; ++k) part[SLOT + k][wp * st + l] = w[k];
            }
            SYNC::run();
            const int w0 = wp & ~(nw - 1);
#pragma unroll
            for (int k = 0; k < W; ++k) {
                unsigned r[kLineWarps];
#pragma unroll
                for (int i = 0; i < kLineWarps; ++i) r[i] = i < nw ? part[SLOT + k][(w0 + i) * st + l] : 0u;
#pragma unroll
                for (int d = 1; d < kLineWarps; d <<= 1)
#pragma unroll
                    for (int i = 0; i + d < kLineWarps; i += 2 * d) r[i] = op(k, r[i], r[i + d]);
                w[k] = r[0];
            }
        }
        if constexpr (CS > 1) {  // the other CTAs' parts of the line, through distributed shared memory
            __shared__ unsigned cpart[W][CS * kTileLines];
            const int l = tid & (st - 1);
            cluster_barrier();
            if (tid < st) {
#pragma unroll
                for (int r = 0; r < CS; ++r)
#pragma unroll
                    for (int k = 0; k < W; ++k) {
                        const uint32_t p = cluster_map(&cpart[k][cluster_rank() * kTileLines + l], r);
                        asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(p), "r"(w[k]) : "memory");
                    }
            }
            cluster_barrier();
#pragma unroll
            for (int k = 0; k < W; ++k) {
                unsigned r[CS];
#pragma unroll
                for (int i = 0; i < CS; ++i) r[i] = cpart[k][i * kTileLines + l];
#pragma unroll
                for (int d = 1; d < CS; d <<= 1)
#pragma unroll
                    for (int i = 0; i + d < CS; i += 2 * d) r[i] = op(k, r[i], r[i + d]);
                w[k] = r[0];
            }
        }
    }
    static __device__ __forceinline__ bool spans_warps(int st) { return GL * st > 32; }
    static constexpr int kPart = kLineWarps * kTileLines;
    static __device__ __forceinline__ unsigned (*scratch())[kPart] {
        __shared__ unsigned part[kSlots][kPart];
        return part;
    }

    template <class SYNC> static __device__ __forceinline__ Scale forward(CT v[E], CT *buf, int t, const Axis<double> &ax, int st) {
        longlong2 u[E];
        get(u, v);
        // the two lines' largest magnitudes (high words order as the values do): each has its own exponent,
        // so that neither loses bits to a larger partner
        unsigned top[2] = {0, 0};
#pragma unroll
        for (int e = 0; e < E; ++e) {
            top[0] = max(top[0], (unsigned)(u[e].x >> 32) & 0x7fffffffu);
            top[1] = max(top[1], (unsigned)(u[e].y >> 32) & 0x7fffffffu);
        }
        reduce<SYNC, 0>(top, st, [](int, unsigned a, unsigned b) { return max(a, b); });
        const int ex = (int)(top[0] >> 20), ey = (int)(top[1] >> 20);
        int bits = fixed::kShortBits<LOG2N>;
        long long cx = 0, cy = 0;
        if constexpr (!kShort) {
            // sums relative to them
            const int ox = (ex - 126) << 20, oy = (ey - 126) << 20, least_x = max(ox, (1 << 20) - 1), least_y = max(oy, (1 << 20) - 1);
            float l1 = 0.f, l2 = 0.f, sx = 0.f, sy = 0.f;  // magnitudes, squares, the two fields' values
#pragma unroll
            for (int e = 0; e < E; ++e) {
                const float x = fixed::relative((unsigned)(u[e].x >> 32), ox, least_x), y = fixed::relative((unsigned)(u[e].y >> 32), oy, least_y);
                l1 += fabsf(x) + fabsf(y);
                l2 = fmaf(x, x, fmaf(y, y, l2));
                sx += x;
                sy += y;
            }
            unsigned sums[4] = {__float_as_uint(l1), __float_as_uint(l2), __float_as_uint(sx), __float_as_uint(sy)};
            reduce<SYNC, 2>(sums, st, [](int, unsigned a, unsigned b) { return __float_as_uint(__fadd_rn(__uint_as_float(a), __uint_as_float(b))); });
            // bits with the points as they are, and with the mean taken out: the sum of squares about it (the
            // truncated values' relative error, 2^-19, covered) bounds the largest deviation and any sum of P
            // points; a hundredth covers the rounding of sums and logarithms
            const float s2 = __uint_as_float(sums[1]), mx = __uint_as_float(sums[2]) * (1.f / B::N), my = __uint_as_float(sums[3]) * (1.f / B::N);
            const float d2 = fmaxf(s2 - B::N * (mx * mx + my * my), 0.f) + s2 * 0x1p-16f;
            const float ld = 0.5f * __log2f(d2) + 0.01f;
            bits = fixed::line_bits<LOG2N>(0.f, __log2f(__uint_as_float(sums[0])) + 0.01f, 0.5f * __log2f(s2) + 0.01f);
            const int about = fixed::line_bits<LOG2N>(fminf(1.f, ld), ld + 0.5f * (LOG2N - 1), ld);
            if (about > bits) {
                bits = about;
                cx = shl((long long)__float2int_rn(mx * 0x1p30f), bits - 30);
                cy = shl((long long)__float2int_rn(my * 0x1p30f), bits - 30);
            }
        }
        const int g = fixed::kGrid - bits, shift_x = ex < fixed::kMinExp ? 1 << 12 : ex + g, shift_y = ey < fixed::kMinExp ? 1 << 12 : ey + g;
#pragma unroll
        for (int e = 0; e < E; ++e)
            u[e] = fixed::mk2(fixed::from_double((unsigned long long)u[e].x, shift_x) - cx,
                              fixed::from_double((unsigned long long)u[e].y, shift_y) - cy);
        B::template forward<SYNC>(u, reinterpret_cast<longlong2 *>(buf), t, ax.tw);
        put(v, u);
        const bool bad = max(ex, ey) == 0x7ff;
        Scale s;
        s.ex = bad ? kNan : ex < fixed::kMinExp ? kZero : ex - 1022 - bits + 2 * T;
        s.ey = bad ? kNan : ey < fixed::kMinExp ? kZero : ey - 1022 - bits + 2 * T;
        return s;
    }

    // v <- d^order c v, as integers whose magnitudes sum to just below 2^63 where that is an upward shift
    template <class SYNC> static __device__ __forceinline__ void multiply(CT v[E], int t, int order, double c, const Axis<double> &ax, Scale &s, int st) {
        longlong2 u[E];
        get(u, v);
        const long long *k = order == 1 ? ax.k1 : ax.k2;
        int pre, post;  // shifts of the points and of the products
        if constexpr (G == 1) {  // a whole line: the points' sum in units of 2^6, rounded up, kept below 2^62
            unsigned long long sum = 1;
#pragma unroll
            for (int e = 0; e < E; ++e) {
                const long long x = u[e].x ^ (u[e].x >> 63), y = u[e].y ^ (u[e].y >> 63);
                if (__ldg(k + e) != 0) sum += ((unsigned long long)x >> 6) + ((unsigned long long)y >> 6) + 2;
            }
            const int lz = fixed::clz64(sum);
            pre = max(lz - 8, 0);
            post = min(max(lz - 6, 0), 2);
        } else if constexpr (LOG2N <= 8) {  // the points' sum in units of 2^40 (enough up to 256 points)
            unsigned r[1] = {2 * E};
#pragma unroll
            for (int e = 0; e < E; ++e) {
                const int hx = fixed::hi32(u[e].x), hy = fixed::hi32(u[e].y);
                if (__ldg(k + G * e + t) != 0) r[0] += ((unsigned)(hx ^ (hx >> 31)) >> 8) + ((unsigned)(hy ^ (hy >> 31)) >> 8);
            }
            reduce<SYNC, 0>(r, st, [](int, unsigned a, unsigned b) { return a + b; });
            const int total = __clz((int)(r[0] + 2u * B::N)) - 9;
            pre = max(total, 0);
            post = min(max(total + 2, 0), 2);
        } else {  // the products' sum in units of 2^36 (two more for each that is cut off); the points' highest bit
            unsigned r[2] = {0, 4 * E};
#pragma unroll
            for (int e = 0; e < E; ++e) {
                const long long w = __ldg(k + G * e + t);
                const unsigned hx = (unsigned)(fixed::hi32(u[e].x) ^ (fixed::hi32(u[e].x) >> 31)), hy = (unsigned)(fixed::hi32(u[e].y) ^ (fixed::hi32(u[e].y) >> 31));
                if (w != 0) {
                    const unsigned wh = ((unsigned)abs(fixed::hi32(w)) >> 4) + 1;
                    r[0] |= hx | hy;
                    r[1] += __umulhi(hx, wh) + __umulhi(hy, wh);
                }
            }
            reduce<SYNC, 0>(r, st, [](int k, unsigned a, unsigned b) { return k == 0 ? a | b : a + b; });
            const int total = __clz((int)(r[1] + 2u * B::N)) - 5;
            pre = max(min(total, __clz((int)r[0]) - 2), 0);
            post = max(total - pre, 0);
        }
        const bool unit = c == 1.0;
        const fixed::Factor f = fixed::factor((unsigned long long)__double_as_longlong(c));
        const int scale = 2 + (order == 1 ? ax.p1 : ax.p2) + (unit ? 0 : f.ex) - pre - post;
        s.ex += scale;
        s.ey += scale;
#pragma unroll
        for (int e = 0; e < E; ++e) {
            long long w = __ldg(k + G * e + t);
            if (!unit) w = fixed::balance(fixed::mulhi(fixed::hi32(w), fixed::lo32(w), fixed::hi32(f.m), fixed::lo32(f.m)) << 2);
            const long long x = shl(fixed::mulhi(shl(u[e].x, pre), w), post), y = shl(fixed::mulhi(shl(u[e].y, pre), w), post);
            u[e] = order == 1 ? fixed::mk2(-y, x) : fixed::mk2(x, y);
        }
        put(v, u);
    }

    template <class SYNC> static __device__ __forceinline__ void inverse(CT v[E], CT *buf, int t, const Axis<double> &ax, Scale s) {
        longlong2 u[E];
        get(u, v);
        B::template inverse<SYNC>(u, reinterpret_cast<longlong2 *>(buf), t, ax.tw);
        const int ex = s.ex + 2 * T, ey = s.ey + 2 * T;
        if (min(ex, ey) > -960 && max(ex, ey) < 950) {
#pragma unroll
            for (int e = 0; e < E; ++e)
                u[e] = fixed::mk2((long long)fixed::to_double(u[e].x, ex), (long long)fixed::to_double(u[e].y, ey));
            put(v, u);
        } else {  // NaN and zero lines, and results near the ends of the float64 range
            const bool bad = ex > kNan / 2;
            auto pow2 = [](int k) { return __longlong_as_double((long long)(k + 1023) << 52); };
            auto value = [&](long long y, int k) {
                const double p = k < 0 ? pow2(-900) : pow2(900);
                const double q = k < 0 ? pow2(max(k + 900, -1022)) : pow2(min(k - 900, 1000));
                return __longlong_as_double((long long)fixed::to_double(y, 0)) * p * q;
            };
#pragma unroll
            for (int e = 0; e < E; ++e)
                v[e] = bad ? make_double2(__longlong_as_double(0x7ff8000000000000LL), __longlong_as_double(0x7ff8000000000000LL))
                           : make_double2(value(u[e].x, ex), value(u[e].y, ey));
        }
    }

    // barriers only, of forward, and of multiply and inverse (see LineFFT): those of the reductions of a
    // line that spans warps as well
    template <class SYNC> static __device__ __forceinline__ void idle_forward(int st) {
        static_assert(CS == 1, "float64 rows are not split over clusters");
        if (spans_warps(st)) {
            SYNC::run();
            SYNC::run();
        }
        B::template idle_forward<SYNC>();
    }
    template <class SYNC> static __device__ __forceinline__ void idle_inverse(int st) {
        static_assert(CS == 1, "float64 rows are not split over clusters");
        if (spans_warps(st)) SYNC::run();
        B::template idle_inverse<SYNC>();
    }
};

}  // namespace reg
}  // namespace lbm
