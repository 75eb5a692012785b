// Spectral line operators: what the passes call to differentiate a line. Line<float> is the
// float32 transform of fft_reg.cuh; Line<double> runs the same passes in 64-bit fixed point
// (fft_fixed.cuh): the line's common exponent from one reduction over its threads, integer points
// between forward() and inverse(), and float64 values again after it. The spectrum between the two
// is opaque to the caller (it may be kept with storeF and read back with loadF); Scale carries
// the line's exponent along with it.
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
    static __device__ __forceinline__ void multiply(CT v[B::E], int t, int order, R c, const Axis<R> &ax, Scale &) {
        B::multiply(v, t, order, c, ax.k1, ax.k2);
    }
    template <class SYNC> static __device__ __forceinline__ void inverse(CT v[B::E], CT *buf, int t, const Axis<R> &ax, Scale, int) {
        B::template inverse<SYNC>(v, buf, t, ax.tw);
    }
};

template <int LOG2N, bool PK, int CS> struct Line<double, LOG2N, PK, CS> : LineFFT<long long, LOG2N, false, CS> {
    using B = LineFFT<long long, LOG2N, false, CS>;
    typedef double2 CT;
    static constexpr int E = B::E, G = B::G, GL = B::GL, T = B::TWIDDLED;
    // values are integers times 2^ex; all of them NaN, or all zero, where ex is one of these
    struct Scale {
        int ex;
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

    // Whether a line's threads span warps (then the reductions take one CTA barrier each).
    static __device__ __forceinline__ bool spans_warps(int st) { return GL * st > 32; }

    // Reduces (a, b) over the line's threads with op, a commutative pair operation. The tree pairs
    // the bits of t from the lowest up whatever st is, so the result does not depend on the tile
    // shape even where op rounds (b: a float sum).
    template <class SYNC, class OP> static __device__ __forceinline__ void reduce(unsigned &a, unsigned &b, int st, OP op) {
        if constexpr (G == 1) return;
        const int tid = threadIdx.x, lane = tid & 31;
        const int n = GL * st;  // threads over which the line's threads spread
        const unsigned mask = n >= 32 ? 0xffffffffu : ((1u << n) - 1u) << (lane & ~(n - 1));
        for (int off = st; off < 32 && off < n; off <<= 1) {
            const unsigned oa = __shfl_xor_sync(mask, a, off), ob = __shfl_xor_sync(mask, b, off);
            op(a, b, oa, ob);
        }
        if (n > 32) {
            __shared__ uint2 part[128];  // one entry per warp and line
            const int nw = n >> 5, w = tid >> 5, l = tid & (st - 1);
            if (lane < st) part[w * st + l] = make_uint2(a, b);
            SYNC::run();
            const int w0 = w & ~(nw - 1);
            uint2 r[8];  // a line spans at most 8 warps; (0, 0) is neutral
#pragma unroll
            for (int i = 0; i < 8; ++i) r[i] = i < nw ? part[(w0 + i) * st + l] : make_uint2(0u, 0u);
#pragma unroll
            for (int d = 1; d < 8; d <<= 1)
#pragma unroll
                for (int i = 0; i + d < 8; i += 2 * d) op(r[i].x, r[i].y, r[i + d].x, r[i + d].y);
            a = r[0].x;
            b = r[0].y;
        }
        if constexpr (CS > 1) {  // the other CTAs' parts of the line, through distributed shared memory
            __shared__ __align__(16) uint2 cpart[CS * 32];
            const int l = tid & (st - 1);
            cluster_barrier();
            if (tid < st) {
#pragma unroll
                for (int r = 0; r < CS; ++r) {
                    const uint32_t p = cluster_map(&cpart[cluster_rank() * 32 + l], r);
                    asm volatile("st.shared::cluster.v2.u32 [%0], {%1, %2};" ::"r"(p), "r"(a), "r"(b) : "memory");
                }
            }
            cluster_barrier();
            uint2 r[CS];
#pragma unroll
            for (int i = 0; i < CS; ++i) r[i] = cpart[i * 32 + l];
#pragma unroll
            for (int d = 1; d < CS; d <<= 1)
#pragma unroll
                for (int i = 0; i + d < CS; i += 2 * d) op(r[i].x, r[i].y, r[i + d].x, r[i + d].y);
            a = r[0].x;
            b = r[0].y;
        }
    }

    template <class SYNC> static __device__ __forceinline__ Scale forward(CT v[E], CT *buf, int t, const Axis<double> &ax, int st) {
        longlong2 u[E];
        get(u, v);
        // the line's largest magnitude (high words order as the values do) and the sum of all
        unsigned top = 0;
        float l1 = 0.f;
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const unsigned hx = (unsigned)(u[e].x >> 32) & 0x7fffffffu, hy = (unsigned)(u[e].y >> 32) & 0x7fffffffu;
            top = max(top, max(hx, hy));
            l1 += fixed::abs_approx(u[e].x) + fixed::abs_approx(u[e].y);
        }
        unsigned l1b = __float_as_uint(l1);
        reduce<SYNC>(top, l1b, st, [](unsigned &a, unsigned &b, unsigned oa, unsigned ob) {
            a = max(a, oa);
            b = __float_as_uint(__fadd_rn(__uint_as_float(b), __uint_as_float(ob)));
        });
        const int emax = (int)(top >> 20);
        // the sum counts where neither it nor its terms leave the float range: 2^c 2^e bounds it
        const int c = emax > 930 && emax < 1120 ? (int)(l1b >> 23) - 126 - (emax - 1022) : 62;
        const int bits = fixed::line_bits<LOG2N>(c);
        const int shift = emax + fixed::kMaxBits - bits;
#pragma unroll
        for (int e = 0; e < E; ++e)
            u[e] = fixed::mk2(fixed::from_double((unsigned long long)u[e].x, shift), fixed::from_double((unsigned long long)u[e].y, shift));
        B::template forward<SYNC>(u, reinterpret_cast<longlong2 *>(buf), t, ax.tw);
        put(v, u);
        Scale s;
        s.ex = emax == 0x7ff ? kNan : emax < fixed::kMinExp ? kZero : emax - 1022 - bits + 2 * T;
        return s;
    }

    // v <- d^order c v
    static __device__ __forceinline__ void multiply(CT v[E], int t, int order, double c, const Axis<double> &ax, Scale &s) {
        longlong2 u[E];
        get(u, v);
        const long long *k = order == 1 ? ax.k1 : ax.k2;
        const bool unit = c == 1.0;
        const fixed::Factor f = fixed::factor((unsigned long long)__double_as_longlong(c));
        if (s.ex != kNan && s.ex != kZero) s.ex += 2 + (order == 1 ? ax.p1 : ax.p2) + (unit ? 0 : f.ex);
#pragma unroll
        for (int e = 0; e < E; ++e) {
            long long w = __ldg(k + G * e + t);
            if (!unit) w = fixed::balance(fixed::mulhi(fixed::hi32(w), fixed::lo32(w), fixed::hi32(f.m), fixed::lo32(f.m)) << 2);
            const long long x = fixed::mulhi(u[e].x, w), y = fixed::mulhi(u[e].y, w);
            u[e] = order == 1 ? fixed::mk2(-y, x) : fixed::mk2(x, y);
        }
        put(v, u);
    }

    template <class SYNC> static __device__ __forceinline__ void inverse(CT v[E], CT *buf, int t, const Axis<double> &ax, Scale s, int st) {
        longlong2 u[E];
        get(u, v);
        // the sum of the spectrum's magnitudes in units of 2^40, rounded up: the shift that brings
        // it just below 2^63
        unsigned sum = 0, zero = 0;
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int hx = fixed::hi32(u[e].x), hy = fixed::hi32(u[e].y);
            sum += ((unsigned)(hx ^ (hx >> 31)) >> 8) + ((unsigned)(hy ^ (hy >> 31)) >> 8);
        }
        reduce<SYNC>(sum, zero, st, [](unsigned &a, unsigned &b, unsigned oa, unsigned ob) {
            a += oa;
            b |= ob;
        });
        int sh = __clz((int)(sum + 2u * B::N)) - 9;
        sh = sh > 0 ? sh : 0;
#pragma unroll
        for (int e = 0; e < E; ++e)
            u[e] = fixed::mk2((long long)((unsigned long long)u[e].x << sh), (long long)((unsigned long long)u[e].y << sh));
        B::template inverse<SYNC>(u, reinterpret_cast<longlong2 *>(buf), t, ax.tw);
        const int ex = s.ex + 2 * T - sh;
        if (ex > -960 && ex < 950) {
#pragma unroll
            for (int e = 0; e < E; ++e)
                u[e] = fixed::mk2((long long)fixed::to_double(u[e].x, ex), (long long)fixed::to_double(u[e].y, ex));
            put(v, u);
        } else {  // NaN and zero lines, and results near the ends of the float64 range
            const bool bad = s.ex == kNan;
            auto pow2 = [](int k) { return __longlong_as_double((long long)(k + 1023) << 52); };
            const double p = ex < 0 ? pow2(-900) : pow2(900);
            const double q = ex < 0 ? pow2(max(ex + 900, -1022)) : pow2(min(ex - 900, 1000));
#pragma unroll
            for (int e = 0; e < E; ++e) {
                const double x = __longlong_as_double((long long)fixed::to_double(u[e].x, 0)) * p * q;
                const double y = __longlong_as_double((long long)fixed::to_double(u[e].y, 0)) * p * q;
                v[e] = bad ? make_double2(__longlong_as_double(0x7ff8000000000000LL), __longlong_as_double(0x7ff8000000000000LL))
                           : make_double2(x, y);
            }
        }
    }

    // barriers only (see LineFFT): the reductions of a line that spans warps add one each
    template <class SYNC> static __device__ __forceinline__ void idle_forward() {
        static_assert(CS == 1, "float64 rows are not split over clusters");
        if constexpr (GL > 32) SYNC::run();
        B::template idle_forward<SYNC>();
    }
    template <class SYNC> static __device__ __forceinline__ void idle_inverse() {
        static_assert(CS == 1, "float64 rows are not split over clusters");
        if constexpr (GL > 32) SYNC::run();
        B::template idle_inverse<SYNC>();
    }
};

}  // namespace reg
}  // namespace lbm
