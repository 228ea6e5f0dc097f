// fx.cuh -- complex128 transforms in 64-bit fixed point for sm_103a.
//
// What bounds complex128 on this part is the FP64 pipe: 2 lanes a clock and SM
// (measured: 2.15 FMAs, 1.8 additions, 1.9 conversions), against 128 for integer
// additions (two instructions per 64-bit sum) and 27 for 32 x 32 -> 64 bit
// multiply-adds.  A 512-point transform takes 26.5 FP64 instructions a point,
// ~1700 issue slots' worth of the pipe; the same butterflies on 64-bit integers
// take ~25 wide multiply-adds and ~65 plain instructions.  So a line's values
// are brought to integers q with one exponent per line, value = q 2^ex, are
// transformed, and are rounded back to FP64 once.
//
// Accuracy.  Every intermediate value of a transform is a sum of the line's
// values with unit-modulus weights, hence at most S = sum(|re| + |im|): with
// S <= 2^60.5 units nothing overflows (the butterflies' half sums reach sqrt(2) S,
// and the products take less than 2^61).  The scale follows S and not N times the
// largest value, because a peaked line (a spectrum of a few modes) would lose up
// to log2 N bits that way.  A flat line loses sqrt(N) to S, though; transforms of
// 256 points and more therefore start with the larger of the scales that S and
// the first stages' own growth (their product of radices times the largest value)
// allow, and shift by what is still needed once, between two stages, after a look
// at the largest value there.  The roots of unity are rounded to 2^-62 (fx_root in
// api.cu): FP64 ones would be most of the error.  Measured against 64-bit-mantissa
// arithmetic (one RK4IP step, relative 2-norm, FP64 transforms / fixed point): Gaussian
// 3.5e-16 / 1.1e-16 at 64 points, 5.0e-16 / 1.3e-16 at 256, 6.7e-16 / 2.3e-16 at 2048;
// white noise 3.8e-16 / 1.8e-16 at 64, 5.9e-16 / 2.4e-16 at 512, 6.4e-16 / 3.1e-16 at
// 1024; 20 steps of one mode at 64 points 4.3e-15 / 5.7e-16.  Non-finite values make their
// whole line NaN; what lies below 2^-59 of a line's largest component is truncated (an
// FP64 transform loses it below 2^-53 of the line's norm), and denormals count as zero.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace xsde {

// Factors of modulus <= 1 as Q62 integers in two signed 32-bit limbs,
// c = (c1 2^32 + c0) 2^-62: (re1, re0, im1, im0).
//
// q * c keeps q's units: q = q1 2^32 + q0 with q0 signed too, and
//   q c = ((q1 c1) << 2) + ((q1 c0 + q0 c1 + round) >> 30),
// the product q0 c0 (below one unit) left out: limbs with signs make its mean zero.
// Three wide multiply-adds for a real product, twelve for a complex one.
struct FxLimbs {
    int hi, lo;
};
__device__ __forceinline__ FxLimbs fx_split(long long q) {
    FxLimbs r;
    r.lo = (int)(uint32_t)(uint64_t)q;
    r.hi = (int)(q >> 32) - (r.lo >> 31);
    return r;
}
constexpr long long kFxHalf = 1ll << 29;

__device__ __forceinline__ long long mul_rsqrt2(long long a) {   // a / sqrt(2)
    constexpr int c1 = 759250125, c0 = -25716447;   // 2^62 / sqrt(2) = 3260954456333195553
    const FxLimbs s = fx_split(a);
    const long long mid = (long long)s.hi * c0 + ((long long)s.lo * c1 + kFxHalf);
    return (long long)(s.hi << 2) * c1 + (mid >> 30);
}

// u * w (S < 0) or u * conj(w) (S > 0)
template <int S> __device__ __forceinline__ longlong2 twiddle_mul(longlong2 u, int4 w) {
    const FxLimbs x = fx_split(u.x), y = fx_split(u.y);
    const int s1 = S < 0 ? w.z : -w.z, s0 = S < 0 ? w.w : -w.w;
    const int n1 = S < 0 ? -w.z : w.z, n0 = S < 0 ? -w.w : w.w;   // minus the imaginary part
    long long mr = (long long)x.hi * w.y + kFxHalf, mi = (long long)x.hi * s0 + kFxHalf;
    mr += (long long)x.lo * w.x;
    mi += (long long)x.lo * s1;
    mr += (long long)y.hi * n0;
    mi += (long long)y.hi * w.y;
    mr += (long long)y.lo * n1;
    mi += (long long)y.lo * w.x;
    const int x4 = x.hi << 2, y4 = y.hi << 2;
    longlong2 r;
    r.x = (long long)y4 * n1 + ((long long)x4 * w.x + (mr >> 30));
    r.y = (long long)y4 * w.x + ((long long)x4 * s1 + (mi >> 30));
    return r;
}

// ---------------------------------------------------------------------------
// line <-> integers.  A `Group` is the set of threads that carry one line and
// combines their values: max(m) and sum(m) on NV unsigned words, the result in
// every thread.
// ---------------------------------------------------------------------------
constexpr int kFxBad = 1 << 20;   // exponent of a line that held NaN or Inf
constexpr int kFxNone = -(1 << 20);   // a factor table without limbs
constexpr int kFxTop = 59;        // bit that the largest exponent's leading one takes

__device__ __forceinline__ uint32_t fx_hi(double v) { return (uint32_t)__double2hiint(v); }

// v 2^-(em - 1023 - kFxTop), truncated (the exponent field of v is at most em;
// field 0, zeros and denormals, gives 0: bringing denormals into range first costs every
// line 1 to 5 %, a branch between the reduction and the conversions)
__device__ __forceinline__ long long fx_from(double v, int em) {
    const long long b = __double_as_longlong(v);
    const int e = (int)((fx_hi(v) >> 20) & 0x7ffu);
    const int r = e ? em - e : 64;
    unsigned long long m = (((unsigned long long)b & 0xfffffffffffffull) | 0x10000000000000ull) << (kFxTop - 52);
    asm("shr.u64 %0, %0, %1;" : "+l"(m) : "r"(r));   // amounts past 63 give 0
    const long long s = b >> 63;
    return ((long long)m ^ s) - s;
}

// q 2^ex for lines whose exponents may leave FP64's normal range
static __device__ __noinline__ double fx_to_slow(long long q, int ex) {
    if (ex == kFxBad) return __longlong_as_double(0x7ff8000000000000ll);
    return scalbn((double)q, ex);
}
// q 2^ex, rounded once: the leading one is brought to bit 63 of (nh, nl), and
// the 53 bits below it, the exponent and the sign are put together by one
// 64-bit addition that also carries the rounding
__device__ __forceinline__ double fx_to(long long q, int ex) {
    const unsigned long long a = (unsigned long long)(q < 0 ? -q : q);
    const uint32_t ah = (uint32_t)(a >> 32), al = (uint32_t)a;
    const bool big = ah != 0u;
    const uint32_t t = big ? ah : al, l = big ? al : 0u;
    const int n = __clz((int)t);
    const uint32_t nh = __funnelshift_l(l, t, n), nl = __funnelshift_l(0u, l, n);
    const int em1 = ex + (big ? 1022 + 63 : 1022 + 31) - n;   // biased exponent less one
    uint32_t hi = (uint32_t)em1 << 20;
    hi = t ? hi | ((uint32_t)(q >> 32) & 0x80000000u) : 0u;
    const unsigned long long add = ((unsigned long long)hi << 32) | ((nl >> 10) & 1u);
    const unsigned long long m = ((unsigned long long)(nh >> 11) << 32) | __funnelshift_r(nl, nh, 11);
    return __longlong_as_double((long long)(m + add));
}

template <int NV, int E> __device__ __forceinline__ void fx_shift(longlong2 (&q)[NV][E], int (&ex)[NV], const int (&sh)[NV]) {
#pragma unroll
    for (int iv = 0; iv < NV; ++iv)
        if (sh[iv] > 0) {
            const long long half = 1ll << (sh[iv] - 1);
#pragma unroll
            for (int m = 0; m < E; ++m) {
                q[iv][m].x = (q[iv][m].x + half) >> sh[iv];
                q[iv][m].y = (q[iv][m].y + half) >> sh[iv];
            }
            if (ex[iv] != kFxBad) ex[iv] += sh[iv];
        }
}

// the shift that keeps sums of 2^lg values within 2^60.5, their |re| and |im|
// being below 2^32 m
__device__ __forceinline__ int fx_growth(uint32_t m, int lg) { return 32 - __clz((int)m) + lg - 28; }
template <int NV, int E> __device__ __forceinline__ void fx_largest(const longlong2 (&q)[NV][E], uint32_t (&mx)[NV]) {
#pragma unroll
    for (int iv = 0; iv < NV; ++iv) {
        int a = 0;
#pragma unroll
        for (int m = 0; m < E; ++m)
            a = max(a, max(abs((int)(q[iv][m].x >> 32)), abs((int)(q[iv][m].y >> 32))));
        mx[iv] = (uint32_t)a + 8u;   // (and a margin for fx_split's carry at 2^61)
    }
}

// Shift every line right for a transform: by room, which takes S to 2^60.5, or
// by what the first MID points' sums need (largest values below 2^32 mx) where
// that is less; `room` keeps the difference for fx_refit.  S is taken over the
// high words' magnitudes (one unit of them covers what the low words add), of which a
// 32-bit sum takes eight: a component just above -2^60 has 2^28 (the shift floors), and
// sixteen of those would be 2^32, zero; after a transform, of values of at most 2^60.5 in
// modulus, a value's two are at most 2^29 + 2.  In units of 2^41 a line's sum stays
// below 2^32.
template <int MID, int NV, int E, typename Group>
__device__ __forceinline__ void fx_fit(longlong2 (&q)[NV][E], int (&ex)[NV], int (&room)[NV], const uint32_t (&mx)[NV],
                                       const Group &g) {
    static_assert(E <= 8, "per-thread sums");
    uint32_t s[NV];
#pragma unroll
    for (int iv = 0; iv < NV; ++iv) {
        uint32_t a[2] = {0u, 0u};   // four points each
#pragma unroll
        for (int m = 0; m < E; ++m)
            a[m / 4] += (uint32_t)abs((int)(q[iv][m].x >> 32)) + (uint32_t)abs((int)(q[iv][m].y >> 32));
        s[iv] = E > 4 ? (((a[0] >> 1) + (a[1] >> 1)) >> 8) + 2u : (a[0] >> 9) + 2u;
    }
    g.sum(s);
    int sh[NV];
#pragma unroll
    for (int iv = 0; iv < NV; ++iv) {
        // s 2^41 <= 2^60.5 2^room: s below 2^(19 + room), and the upper half octave once more
        const int n = __clz((int)s[iv]);
        const int need = max(0, 13 - n - ((s[iv] << n) < 0xB504F333u ? 1 : 0));
        sh[iv] = MID > 0 ? min(need, max(0, fx_growth(mx[iv], 31 - __clz(MID)))) : need;
        room[iv] = need - sh[iv];
    }
    fx_shift<NV, E>(q, ex, sh);
}

// the second look, with REST = N / (points combined so far) still to be summed
template <int REST, int NV, int E, typename Group>
__device__ __forceinline__ void fx_refit(longlong2 (&q)[NV][E], int (&ex)[NV], const int (&room)[NV], const Group &g) {
    uint32_t mx[NV];
    fx_largest<NV, E>(q, mx);
    g.max(mx);
    int sh[NV];
#pragma unroll
    for (int iv = 0; iv < NV; ++iv) sh[iv] = min(room[iv], max(0, fx_growth(mx[iv], 31 - __clz(REST))));
    fx_shift<NV, E>(q, ex, sh);
}

template <int MID, int NV, int E, typename Group>
__device__ __forceinline__ void fx_load(const double2 (&x)[NV][E], longlong2 (&q)[NV][E], int (&ex)[NV], int (&room)[NV],
                                        const Group &g) {
    uint32_t mx[NV];
#pragma unroll
    for (int iv = 0; iv < NV; ++iv) {
        uint32_t a = 0;
#pragma unroll
        for (int m = 0; m < E; ++m)
            a = max(a, max(fx_hi(x[iv][m].x) & 0x7fffffffu, fx_hi(x[iv][m].y) & 0x7fffffffu));
        mx[iv] = a;
    }
    g.max(mx);
#pragma unroll
    for (int iv = 0; iv < NV; ++iv) {
        const int em = (int)(mx[iv] >> 20);
        ex[iv] = em == 0x7ff ? kFxBad : em - 1023 - kFxTop;
#pragma unroll
        for (int m = 0; m < E; ++m) {
            q[iv][m].x = fx_from(x[iv][m].x, em);
            q[iv][m].y = fx_from(x[iv][m].y, em);
        }
        mx[iv] = ((((mx[iv] & 0xfffffu) | 0x100000u) + 1u) << (kFxTop - 52)) + 8u;   // as fx_largest
    }
    fx_fit<MID, NV, E>(q, ex, room, mx, g);
}

template <int NV, int E>
__device__ __forceinline__ void fx_store(const longlong2 (&q)[NV][E], const int (&ex)[NV], double2 (&x)[NV][E]) {
#pragma unroll
    for (int iv = 0; iv < NV; ++iv) {
        if (ex[iv] > -900 && ex[iv] < 900) {
#pragma unroll
            for (int m = 0; m < E; ++m) x[iv][m] = make_double2(fx_to(q[iv][m].x, ex[iv]), fx_to(q[iv][m].y, ex[iv]));
        } else {
#pragma unroll
            for (int m = 0; m < E; ++m)
                x[iv][m] = make_double2(fx_to_slow(q[iv][m].x, ex[iv]), fx_to_slow(q[iv][m].y, ex[iv]));
        }
    }
}

// The T consecutive threads of a line (T a power of two; all threads of the
// warps call).  T > 32: `scratch` holds 2 * (T / 32) * 2 words of this line;
// max and sum use halves of it, and fx_load always calls one after the other
// with the line's barrier in between, so a slot is never rewritten while read.
template <int T, typename Sync> struct FxLineGroup {
    uint32_t *scratch;
    int t;
    Sync sync;
    template <bool MAX, int NV> __device__ __forceinline__ void reduce(uint32_t (&m)[NV]) const {
        if constexpr (T < 32) {
#pragma unroll
            for (int o = T / 2; o > 0; o >>= 1)
#pragma unroll
                for (int i = 0; i < NV; ++i) {
                    const uint32_t other = __shfl_xor_sync(0xffffffffu, m[i], o);
                    m[i] = MAX ? ::max(m[i], other) : m[i] + other;
                }
        } else {
#pragma unroll
            for (int i = 0; i < NV; ++i)
                m[i] = MAX ? __reduce_max_sync(0xffffffffu, m[i]) : __reduce_add_sync(0xffffffffu, m[i]);
            if constexpr (T > 32) {
                constexpr int W = T / 32;
                uint32_t *s = scratch + (MAX ? 0 : 2 * W);
                if ((t & 31) == 0)
#pragma unroll
                    for (int i = 0; i < NV; ++i) s[i * W + (t >> 5)] = m[i];
                sync();
#pragma unroll
                for (int i = 0; i < NV; ++i) {
                    uint32_t a = 0;
#pragma unroll
                    for (int w = 0; w < W; ++w) a = MAX ? ::max(a, s[i * W + w]) : a + s[i * W + w];
                    m[i] = a;
                }
            }
        }
    }
    template <int NV> __device__ __forceinline__ void max(uint32_t (&m)[NV]) const { reduce<true>(m); }
    template <int NV> __device__ __forceinline__ void sum(uint32_t (&m)[NV]) const { reduce<false>(m); }
    static constexpr int kWords = T > 32 ? 4 * (T / 32) : 0;
};

// Column tiles: C columns (a power of two below 32) interleaved over the T * C
// threads of the block, thread = t * C + c; `scratch` holds 4 * (T * C / 32) * C words.
template <int C, int T> struct FxColGroup {
    static constexpr int W = C * T / 32;   // warps
    uint32_t *scratch;
    int tid;
    template <bool MAX, int NV> __device__ __forceinline__ void reduce(uint32_t (&m)[NV]) const {
#pragma unroll
        for (int o = 16; o >= C; o >>= 1)
#pragma unroll
            for (int i = 0; i < NV; ++i) {
                const uint32_t other = __shfl_xor_sync(0xffffffffu, m[i], o);
                m[i] = MAX ? ::max(m[i], other) : m[i] + other;
            }
        if constexpr (W > 1) {
            uint32_t *s = scratch + (MAX ? 0 : 2 * W * C);
            const int lane = tid & 31, c = tid % C;
            if (lane < C)
#pragma unroll
                for (int i = 0; i < NV; ++i) s[(i * W + (tid >> 5)) * C + c] = m[i];
            __syncthreads();
#pragma unroll
            for (int i = 0; i < NV; ++i) {
                uint32_t a = 0;
#pragma unroll
                for (int w = 0; w < W; ++w) a = MAX ? ::max(a, s[(i * W + w) * C + c]) : a + s[(i * W + w) * C + c];
                m[i] = a;
            }
        }
    }
    template <int NV> __device__ __forceinline__ void max(uint32_t (&m)[NV]) const { reduce<true>(m); }
    template <int NV> __device__ __forceinline__ void sum(uint32_t (&m)[NV]) const { reduce<false>(m); }
    static constexpr int kWords = W > 1 ? 4 * W * C : 0;
};

}  // namespace xsde
