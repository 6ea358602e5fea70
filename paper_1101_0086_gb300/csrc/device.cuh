// Device building blocks of the MPA node transform and the split-step step:
// complex arithmetic, fixed-size DFTs in registers, the exact fixed-point
// dispersion phase, and a batched self-sorting (Stockham) FFT over shared
// memory.
//
// Fourier convention (text after Eq. (1)): forward F uses exp(+2 pi i kn/N)
// (sign S = +1), the inverse exp(-2 pi i kn/N) (S = -1, 1/N applied by the
// caller).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace mpa {

template <typename T> struct cx_of;
template <> struct cx_of<float> { typedef float2 type; };
template <> struct cx_of<double> { typedef double2 type; };
template <typename T> using cx = typename cx_of<T>::type;

__device__ __forceinline__ float2 mkc(float a, float b) { return make_float2(a, b); }
__device__ __forceinline__ double2 mkc(double a, double b) { return make_double2(a, b); }

template <class C> __device__ __forceinline__ C cadd(C a, C b) { return mkc(a.x + b.x, a.y + b.y); }
template <class C> __device__ __forceinline__ C csub(C a, C b) { return mkc(a.x - b.x, a.y - b.y); }

// FP32 complex add, subtract and real scaling as one packed f32x2
// instruction each (sm_100 and later): the same IEEE results as two scalar
// operations, half the issue slots.  MPA_F32X2=0 keeps the scalar forms.
#ifndef MPA_F32X2
#define MPA_F32X2 1
#endif
// packed real scalings (neutral in time, fewer instructions: on) and the
// cos/sin series of the phase in the two lanes of packed FMAs (slowed the
// forward column pass from 3.8 to 3.3-3.5 TB/s: off)
#ifndef MPA_F32X2_SCALE
#define MPA_F32X2_SCALE 1
#endif
#ifndef MPA_F32X2_POLY
#define MPA_F32X2_POLY 0
#endif
#if MPA_F32X2
__device__ __forceinline__ unsigned long long f2_bits(float2 a) {
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a.x), "f"(a.y));
    return r;
}
__device__ __forceinline__ float2 f2_from(unsigned long long v) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
template <> __device__ __forceinline__ float2 cadd<float2>(float2 a, float2 b) {
    unsigned long long r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(f2_bits(a)), "l"(f2_bits(b)));
    return f2_from(r);
}
template <> __device__ __forceinline__ float2 csub<float2>(float2 a, float2 b) {
    unsigned long long r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(f2_bits(a)), "l"(f2_bits(b)));
    return f2_from(r);
}
// lane-wise a * b and a * b + c
__device__ __forceinline__ float2 mul2(float2 a, float2 b) {
    unsigned long long r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(f2_bits(a)), "l"(f2_bits(b)));
    return f2_from(r);
}
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
    unsigned long long r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(f2_bits(a)), "l"(f2_bits(b)), "l"(f2_bits(c)));
    return f2_from(r);
}
#else
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return make_float2(__fmul_rn(a.x, b.x), __fmul_rn(a.y, b.y)); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
    return make_float2(fmaf(a.x, b.x, c.x), fmaf(a.y, b.y, c.y));
}
#endif
template <class C> __device__ __forceinline__ C cmul(C a, C b) {
    return mkc(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
template <class C> __device__ __forceinline__ C cconj(C a) { return mkc(a.x, -a.y); }
template <class C, class T> __device__ __forceinline__ C cscale(C a, T s) { return mkc(a.x * s, a.y * s); }
#if MPA_F32X2 && MPA_F32X2_SCALE
template <> __device__ __forceinline__ float2 cscale<float2, float>(float2 a, float s) { return mul2(a, make_float2(s, s)); }
#endif
// a * (S i)
template <int S, class C> __device__ __forceinline__ C mul_si(C a) {
    return S > 0 ? mkc(-a.y, a.x) : mkc(a.y, -a.x);
}
// a * exp(S i theta) given c = (cos, sin) of theta
template <int S, class C> __device__ __forceinline__ C mul_dir(C a, C w) {
    return S > 0 ? cmul(a, w) : cmul(a, cconj(w));
}

// ------------------------------------------------------------------ DFTs
// cos and sin of multiples of 2 pi/32 (closed forms: cos(pi/4) = sqrt(2)/2,
// cos(pi/8) = sqrt(2+sqrt(2))/2, sin(pi/8) = sqrt(2-sqrt(2))/2,
// cos(pi/16) = sqrt(2+sqrt(2+sqrt(2)))/2, sin(pi/16) = sqrt(2-sqrt(2+sqrt(2)))/2,
// cos(3pi/16) = sqrt(2+sqrt(2-sqrt(2)))/2, sin(3pi/16) = sqrt(2-sqrt(2-sqrt(2)))/2).
#define MPA_COS_PI_4 0.70710678118654752440
#define MPA_COS_PI_8 0.92387953251128675613
#define MPA_SIN_PI_8 0.38268343236508977173
#define MPA_COS_PI_16 0.98078528040323044913
#define MPA_SIN_PI_16 0.19509032201612826785
#define MPA_COS_3PI_16 0.83146961230254523708
#define MPA_SIN_3PI_16 0.55557023301960222474

// (cos, sin) of 2 pi m/32 for 0 < m < 16, m not a multiple of 4
template <int M32> struct Cs32 {
    static constexpr double c = (M32 == 1) ? MPA_COS_PI_16 : (M32 == 2) ? MPA_COS_PI_8 : (M32 == 3) ? MPA_COS_3PI_16
                              : (M32 == 5) ? MPA_SIN_3PI_16 : (M32 == 6) ? MPA_SIN_PI_8 : (M32 == 7) ? MPA_SIN_PI_16
                              : (M32 == 9) ? -MPA_SIN_PI_16 : (M32 == 10) ? -MPA_SIN_PI_8 : (M32 == 11) ? -MPA_SIN_3PI_16
                              : (M32 == 13) ? -MPA_COS_3PI_16 : (M32 == 14) ? -MPA_COS_PI_8 : -MPA_COS_PI_16;
    static constexpr double s = (M32 == 1) ? MPA_SIN_PI_16 : (M32 == 2) ? MPA_SIN_PI_8 : (M32 == 3) ? MPA_SIN_3PI_16
                              : (M32 == 5) ? MPA_COS_3PI_16 : (M32 == 6) ? MPA_COS_PI_8 : (M32 == 7) ? MPA_COS_PI_16
                              : (M32 == 9) ? MPA_COS_PI_16 : (M32 == 10) ? MPA_COS_PI_8 : (M32 == 11) ? MPA_COS_3PI_16
                              : (M32 == 13) ? MPA_SIN_3PI_16 : (M32 == 14) ? MPA_SIN_PI_8 : MPA_SIN_PI_16;
};

// v * exp(S 2 pi i K/R), R <= 32, 0 <= K < R/2 (compile-time special cases)
template <int R, int K, int S, class C> __device__ __forceinline__ C tw_const(C v) {
    typedef decltype(v.x) T;
    constexpr int M32 = K * (32 / R);
    if constexpr (M32 == 0) {
        return v;
    } else if constexpr (M32 == 8) {
        return mul_si<S>(v);
    } else if constexpr (M32 == 4 || M32 == 12) {
        const T c = (T)MPA_COS_PI_4;
        constexpr T re = (M32 == 4) ? T(1) : T(-1);
        // (re + S i) c
        return mkc(c * (re * v.x - T(S) * v.y), c * (re * v.y + T(S) * v.x));
    } else {
        const T cr = (T)Cs32<M32>::c, si = T(S) * (T)Cs32<M32>::s;
        return mkc(v.x * cr - v.y * si, v.x * si + v.y * cr);
    }
}

// Butterflies with a non-trivial constant twiddle (K/R not a multiple of 1/4)
// as fused multiply-adds: x0 = e + w o with the twiddle's products folded into
// the additions, x1 = 2 e - x0 (= e - w o): six operations instead of eight
// (two products, two fused products and four additions).  The difference from
// x1 = e - w o is one rounding of x0, of the size of the rounding of the
// product itself.  MPA_FMA_BFLY=0 keeps the plain form.
#ifndef MPA_FMA_BFLY
#define MPA_FMA_BFLY 1
#endif
__device__ __forceinline__ float ffma(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double ffma(double a, double b, double c) { return fma(a, b, c); }
template <int R, int K, int S, class C> __device__ __forceinline__ void bfly_tw(C& x0, C& x1, C e, C o) {
    typedef decltype(e.x) T;
    constexpr int M32 = K * (32 / R);
    T ax, ay;
    if constexpr (M32 == 4 || M32 == 12) {
        // w = c (re + S i), c = cos(pi/4): x0 = e + c (re o.x - S o.y, re o.y + S o.x)
        constexpr T re = (M32 == 4) ? T(1) : T(-1);
        const T c = (T)MPA_COS_PI_4;
        ax = ffma(c, re * o.x - T(S) * o.y, e.x);
        ay = ffma(c, re * o.y + T(S) * o.x, e.y);
    } else {
        const T cr = (T)Cs32<M32>::c, si = T(S) * (T)Cs32<M32>::s;
        ax = ffma(o.x, cr, ffma(-o.y, si, e.x));
        ay = ffma(o.x, si, ffma(o.y, cr, e.y));
    }
    x0 = mkc(ax, ay);
    x1 = mkc(ffma(T(2), e.x, -ax), ffma(T(2), e.y, -ay));
}

template <int R, int S, int K, class C> __device__ __forceinline__ void dft_combine(C* x, const C* e, const C* o) {
    if constexpr (K < R / 2) {
        constexpr int M32 = K * (32 / R);
        if constexpr (MPA_FMA_BFLY && M32 != 0 && M32 != 8) {
            bfly_tw<R, K, S>(x[K], x[K + R / 2], e[K], o[K]);
        } else {
            const C t = tw_const<R, K, S>(o[K]);
            x[K] = cadd(e[K], t);
            x[K + R / 2] = csub(e[K], t);
        }
        dft_combine<R, S, K + 1>(x, e, o);
    }
}

// In-register DFT of R points (power of two <= 32): X_k = sum_r x_r W^{rk},
// W = exp(S 2 pi i / R), by even/odd splitting.
template <int R, int S, class C> struct Dft {
    static __device__ __forceinline__ void run(C* x) {
        C e[R / 2], o[R / 2];
#pragma unroll
        for (int i = 0; i < R / 2; ++i) {
            e[i] = x[2 * i];
            o[i] = x[2 * i + 1];
        }
        Dft<R / 2, S, C>::run(e);
        Dft<R / 2, S, C>::run(o);
        dft_combine<R, S, 0>(x, e, o);
    }
};
template <int S, class C> struct Dft<1, S, C> {
    static __device__ __forceinline__ void run(C*) {}
};
template <int S, class C> struct Dft<2, S, C> {
    static __device__ __forceinline__ void run(C* x) {
        const C a = x[0], b = x[1];
        x[0] = cadd(a, b);
        x[1] = csub(a, b);
    }
};

// --------------------------------------------------------- exact phase
// Per-node (or per-linear-step) constants.  The dispersion phase
// beta(w_k, z) = w^2/2 I2 + w^3/6 I3 with w = 2 pi k'/T is, in turns,
//   theta = k'^2 a + k'^3 b,  a = pi I2 / T^2,  b = 2 pi^2 I3 / (3 T^3).
// The host stores a mod 1 and b mod 1 as 128-bit binary fractions (exact
// for the FP64 values of a and b); the device reduces theta mod 1 exactly in
// 64-bit integer arithmetic, so no FP64 arithmetic and no large-argument
// range reduction is needed however large beta grows.
struct NodeC {
    unsigned long long a_hi, a_lo, b_hi, b_lo;
    double pre;  // MPA: exp(int_{z0}^{z_j} G) = exp(-gamma (z_j - z0)); SS: linear-step gain
    double post; // MPA: sigma(z_j) dz / pre (weight of V_j in Eq. (6))
};

// The scan's per-node constants (FP32): the step of the phase coefficients
// from node j to node j + 1 (the phases of Eq. (6) are walked node by node,
// theta_{j+1} = theta_j + k'^2 da + k'^3 db), the real factors of NodeC in
// FP32, twice each (the operands of packed products), and the next node
// whose step differs from this one's (INT_MAX: none; the step is the same for
// all nodes of one fiber segment).
struct ScanNode {
    unsigned long long da_hi, da_lo, db_hi, db_lo;
    float pre[2], post[2];
    int next, pad[3];
};

// frac(k'^2 a + k'^3 b) as an unsigned Q0.64 number of turns (within 2 ulp).
// frac(k'^3 b) = frac(k' frac(k'^2 b)) since k'^3 b - k' frac(k'^2 b) is an
// integer multiple of k'.
__device__ __forceinline__ unsigned long long phase_q64(long long kp, unsigned long long a_hi, unsigned long long a_lo,
                                                        unsigned long long b_hi, unsigned long long b_lo) {
    const unsigned long long ak = (unsigned long long)(kp < 0 ? -kp : kp);
    const unsigned long long u = ak * ak;  // < 2^50 for N <= 2^25
    const unsigned long long ta = u * a_hi + __umul64hi(u, a_lo);
    const unsigned long long f_lo = u * b_lo;
    const unsigned long long f_hi = u * b_hi + __umul64hi(u, b_lo);
    unsigned long long tb = ak * f_hi + __umul64hi(ak, f_lo);
    if (kp < 0) tb = 0ull - tb;  // odd power of k'
    return ta + tb;
}
__device__ __forceinline__ unsigned long long phase_q64(long long kp, const NodeC& c) {
    return phase_q64(kp, c.a_hi, c.a_lo, c.b_hi, c.b_lo);
}

// exp(2 pi i theta) for theta a Q0.64 fraction of a turn: reinterpret as a
// signed fraction in [-1/2, 1/2) and evaluate sin/cos of pi * (2 theta).
template <typename T> __device__ __forceinline__ cx<T> expi_turns(unsigned long long th);
template <> __device__ __forceinline__ float2 expi_turns<float>(unsigned long long th) {
    const float x = __ll2float_rn((long long)th) * 1.0842021724855044e-19f;  // 2^-63
    float s, c;
    sincospif(x, &s, &c);
    return make_float2(c, s);
}
template <> __device__ __forceinline__ double2 expi_turns<double>(unsigned long long th) {
    const double x = __ll2double_rn((long long)th) * 1.0842021724855044e-19;  // 2^-63
    double s, c;
    sincospi(x, &s, &c);
    return make_double2(c, s);
}

// exp(2 pi i theta) for a Q0.64 turn fraction in FP32 without tables:
// split theta into the nearest quarter turn q and a residual angle
// x = 2 pi (theta - q/4), |x| <= pi/4, evaluate cos x and sin x by their
// Taylor series through x^8 and x^9 (truncation below 2.5e-8 and 1.8e-9),
// and rotate by i^q.
__device__ __forceinline__ float2 expi_turns_poly(unsigned long long th) {
    const unsigned long long q = (th + (1ull << 61)) >> 62;  // 0..3 (the sum wraps at 2^64)
    // residual in units of 2^-32 turn (|d| <= 2^29; the dropped bits are < 2^-32 turn)
    const int d = (int)((long long)(th - (q << 62)) >> 32);
    const float x = __int2float_rn(d) * 1.4629180792671596e-09f;  // 2 pi 2^-32
    const float x2 = x * x;
#if MPA_F32X2 && MPA_F32X2_POLY
    // the cos and sin series side by side in the two lanes of packed FMAs
    const float2 xx = make_float2(x2, x2);
    float2 p = fma2(xx, make_float2(2.4801587e-05f, 2.7557319e-06f), make_float2(-1.3888889e-03f, -1.9841270e-04f));
    p = fma2(p, xx, make_float2(4.1666668e-02f, 8.3333338e-03f));  // 1/4!, 1/5!
    p = fma2(p, xx, make_float2(-0.5f, -0.16666667f));
    const float c = fmaf(p.x, x2, 1.0f);
    const float sn = fmaf(p.y * x2, x, x);
#else
    float c = fmaf(x2, 2.4801587e-05f, -1.3888889e-03f);  // 1/8!, -1/6!
    c = fmaf(c, x2, 4.1666668e-02f);                     // 1/4!
    c = fmaf(c, x2, -0.5f);
    c = fmaf(c, x2, 1.0f);
    float sn = fmaf(x2, 2.7557319e-06f, -1.9841270e-04f);  // 1/9!, -1/7!
    sn = fmaf(sn, x2, 8.3333338e-03f);                     // 1/5!
    sn = fmaf(sn, x2, -0.16666667f);
    sn = fmaf(sn * x2, x, x);
#endif
    // multiply by i^q without branches: odd q swaps (c, s) -> (-s, c), q & 2 negates
    const bool odd = (q & 1) != 0;
    const float a = odd ? -sn : c, b = odd ? c : sn;
    const unsigned neg = (unsigned)(q & 2) << 30;
    return make_float2(__uint_as_float(__float_as_uint(a) ^ neg), __uint_as_float(__float_as_uint(b) ^ neg));
}

// expi_turns_poly of two phases at once: the same operations, the series of
// both phases in the two lanes of packed instructions, and the quarter turn
// taken from the bits of theta + 1/8 turn (bit 31 of its high word: half a
// turn on, a sign; bit 30: a quarter turn on, cos and sin swapped).
__device__ __forceinline__ void expi_turns_poly2(unsigned long long ta, unsigned long long tb, float2& ea, float2& eb) {
    const unsigned ha = (unsigned)(ta >> 32) + (1u << 29), hb = (unsigned)(tb >> 32) + (1u << 29);
    const int da = (int)(ha & 0x3FFFFFFFu) - (1 << 29), db = (int)(hb & 0x3FFFFFFFu) - (1 << 29);
    const float2 k = make_float2(1.4629180792671596e-09f, 1.4629180792671596e-09f);  // 2 pi 2^-32
    const float2 x = mul2(make_float2(__int2float_rn(da), __int2float_rn(db)), k), x2 = mul2(x, x);
    float2 c = fma2(x2, make_float2(2.4801587e-05f, 2.4801587e-05f), make_float2(-1.3888889e-03f, -1.3888889e-03f));
    c = fma2(c, x2, make_float2(4.1666668e-02f, 4.1666668e-02f));
    c = fma2(c, x2, make_float2(-0.5f, -0.5f));
    c = fma2(c, x2, make_float2(1.0f, 1.0f));
    float2 sn = fma2(x2, make_float2(2.7557319e-06f, 2.7557319e-06f), make_float2(-1.9841270e-04f, -1.9841270e-04f));
    sn = fma2(sn, x2, make_float2(8.3333338e-03f, 8.3333338e-03f));
    sn = fma2(sn, x2, make_float2(-0.16666667f, -0.16666667f));
    sn = fma2(mul2(sn, x2), x, x);
    const bool oa = (ha & 0x40000000u) != 0, ob = (hb & 0x40000000u) != 0;
    const unsigned na = ha & 0x80000000u, nb = hb & 0x80000000u;
    const float ax = oa ? -sn.x : c.x, ay = oa ? c.x : sn.x, bx = ob ? -sn.y : c.y, by = ob ? c.y : sn.y;
    ea = make_float2(__uint_as_float(__float_as_uint(ax) ^ na), __uint_as_float(__float_as_uint(ay) ^ na));
    eb = make_float2(__uint_as_float(__float_as_uint(bx) ^ nb), __uint_as_float(__float_as_uint(by) ^ nb));
}

// Element r of a run of phases: an even r evaluates the pair r, r + 1 and keeps
// the second for the next call.
template <int R> __device__ __forceinline__ float2 expi_pair(const unsigned long long (&th)[R], int r, float2& odd) {
    if (r & 1) return odd;
    float2 e;
    expi_turns_poly2(th[r], th[r + 1], e, odd);
    return e;
}

// (sin, cos) of a Kerr phase phi = sigma |A|^2 dz of the split-step.  These
// phases are small (about 1e-3 rad on the benchmark links), so for
// |phi| <= 1/16 the Taylor series of cos and sin are used: through phi^8 and
// phi^9 in FP64 (the first dropped terms are below 2.6e-19 and 2.3e-20
// relative) and through phi^4 and phi^5 in FP32 (below 8.3e-11 and 1.2e-11);
// larger phases take the library's sincos.  The FP64 series costs ten
// multiply-adds instead of a full-range evaluation on a GPU whose FP64
// rate is a small fraction of its FP32 rate.
__device__ __forceinline__ void sincos_kerr(double phi, double* s, double* c) {
    if (fabs(phi) <= 0.0625) {
        const double p2 = phi * phi;
        double cc = fma(p2, 1.0 / 40320.0, -1.0 / 720.0);
        cc = fma(cc, p2, 1.0 / 24.0);
        cc = fma(cc, p2, -0.5);
        *c = fma(cc, p2, 1.0);
        double ss = fma(p2, 1.0 / 362880.0, -1.0 / 5040.0);
        ss = fma(ss, p2, 1.0 / 120.0);
        ss = fma(ss, p2, -1.0 / 6.0);
        *s = fma(ss * p2, phi, phi);
    } else {
        sincos(phi, s, c);
    }
}
__device__ __forceinline__ void sincos_kerr(float phi, float* s, float* c) {
    if (fabsf(phi) <= 0.0625f) {
        const float p2 = phi * phi;
        *c = fmaf(fmaf(p2, 1.0f / 24.0f, -0.5f), p2, 1.0f);
        *s = fmaf(fmaf(p2, 1.0f / 120.0f, -1.0f / 6.0f) * p2, phi, phi);
    } else {
        sincosf(phi, s, c);
    }
}

// Exact phases theta(k'_0 + s D), s = -R/2 .. R/2-1, produced in s order
// by finite differences in Q0.64 arithmetic: theta is a cubic in s, so
// after four direct evaluations every further value costs three 64-bit
// additions (each direct value is within 2 ulp of 2^-64; over 32 values
// the cubic extrapolation keeps the error below 2^-48 turns).
struct PhaseRun {
    unsigned long long t0, t1, t2, t3, d1, d2, d3;
    int n;
    __device__ __forceinline__ PhaseRun(long long k_first, long long D, const NodeC& c) : n(0) {
        t0 = phase_q64(k_first, c);
        t1 = phase_q64(k_first + D, c);
        t2 = phase_q64(k_first + 2 * D, c);
        t3 = phase_q64(k_first + 3 * D, c);
        d1 = t3 - t2;
        d2 = t3 - 2 * t2 + t1;
        d3 = t3 - 3 * t2 + 3 * t1 - t0;
    }
    // value number n (n = 0, 1, 2, ...) of the progression
    __device__ __forceinline__ unsigned long long next() {
        const int m = n++;
        if (m == 0) return t0;
        if (m == 1) return t1;
        if (m == 2) return t2;
        if (m == 3) return t3;
        d2 += d3;
        d1 += d2;
        t3 += d1;
        return t3;
    }
};

// Phases of the R elements k'_s = k'_0 + s D, s = -R/2 .. R/2-1 of one
// butterfly by exact finite differences in Q0.64 arithmetic: theta is a
// cubic in s, so after four direct evaluations every further value costs
// three 64-bit additions (the direct values are within 2 ulp of 2^-64, so
// over 32 values the error stays below 2^-48 turns).  th[r] receives the phase
// of element r, where s = r for r < R/2 and s = r - R for r >= R/2.
template <int R>
__device__ __forceinline__ void phase_run(long long k0, long long D, const NodeC& c, unsigned long long (&th)[R]) {
    static_assert(R >= 4, "finite differences need four points");
    const long long ks = k0 - (long long)(R / 2) * D;
    unsigned long long t0 = phase_q64(ks, c), t1 = phase_q64(ks + D, c), t2 = phase_q64(ks + 2 * D, c),
                       t3 = phase_q64(ks + 3 * D, c);
    unsigned long long d1 = t3 - t2, d2 = t3 - 2 * t2 + t1, d3 = t3 - 3 * t2 + 3 * t1 - t0;
    th[R / 2] = t0;
    th[R / 2 + 1] = t1;
    th[R / 2 + 2] = t2;
    th[R / 2 + 3] = t3;
    unsigned long long t = t3;
#pragma unroll
    for (int s = -R / 2 + 4; s < R / 2; ++s) {
        d2 += d3;
        d1 += d2;
        t += d1;
        th[(s + R) % R] = t;
    }
}

// exp(2 pi i e / n) for an integer e (|e| small enough to be exact in T
// after reduction to [-n/2, n/2)), n a power of two given by log2.
template <typename T> __device__ __forceinline__ cx<T> expi_ratio(long long e, int log2n) {
    const long long n = 1ll << log2n;
    e &= (n - 1);
    if (e >= (n >> 1)) e -= n;
    T s, c;
    if constexpr (sizeof(T) == 4) {
        // |e| <= 2^24 here: a 32-bit conversion (a 64-bit one runs on the
        // FP64 pipe) and an exact scaling by the power of two 2^(1 - log2n)
        const float x = (float)(int)e * __int_as_float((128 - log2n) << 23);
        sincospif(x, &s, &c);
    } else {
        const double x = (double)e * 2.0 / (double)n;  // exact: |e| <= 2^52
        sincospi(x, &s, &c);
    }
    return mkc(c, s);
}

// ------------------------------------------------- dependent launches
// A kernel launched with launch_pdl (launch.h) may start while the kernel
// before it in its stream still runs: it prepares what needs no memory (its
// twiddle tables), then pdl_wait() returns once every earlier kernel of the
// stream has completed and its writes are visible.  pdl_go() lets the next
// kernel start in the same way as soon as every block of this one has called
// it.  Every global access comes after pdl_wait().  Both do nothing in a
// kernel launched without the attribute.  Kernels that a scan follows call
// pdl_go() at their end: a scan of a few blocks that starts while most SMs are
// still busy is packed onto the first free ones (2^14 x 801 nodes: 72 -> 108
// us).
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_go() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// ------------------------------------------------- thread groups
// A transform runs on the whole block (GRP = 0: threadIdx.x, __syncthreads)
// or on one of several NT-thread groups of the block (GRP = 1: the thread's
// index within its group, and named barrier 1 + group over the group's NT
// threads, so groups never wait on one another).
template <int GRP, int NT> __device__ __forceinline__ int gtid() {
    if constexpr (GRP == 0) return threadIdx.x;
    else return threadIdx.x & (NT - 1);
}
template <int GRP, int NT> __device__ __forceinline__ void gsync() {
    if constexpr (GRP == 0) {
        __syncthreads();
    } else {
        static_assert((NT & (NT - 1)) == 0 && NT % 32 == 0, "groups of whole warps, a power of two");
        asm volatile("bar.sync %0, %1;" ::"r"(1 + (int)(threadIdx.x / NT)), "n"(NT) : "memory");
    }
}

// ------------------------------------------------- shared-memory Stockham
// Padding of the shared-memory tile: one extra element per 2^PSH elements
// keeps every pass free of bank conflicts (PSH = log2 of the largest radix).
template <int PSH> __host__ __device__ __forceinline__ int phys(int i) { return i + (i >> PSH); }

// Tile layouts of G independent transforms of length L:
//   COL: element (l, g) at l*G + g  (a tile of G columns of an N2 x N1 matrix)
//   ROW: element (l, g) at g*L + l  (G contiguous rows)
enum { LAYOUT_COL = 0, LAYOUT_ROW = 1 };

template <int LAYOUT, int L, int G> __host__ __device__ __forceinline__ int eidx(int l, int g) {
    return LAYOUT == LAYOUT_COL ? l * G + g : g * L + l;
}

// The padded slot phys(eidx(l, g)) for l = lb + c written as base(lb, g) +
// off(c): with c a compile-time constant of an unrolled loop, off(c) folds
// into the shared-memory instruction's immediate offset, so each element
// costs no integer work.  The padding term i >> PSH is
//   COL, G >= 2^PSH: l (G >> PSH) + (g >> PSH)        (no condition)
//   COL, G <  2^PSH: l >> SH, SH = PSH - log2 G       (as g < G)
//   ROW, L >= 2^PSH: g (L >> PSH) + (l >> PSH)        (SH = PSH)
//   ROW, L <  2^PSH: g >> (PSH - log2 L)              (no condition)
// and the split is exact when (lb + c) >> SH = (lb >> SH) + (c >> SH) for
// every c the caller adds (strided() states the cases the passes use).
// Sites of the column layout that use the split form: bits 0-3 for
// transforms with the small radix last (SF false), bits 4-7 for those with
// it first (bit 0: first-pass scatter, 1: middle-pass reads, 2: middle-pass
// writes, 3: last-pass gather); the row layout uses it wherever it is
// exact.  Measured on the 2^20 link (split 2^12 x 2^8): the split row
// layout takes the row pass from 3223 to 3316 GB/s.  In the column layout
// it cuts instructions in both directions, but the forward column pass
// (radix 8 then 32, a 32-element gather per thread) fell from 3816 to
// 3417 GB/s while the inverse one (32 then 8) rose from 2906 to 2992 GB/s.
#ifndef MPA_SLOT_COL
#define MPA_SLOT_COL 0x0F
#endif
template <int LAYOUT, bool SF, int SITE> __host__ __device__ constexpr bool slot_site_on() {
    return LAYOUT != LAYOUT_COL || ((MPA_SLOT_COL >> (SITE + (SF ? 4 : 0))) & 1) != 0;
}

template <int LAYOUT, int L, int G, int PSH> struct Slot {
    __host__ __device__ static constexpr int lg(int x) { return x <= 1 ? 0 : 1 + lg(x / 2); }
    static constexpr int P2 = 1 << PSH;
    static constexpr bool COL = LAYOUT == LAYOUT_COL;
    // l enters through a shift by SH (else the split needs no condition)
    static constexpr bool LDEP = COL ? (G < P2) : (L >= P2);
    static constexpr int SH = COL ? (G < P2 ? PSH - lg(G) : 0) : (L >= P2 ? PSH : 0);
    static __host__ __device__ __forceinline__ int base(int lb, int g) {
        if constexpr (COL) {
            if constexpr (G >= P2) return lb * (G + (G >> PSH)) + g + (g >> PSH);
            else return lb * G + g + (lb >> SH);
        } else {
            if constexpr (L >= P2) return g * (L + (L >> PSH)) + lb + (lb >> PSH);
            else return g * L + (g >> (PSH - lg(L))) + lb;
        }
    }
    static __host__ __device__ constexpr int off(int c) {
        return COL ? (G >= P2 ? c * (G + (G >> PSH)) : c * G + (c >> SH)) : (L >= P2 ? c + (c >> PSH) : c);
    }
    // lb + r STRIDE with 0 <= lb < STRIDE, r < R: the shift splits if STRIDE
    // is a multiple of 2^SH or the whole range R STRIDE fits below 2^SH
    template <int STRIDE, int R> __host__ __device__ static constexpr bool strided() {
        return !LDEP || STRIDE % (1 << SH) == 0 || STRIDE * R <= (1 << SH);
    }
};

// Two-level table of W_L^e = exp(2 pi i e/L): hi[e >> SH] * lo[e & (2^SH-1)].
template <int L> struct TwDims {
    static constexpr int logL = (L >= 16384) ? 14 : (L >= 8192) ? 13 : (L >= 4096) ? 12 : (L >= 2048) ? 11
                              : (L >= 1024) ? 10 : (L >= 512) ? 9 : (L >= 256) ? 8 : (L >= 128) ? 7
                              : (L >= 64) ? 6 : (L >= 32) ? 5 : (L >= 16) ? 4 : (L >= 8) ? 3 : (L >= 4) ? 2 : 1;
    static constexpr int SH = (logL + 1) / 2;
    static constexpr int NLO = 1 << SH;
    static constexpr int NHI = L >> SH;
};

// FP64 transforms of up to 2048 points keep the whole table of W_L instead
// (hi[e], no product per lookup): FP64 instructions are the bound of the
// FP64 passes (1.7 a clock and SM), shared-memory reads are not.
// EX (FP32: the single-field tiles and the on-chip transforms of few nodes, up
// to 2048 points): factors within about half a unit in the last place, since
// passes of radix 4 to 16 apply more of them than radix-32 passes.  Split steps
// apply the same factors at every step, so a factor's error adds up from step to
// step where roundings of the data average out.  Error of 40 steps against FP64,
// 2^18 samples: factors hi lo (three roundings) 1.27e-5, EX 6.7e-6 (the large
// tiles' two radix-32 passes 1.14e-5); 2^10: 4.3e-6, 2.9e-6 (3.7e-6).  Up to 128
// points the whole table, one lookup a factor.  From 256 on a whole table costs
// up to 16 KB, bank conflicts and one CTA an SM less (us a step at 2^18 13.1 ->
// 16.1, at 2^22 67 -> 85), so the two-level one holds lo - 1 instead of lo and
// what FP32 leaves of hi = W_NHI^h (NHI <= 32): hi + (res + hi (lo - 1)), two
// additions more than hi lo (13.4 and 68 us; 2^20 22.5 -> 23.2).
template <typename T, int L, bool EX = false> struct Tw {
    static constexpr bool FULL = L >= 16 && (sizeof(T) == 8 ? L <= 2048 : EX && L <= 128);
    static constexpr bool COMP = EX && !FULL && L <= 2048;
    static_assert(!COMP || (sizeof(T) == 4 && TwDims<L>::NHI <= 32), "hi from the table of W_32");
    // entries in shared memory: [hi][lo][res of hi]
    static constexpr int N = FULL ? L : TwDims<L>::NLO + (COMP ? 2 : 1) * TwDims<L>::NHI;
};

// cos(2 pi m / 32) in FP32 and what FP32 leaves of it, from the closed forms
// above: selected in registers (a table in constant memory costs each launch
// cold, divergent reads: 0.2 us).
template <int K> __host__ __device__ __forceinline__ void w32_pick(int k, float& hi, float& res) {
    if constexpr (K < 8) {
        constexpr double c = K == 4 ? MPA_COS_PI_4 : Cs32<K>::c;
        constexpr float h = (float)c, r = (float)(c - (double)h);
        hi = k == K ? h : hi;
        res = k == K ? r : res;
        w32_pick<K + 1>(k, hi, res);
    }
}
__host__ __device__ __forceinline__ void w32_cos(int m, float& hi, float& res) {
    m &= 31;
    if (m > 16) m = 32 - m;
    const int k = m > 8 ? 16 - m : m;  // the first quarter turn
    hi = k == 0 ? 1.f : 0.f;
    res = 0.f;
    w32_pick<1>(k, hi, res);
    if (m > 8) {
        hi = -hi;
        res = -res;
    }
}
// W_32^m
__host__ __device__ __forceinline__ void w32(int m, float2& hi, float2& res) {
    w32_cos(m, hi.x, res.x);
    w32_cos(m + 24, hi.y, res.y);  // sin x = cos(x - turn / 4)
}

// Slot of entry e of the low twiddle table.  A row-pass warp looks up
// e = s j for 32 consecutive j and a power of two s; 8-byte entries sit in 16
// bank pairs, so in natural order the stride s = 4, 8, 16 lookups would
// collide 4- to 8-fold.  XOR-ing the entry's 16-block index into its low
// four bits spreads every such stride over distinct bank pairs.
template <int NLO> __host__ __device__ __forceinline__ int tw_lo_slot(int e) {
    if constexpr (NLO >= 32) return e ^ ((e >> 4) & 15);
    else return e;
}

template <typename T, int L, bool EX = false>
__device__ __forceinline__ void tw_init(cx<T>* hi, cx<T>* lo, int tid, int nt) {
    typedef TwDims<L> D;
    if constexpr (Tw<T, L, EX>::FULL && EX) {
        for (int m = tid; m < L; m += nt) hi[m] = expi_ratio<T>(m, D::logL);
    } else if constexpr (Tw<T, L, EX>::FULL) {
        // the first octant evaluated, the others its reflections (exact)
        for (int m = tid; m <= L / 8; m += nt) {
            const cx<T> w = expi_ratio<T>(m, D::logL);
            hi[m] = w;
            hi[L / 4 - m] = mkc(w.y, w.x);
            hi[L / 4 + m] = mkc(-w.y, w.x);
            hi[L / 2 - m] = mkc(-w.x, w.y);
            hi[L / 2 + m] = mkc(-w.x, -w.y);
            hi[3 * L / 4 - m] = mkc(-w.y, -w.x);
            hi[3 * L / 4 + m] = mkc(w.y, -w.x);
            if (m > 0) hi[L - m] = mkc(w.x, -w.y);
        }
    } else if constexpr (Tw<T, L, EX>::COMP) {
        for (int i = tid; i < D::NLO + D::NHI; i += nt) {
            if (i < D::NLO) {
                // cos x - 1 = -2 sin^2(x/2), sin x = 2 sin(x/2) cos(x/2)
                const cx<T> w = expi_ratio<T>(i, D::logL + 1);
                lo[tw_lo_slot<D::NLO>(i)] = mkc(T(-2) * w.y * w.y, T(2) * w.y * w.x);
            } else {
                const int m = i - D::NLO;
                w32(m * (32 / D::NHI), hi[m], lo[D::NLO + m]);
            }
        }
    } else {
        for (int i = tid; i < D::NLO + D::NHI; i += nt) {
            if (i < D::NLO) lo[tw_lo_slot<D::NLO>(i)] = expi_ratio<T>(i, D::logL);
            else hi[i - D::NLO] = expi_ratio<T>((long long)(i - D::NLO) << D::SH, D::logL);
        }
    }
}

template <typename T, int L, bool EX>
__device__ __forceinline__ cx<T> tw_get(const cx<T>* hi, const cx<T>* lo, int e) {
    typedef TwDims<L> D;
    if constexpr (Tw<T, L, EX>::FULL) return hi[e];
    else if constexpr (Tw<T, L, EX>::COMP) {
        const cx<T> h = hi[e >> D::SH], l = lo[tw_lo_slot<D::NLO>(e & (D::NLO - 1))], q = lo[D::NLO + (e >> D::SH)];
        return mkc(h.x + ffma(h.x, l.x, ffma(-h.y, l.y, q.x)), h.y + ffma(h.x, l.y, ffma(h.y, l.x, q.y)));
    } else if constexpr (D::NHI == 1) return lo[tw_lo_slot<D::NLO>(e)];
    else return cmul(hi[e >> D::SH], lo[tw_lo_slot<D::NLO>(e & (D::NLO - 1))]);
}

// exp(2 pi i theta) of a Q0.64 turn fraction in FP64 beside a full table of
// W_L (256 <= L <= 2048): theta = m / L + x / (2 pi) with |x| <= pi / L, and
// W_L^m (1 + (cos x - 1) + i sin x) by short Taylor series (the first dropped
// terms, x^8/40320 and x^7/5040, are below 1.3e-20 and 8.4e-18): 13 FP64
// instructions instead of a full-range sincospi, with the table's correctly
// rounded entry entering last.  x comes from the integer's upper 51 bits by
// the addition of 1.5 2^52 (exact), not by a conversion.
template <int L> __device__ __forceinline__ double2 expi_tab(unsigned long long th, const double2* tab) {
    constexpr int LG = TwDims<L>::logL, SH = 13 - LG;
    static_assert(Tw<double, L>::FULL && L >= 256, "a full table of at least 256 entries");
    const unsigned m = (unsigned)((th + (1ull << (63 - LG))) >> (64 - LG));  // nearest (wraps to 0)
    const long long d = (long long)(th - ((unsigned long long)m << (64 - LG))) >> SH;  // |d| <= 2^50
    const double x = (__longlong_as_double(0x4338000000000000ll + d) - 6755399441055744.0) *
                     (3.4061215800865545e-19 * (double)(1 << SH));  // 2 pi 2^-64 2^SH
    const double2 t = tab[m & (L - 1)];
    const double x2 = x * x;
    const double c = x2 * fma(x2, fma(x2, -1.0 / 720.0, 1.0 / 24.0), -0.5);
    const double s = fma(x * x2, fma(x2, 1.0 / 120.0, -1.0 / 6.0), x);
    return make_double2(fma(t.x, c, fma(-t.y, s, t.x)), fma(t.y, c, fma(t.x, s, t.y)));
}
// exp(2 pi i theta) in a kernel that holds the twiddle tables of W_L
template <typename T, int L> __device__ __forceinline__ cx<T> expi_at(unsigned long long th, const cx<T>* hi) {
    if constexpr (Tw<T, L>::FULL && L >= 256) return expi_tab<L>(th, hi);
    else return expi_turns<T>(th);
}

// v[r] *= W_L^{S r e1} for r = 1..R-1 (R <= 32): table lookups of
// w1, w2, w4 (combined into w1..w7) and w8, w16 (w24 = w8 w16), then
// w_r = w_{r mod 8} w_{8 floor(r/8)}, at most three products deep.
template <typename T, int L, int R, int S, bool EX>
__device__ __forceinline__ void twiddle_row(cx<T>* v, int e1, const cx<T>* hi, const cx<T>* lo) {
    typedef cx<T> C;
    if constexpr (Tw<T, L, EX>::FULL) {
#pragma unroll
        for (int r = 1; r < R; ++r) v[r] = mul_dir<S>(v[r], hi[r * e1]);
    } else {
        C w[8];
        w[1] = tw_get<T, L, EX>(hi, lo, e1);
        if constexpr (R > 2) w[2] = tw_get<T, L, EX>(hi, lo, 2 * e1);
        if constexpr (R > 2) w[3] = cmul(w[1], w[2]);
        if constexpr (R > 4) {
            w[4] = tw_get<T, L, EX>(hi, lo, 4 * e1);
            w[5] = cmul(w[1], w[4]);
            w[6] = cmul(w[2], w[4]);
            w[7] = cmul(w[3], w[4]);
        }
        C u[4];
        if constexpr (R > 8) u[1] = tw_get<T, L, EX>(hi, lo, 8 * e1);
        if constexpr (R > 16) {
            u[2] = tw_get<T, L, EX>(hi, lo, 16 * e1);
            u[3] = cmul(u[1], u[2]);
        }
#pragma unroll
        for (int r = 1; r < R; ++r) {
            const int a = r & 7, b = r >> 3;
            C t;
            if (b == 0) t = w[a];
            else if (a == 0) t = u[b];
            else t = cmul(w[a], u[b]);
            v[r] = mul_dir<S>(v[r], t);
        }
    }
}

// Direct twiddle table of a pass (FP32): W_{NS R}^{r k}, r < R, k < NS, laid
// out as [r / 2][k][r mod 2], so that a thread reads its R factors as R / 2
// 16-byte loads at compile-time offsets from its k; neighbouring threads hold
// neighbouring k (or the same: a broadcast), without bank conflicts.  Against
// twiddle_row it trades the lookups' products, 21 to 26 of them for R = 32, and
// their index arithmetic for loads (4.2 instructions an element and pass).
template <int NS, int R> __device__ __forceinline__ void dt_fill(float2* t, int tid, int nt) {
    constexpr int LG = TwDims<NS * R>::logL;
    static_assert((1 << LG) == NS * R, "a power of two");
    for (int i = tid; i < NS * R; i += nt) {
        const int k = (i >> 1) % NS, r = 2 * ((i >> 1) / NS) + (i & 1);
        t[i] = expi_ratio<float>((long long)r * k, LG);
    }
}
template <int NS, int R, int S> __device__ __forceinline__ void dt_row(float2* v, const float2* t, int k) {
    const float4* q = reinterpret_cast<const float4*>(t) + k;
#pragma unroll
    for (int h = 0; h < R / 2; ++h) {
        const float4 w = q[h * NS];
        if (h > 0) v[2 * h] = mul_dir<S>(v[2 * h], make_float2(w.x, w.y));
        v[2 * h + 1] = mul_dir<S>(v[2 * h + 1], make_float2(w.z, w.w));
    }
}

// One radix-R Stockham pass over the tile (in place, barrier-separated
// read and write phases).  Butterfly j of transform g reads elements
// j + r L/R, applies W_{NS R}^{S r (j mod NS)}, does the R-point DFT and
// writes to (j - j mod NS) R + j mod NS + r NS.
template <typename T, int L, int G, int NT, int R, int NS, int S, int LAYOUT, int PSH, bool SF, int GRP = 0, bool DT = false,
          bool EX = false>
__device__ __forceinline__ void stockham_pass(cx<T>* s, const cx<T>* hi, const cx<T>* lo, const cx<T>* dt = nullptr) {
    typedef cx<T> C;
    constexpr int NB = (L / R) * G;
    static_assert(NB % NT == 0, "butterflies must divide among threads");
    constexpr int Q = NB / NT;
    C v[Q][R];
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        const int b = gtid<GRP, NT>() + q * NT;
        const int j = LAYOUT == LAYOUT_COL ? b / G : b % (L / R);
        const int g = LAYOUT == LAYOUT_COL ? b % G : b / (L / R);
        typedef Slot<LAYOUT, L, G, PSH> SL;
        if constexpr (slot_site_on<LAYOUT, SF, 1>() && SL::template strided<L / R, R>()) {
            const C* sb = s + SL::base(j, g);
#pragma unroll
            for (int r = 0; r < R; ++r) v[q][r] = sb[SL::off(r * (L / R))];
        } else {
#pragma unroll
            for (int r = 0; r < R; ++r) v[q][r] = s[phys<PSH>(eidx<LAYOUT, L, G>(j + r * (L / R), g))];
        }
        if constexpr (DT) dt_row<NS, R, S>(v[q], dt, j & (NS - 1));
        else if constexpr (NS > 1) twiddle_row<T, L, R, S, EX>(v[q], (j & (NS - 1)) * (L / (NS * R)), hi, lo);
        Dft<R, S, C>::run(v[q]);
    }
    gsync<GRP, NT>();
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        const int b = gtid<GRP, NT>() + q * NT;
        const int j = LAYOUT == LAYOUT_COL ? b / G : b % (L / R);
        const int g = LAYOUT == LAYOUT_COL ? b % G : b / (L / R);
        const int k = j & (NS - 1);
        const int dst = (j - k) * R + k;
        typedef Slot<LAYOUT, L, G, PSH> SL;
        // dst = m NS R + k (k < NS): the offsets r NS stay below NS R
        if constexpr (slot_site_on<LAYOUT, SF, 2>() && SL::template strided<NS, R>()) {
            C* sb = s + SL::base(dst, g);
#pragma unroll
            for (int r = 0; r < R; ++r) sb[SL::off(r * NS)] = v[q][r];
        } else {
#pragma unroll
            for (int r = 0; r < R; ++r) s[phys<PSH>(eidx<LAYOUT, L, G>(dst + r * NS, g))] = v[q][r];
        }
    }
    gsync<GRP, NT>();
}

// Pass schedule of a length-L transform with radices RMAX and one smaller
// radix 2^b when log2 L is not a multiple of log2 RMAX.  SMALL_FIRST puts
// the small radix first (the transform then ends with an RMAX pass), else
// last.  Two transforms meet in registers when the last radix of the first
// equals the first radix of the second: the last pass leaves element
// j + r L/R of butterfly j in v[r], which is exactly what a first pass of
// the same radix reads.
template <int L, int RMAX> struct Sched {
    __host__ __device__ static constexpr int lg(int x) { return x <= 1 ? 0 : 1 + lg(x / 2); }
    static constexpr int LOGL = lg(L), LOGR = lg(RMAX);
    static constexpr int NFULL = LOGL / LOGR;
    static constexpr int SMALL = 1 << (LOGL % LOGR);  // 1 if none
    static constexpr int NP = NFULL + (SMALL > 1 ? 1 : 0);
    template <bool SF> __host__ __device__ static constexpr int radix(int p) {
        return SMALL == 1 ? RMAX : SF ? (p == 0 ? SMALL : RMAX) : (p == NP - 1 ? SMALL : RMAX);
    }
    template <bool SF> __host__ __device__ static constexpr int ns(int p) { return p == 0 ? 1 : ns<SF>(p - 1) * radix<SF>(p - 1); }
};

template <typename T, int L, int G, int NT, int RMAX, int S, int LAYOUT, int PSH, bool SF, int P, int NP, int GRP, bool DT, bool EX>
__device__ __forceinline__ void mid_passes(cx<T>* s, const cx<T>* hi, const cx<T>* lo, const cx<T>* dt) {
    if constexpr (P < NP - 1) {
        typedef Sched<L, RMAX> SC;
        stockham_pass<T, L, G, NT, SC::template radix<SF>(P), SC::template ns<SF>(P), S, LAYOUT, PSH, SF, GRP,
                      DT && P == 1, EX>(s, hi, lo, dt);
        mid_passes<T, L, G, NT, RMAX, S, LAYOUT, PSH, SF, P + 1, NP, GRP, DT, EX>(s, hi, lo, dt);
    }
}

// Butterfly b of a radix-R pass -> (j, g).
template <int LAYOUT, int L, int G, int R> __host__ __device__ __forceinline__ void bmap(int b, int& j, int& g) {
    if constexpr (LAYOUT == LAYOUT_COL) {
        j = b / G;
        g = b % G;
    } else {
        j = b % (L / R);
        g = b / (L / R);
    }
}

// A whole transform with register endpoints.  vin[q][r] holds input element
// j + r L/R0 of butterfly b = tid + q NT (R0 = first radix), vout[q][r]
// receives output element j + r L/RL (RL = last radix).  Shared memory is
// used by the middle passes only; the transform ends with a barrier so the
// caller may reuse `s`.  GRP as for gtid/gsync.  USE_DT: the second pass reads
// its twiddles from a direct table of DTN entries (where that is at most 1024;
// 0: none) that the caller fills with dt_init and passes to run.  EX: the
// factors of Tw's EX tables.
template <typename T, int L, int G, int NT, int RMAX, int S, int LAYOUT, int PSH, bool SF, int GRP = 0, bool USE_DT = false,
          bool EX = false>
struct Xform {
    typedef Sched<L, RMAX> SC;
    typedef cx<T> C;
    static constexpr int NP = SC::NP;
    static constexpr int R0 = SC::template radix<SF>(0);
    static constexpr int RL = SC::template radix<SF>(NP - 1);
    static constexpr int Q0 = (L / R0) * G / NT;
    static constexpr int QL = (L / RL) * G / NT;
    static_assert((L / R0) * G % NT == 0 && (L / RL) * G % NT == 0, "butterflies must divide among threads");
    static constexpr int NS1 = NP > 1 ? SC::template ns<SF>(NP > 1 ? 1 : 0) : 1;
    static constexpr int R1 = NP > 1 ? SC::template radix<SF>(NP > 1 ? 1 : 0) : 1;
    static constexpr int DTN = USE_DT && NP > 1 && NS1 * R1 <= 1024 ? NS1 * R1 : 0;
    static constexpr bool DT = DTN > 0;
    static __device__ __forceinline__ void dt_init(C* t, int tid, int nt) {
        if constexpr (DT) dt_fill<NS1, R1>(t, tid, nt);
    }

    struct NoHook {
        __device__ __forceinline__ void operator()() const {}
    };
    static __device__ __forceinline__ void run(C (&vin)[Q0][R0], C (&vout)[QL][RL], C* s, const C* hi, const C* lo,
                                               const C* dt = nullptr) {
        run(vin, vout, s, hi, lo, dt, NoHook());
    }
    // hook() runs once the first pass has left the registers for shared
    // memory (after its barrier; at the start for a single-pass transform),
    // where the caller's own work needs the fewest registers.
    template <class Hook>
    static __device__ __forceinline__ void run(C (&vin)[Q0][R0], C (&vout)[QL][RL], C* s, const C* hi, const C* lo,
                                               const C* dt, Hook&& hook) {
        if constexpr (NP == 1) {
            hook();
#pragma unroll
            for (int q = 0; q < Q0; ++q) {
                Dft<R0, S, C>::run(vin[q]);
#pragma unroll
                for (int r = 0; r < R0; ++r) vout[q][r] = vin[q][r];
            }
        } else {
            // first pass: DFT of the register inputs (NS = 1), scatter to j R0 + r
#pragma unroll
            for (int q = 0; q < Q0; ++q) {
                int j, g;
                bmap<LAYOUT, L, G, R0>(gtid<GRP, NT>() + q * NT, j, g);
                Dft<R0, S, C>::run(vin[q]);
                // j R0 + r, r < R0: the shift always splits (j R0 is a multiple
                // of 2^SH, or R0 divides 2^SH and r < R0 adds no carry)
                typedef Slot<LAYOUT, L, G, PSH> SL;
                if constexpr (slot_site_on<LAYOUT, SF, 0>()) {
                    C* sb = s + SL::base(j * R0, g);
#pragma unroll
                    for (int r = 0; r < R0; ++r) sb[SL::off(r)] = vin[q][r];
                } else {
#pragma unroll
                    for (int r = 0; r < R0; ++r) s[phys<PSH>(eidx<LAYOUT, L, G>(j * R0 + r, g))] = vin[q][r];
                }
            }
            gsync<GRP, NT>();
            hook();
            mid_passes<T, L, G, NT, RMAX, S, LAYOUT, PSH, SF, 1, NP, GRP, DT, EX>(s, hi, lo, dt);
            // last pass (NS = L/RL, so k = j): gather j + r L/RL, twiddle W_L^{S r j}, DFT
#pragma unroll
            for (int q = 0; q < QL; ++q) {
                int j, g;
                bmap<LAYOUT, L, G, RL>(gtid<GRP, NT>() + q * NT, j, g);
                typedef Slot<LAYOUT, L, G, PSH> SL;
                if constexpr (slot_site_on<LAYOUT, SF, 3>() && SL::template strided<L / RL, RL>()) {
                    const C* sb = s + SL::base(j, g);
#pragma unroll
                    for (int r = 0; r < RL; ++r) vout[q][r] = sb[SL::off(r * (L / RL))];
                } else {
#pragma unroll
                    for (int r = 0; r < RL; ++r) vout[q][r] = s[phys<PSH>(eidx<LAYOUT, L, G>(j + r * (L / RL), g))];
                }
                if constexpr (DT && NP == 2) dt_row<NS1, R1, S>(vout[q], dt, j);
                else twiddle_row<T, L, RL, S, EX>(vout[q], j, hi, lo);
                Dft<RL, S, C>::run(vout[q]);
            }
            gsync<GRP, NT>();
        }
    }
};

// Precision-dependent tiling: elements per thread E, largest radix, the
// padding shift, the minimum column-tile width (64-byte row segments) and
// the target tile size in elements.
// KIND 0 = column pass, 1 = row pass (tuned separately).
#ifndef MPA_KC_E
#define MPA_KC_E 32
#endif
#ifndef MPA_KC_TE
#define MPA_KC_TE 8192
#endif
#ifndef MPA_KR_E
#define MPA_KR_E 32
#endif
#ifndef MPA_KR_TE
#define MPA_KR_TE 8192
#endif
#ifndef MPA_KCW_E
#define MPA_KCW_E 16
#endif
// KIND 2 = wavefront column pass.
// KIND 3, 4 = both passes over a single field (transforms, split steps), whose
// few large tiles would leave SMs idle: fine and medium tiles.
template <typename T, int KIND = 0> struct Tiling;
template <> struct Tiling<float, 3> {
    static constexpr int E = 8, RMAX = 8, PSH = 3, CMIN = 4, TE = 1024;
};
template <> struct Tiling<float, 4> {
    static constexpr int E = 16, RMAX = 16, PSH = 4, CMIN = 4, TE = 1024;
};
template <> struct Tiling<double, 3> {
    static constexpr int E = 4, RMAX = 4, PSH = 2, CMIN = 1, TE = 256;
};
template <> struct Tiling<double, 4> {
    static constexpr int E = 8, RMAX = 8, PSH = 3, CMIN = 1, TE = 256;
};
// KIND 5 = on-chip node transforms of few nodes (kn_fine).
template <> struct Tiling<float, 5> {
    static constexpr int E = 16, RMAX = 16, PSH = 4;
};
// The tiles of a single-field pass of length L over `elems` elements: 0 the
// large tiles of the MPA passes, 1 fine, 2 medium.  Measured, us a split step
// (both passes), large / medium / fine.  FP32 (launches and latency, then
// warps to hide it): 2^12 30.7 / 16.0 / 11.9, 2^18 26.4 / 18.2 / 13.8, 2^19
// 26.3 / 18.0 / 18.1, 2^20 28.8 / 23.2 / 28.6, 2^22 74.3 / 71.0 / 97.4.  FP64
// (an FP64 instruction occupies one of an SM's four schedulers for 76 clocks,
// so small fields need their elements spread over all of them): 2^12 244 / 71
// / 46, 2^16 228 / 69 / 42, 2^17 221 / 70.6 / 68.4, 2^18 230 / 123 / 128, 2^20
// 443 / 421 / 425, 2^22 1709 / 1691 / 1835.  Rows above 2048 points keep the
// large tiles (one or a few rows each), and so do FP32 columns of 2048 points
// beyond 2^22 (HBM-bound, 64-byte row segments against the medium tiles' 32:
// a 2^24 step 277 against 299 us).
template <typename T> __host__ __device__ constexpr int field_tiles(int L, long long elems) {
    return L > 2048 || (sizeof(T) == 4 && L == 2048 && elems > (1ll << 22)) ? 0
         : elems <= (sizeof(T) == 8 ? 1ll << 16 : 1ll << 18)               ? 1
                                                                           : 2;
}
#ifndef MPA_RMAX32
#define MPA_RMAX32 32
#endif
template <int KIND> struct Tiling<float, KIND> {
    // radix-32 passes (one smem exchange for a 1024-point transform) where a
    // thread holds 32 elements; the wavefront pass (16 per thread) uses 16
    static constexpr int E = KIND == 0 ? MPA_KC_E : KIND == 1 ? MPA_KR_E : MPA_KCW_E;
    static constexpr int RMAX = E >= 32 ? MPA_RMAX32 : 16, PSH = RMAX == 32 ? 5 : 4, CMIN = 8;
    static constexpr int TE = KIND == 1 ? MPA_KR_TE : MPA_KC_TE;
};
template <int KIND> struct Tiling<double, KIND> {
    // radix-16 passes: 1024 points in 29 FP64 instructions an element (16 x
    // 16 x 4), 41 with radix 8 (8 x 8 x 8 x 2 and two-level twiddle tables)
    static constexpr int E = 16, RMAX = 16, PSH = 4, CMIN = 4, TE = 4096;
};

}  // namespace mpa
