// nvec.cuh -- n-vector arithmetic shared by the pyrochlore and the
// generic-lattice sweeps (Eq. 1 with n = 2, 3; Wolff's embedded cluster):
// explicitly rounded FP64 operations (no fused multiply-add, so results are
// those of a plain IEEE evaluation in the written order) or plain FP32, the
// per-sweep random axis, projections, normalisation and bond thresholds.
#pragma once

#include "pyro_internal.cuh"

namespace pyro {

template <typename T>
struct Ar;

template <>
struct Ar<double> {
    static __device__ __forceinline__ double mul(double a, double b) { return __dmul_rn(a, b); }
    static __device__ __forceinline__ double add(double a, double b) { return __dadd_rn(a, b); }
    static __device__ __forceinline__ double sub(double a, double b) { return __dadd_rn(a, -b); }
    static __device__ __forceinline__ double div(double a, double b) { return __ddiv_rn(a, b); }
    static __device__ __forceinline__ double sqrt_(double a) { return __dsqrt_rn(a); }
    static __device__ __forceinline__ double bond_p(double K2, double x) { return -expm1(-__dmul_rn(K2, x)); }
};

template <>
struct Ar<float> {
    static __device__ __forceinline__ float mul(float a, float b) { return a * b; }
    static __device__ __forceinline__ float add(float a, float b) { return a + b; }
    static __device__ __forceinline__ float sub(float a, float b) { return a - b; }
    static __device__ __forceinline__ float div(float a, float b) { return a / b; }
    static __device__ __forceinline__ float sqrt_(float a) { return sqrtf(a); }
    static __device__ __forceinline__ float bond_p(float K2, float x) { return -expm1f(-(K2 * x)); }
};

// Uniform unit vector from the (seed, sweep, tag) stream, FP64 with
// correctly rounded operations: rejection in the square, then n = 2:
// (u0, u1)/sqrt(s); n = 3: Marsaglia's (2 u0 sqrt(1-s), 2 u1 sqrt(1-s), 1-2s).
template <int NC>
__device__ __forceinline__ void unit_vector_dev(uint64_t seed, uint32_t sweep, uint32_t tag, uint64_t call_base,
                                                double r[3])
{
#pragma unroll 1
    for (int att = 0; att < MAX_AXIS_ATTEMPTS; ++att) {
        const uint4 w = philox_call(seed, sweep, tag, call_base + (uint64_t)att);
        const double u0 = (double)(int32_t)w.x * 4.656612873077392578125e-10;
        const double u1 = (double)(int32_t)w.y * 4.656612873077392578125e-10;
        const double s = __dadd_rn(__dmul_rn(u0, u0), __dmul_rn(u1, u1));
        if (s > 0.0 && s < 1.0) {
            if (NC == 2) {
                const double q = __dsqrt_rn(s);
                r[0] = __ddiv_rn(u0, q);
                r[1] = __ddiv_rn(u1, q);
                r[2] = 0.0;
            } else {
                const double t = __dsqrt_rn(__dadd_rn(1.0, -s));
                r[0] = __dmul_rn(__dmul_rn(2.0, u0), t);
                r[1] = __dmul_rn(__dmul_rn(2.0, u1), t);
                r[2] = __dadd_rn(1.0, -__dmul_rn(2.0, s));
            }
            return;
        }
    }
    r[0] = 1.0;
    r[1] = 0.0;
    r[2] = 0.0;
}

template <int NC, typename T>
__device__ __forceinline__ T project(const T *spins, int64_t N, int64_t i, const T r[3])
{
    using A = Ar<T>;
    T p = A::mul(spins[i], r[0]);
#pragma unroll
    for (int k = 1; k < NC; ++k) p = A::add(p, A::mul(spins[k * N + i], r[k]));
    return p;
}

// t <- t / sqrt(t . t), every operation correctly rounded: the bits of sqrt_
// and div, in fewer operations for the vectors a sweep meets, whose squared
// length q is within a few units in the last place of 1.  With M mantissa
// bits and d = bits(q) - bits(1), sqrt(1 + x) = 1 + x/2 - x^2/8 ..: for q d
// units of 2^-M above 1 (below: -d units of 2^-(M+1)) the correctly rounded
// root is floor(d / 2) units from 1, the x^2/8 term being far below half a
// unit for the d taken here; it only breaks the ties of odd d downwards.
//
// FP32: the quotients by s = 1 + e follow from one correctly rounded
// reciprocal r by Markstein's theorem (IBM J. Res. Dev. 34, 1990): with the
// faithful quotient g = fma(-e, t, t) (e^2 < 2^-27), fma(t - s g, r, g) is the
// correctly rounded t / s, the residual t - s g being exact in one fma (not
// for tiny t: those divide).
template <int NC>
__device__ __forceinline__ void normalise(float t[NC])
{
    float q = t[0] * t[0];
#pragma unroll
    for (int k = 1; k < NC; ++k) q = Ar<float>::add(q, Ar<float>::mul(t[k], t[k]));
    const int d = __float_as_int(q) - 0x3F800000;
    if (d > -1024 && d < 1024) {
        const int h = d >> 1;
        if (h == 0) return;  // the length rounds to 1
        const float s = __int_as_float(0x3F800000 + h), e = s - 1.0f, r = __frcp_rn(s);
        bool ok = true;
        float o[NC];
#pragma unroll
        for (int k = 0; k < NC; ++k) {
            const float g = __fmaf_rn(-e, t[k], t[k]);
            o[k] = __fmaf_rn(__fmaf_rn(-s, g, t[k]), r, g);
            ok &= fabsf(t[k]) > 1e-25f;
        }
        if (ok) {
#pragma unroll
            for (int k = 0; k < NC; ++k) t[k] = o[k];
            return;
        }
    }
    q = sqrtf(q);
#pragma unroll
    for (int k = 0; k < NC; ++k) t[k] = t[k] / q;
}

// FP64: by integer arithmetic, since roots and quotients took four fifths of
// the FP64 flip, whose two FP64 lanes a clock per SM bound it.  Quotient of
// t = T 2^e by s = 1 + h 2^-52, h > 0: T/s = T - T h / (2^52 + h); by
// s = 1 - k 2^-53: T/s = T + T k / (2^53 - k).  The fraction, rounded to
// nearest, is its quotient by the power of two alone, rounded, or one step
// from that (checked by the remainder); no quotient of two floats lies
// halfway.  A result past the binade of t, a zero and a denormal divide.
template <int NC>
__device__ __forceinline__ void normalise(double t[NC])
{
    using A = Ar<double>;
    double q = A::mul(t[0], t[0]);
#pragma unroll
    for (int k = 1; k < NC; ++k) q = A::add(q, A::mul(t[k], t[k]));
    constexpr long long ONE = 0x3FF0000000000000ll, FIELD = (1ll << 52) - 1;
    const long long d = __double_as_longlong(q) - ONE;
    if (d > -128 && d < 128) {
        const int h = (int)d >> 1;
        if (h == 0) return;  // the length rounds to 1
        const int m = abs(h), sh = h > 0 ? 52 : 53;
        const long long D = (1ll << sh) + h;
        bool ok = true;
        double o[NC];
#pragma unroll
        for (int k = 0; k < NC; ++k) {
            const long long b = __double_as_longlong(t[k]);
            const long long mant = b & FIELD;
            const long long n = (mant | (1ll << 52)) * m;  // below 2^59
            long long i = (n + (1ll << (sh - 1))) >> sh;
            const long long r2 = 2 * (n - i * D);
            if (h > 0) i -= r2 < -D;  // the divisor exceeds the power of two
            else i += r2 > D;
            const long long to = h > 0 ? mant - i : mant + i;
            ok &= to >= 0 && to <= FIELD && ((b >> 53) & 0x3FF) != 0;  // exponent field above 1
            o[k] = __longlong_as_double(h > 0 ? b - i : b + i);
        }
        if (ok) {
#pragma unroll
            for (int k = 0; k < NC; ++k) t[k] = o[k];
            return;
        }
    }
    q = A::sqrt_(q);
#pragma unroll
    for (int k = 0; k < NC; ++k) t[k] = A::div(t[k], q);
}

// Threshold of a bond with activation probability p: active iff its 32-bit
// uniform w < floor(p 2^32) (p = 1 gives 2^32).
__device__ __forceinline__ uint64_t prob_threshold(double p)
{
    if (!(p > 0.0)) return 0;
    const double t = floor(__dmul_rn(p, 4294967296.0));
    return t >= 4294967296.0 ? (1ull << 32) : (uint64_t)t;
}

__device__ __forceinline__ uint64_t prob_threshold(float p)
{
    if (!(p > 0.0f)) return 0;
    if (p >= 1.0f) return 1ull << 32;
    // p < 1: p 2^32 (exact, a power-of-two scaling) is below 2^32, and the
    // truncating conversion is the floor
    return __float2uint_rz(p * 4294967296.0f);
}

}  // namespace pyro
