// Column-strip wavefront smoother of the level-wise schedule: the call that
// fmg.cu makes (StripCall, strip_launch) and the device helpers both share.
#pragma once

#include "common.cuh"

namespace fm {

// A product and a sum the compiler may not fuse with what surrounds them.
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float add_rn(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double add_rn(double a, double b) { return __dadd_rn(a, b); }

// FP64 -> FP32 (round to nearest even) and back in integers.  The conversion
// instructions run in the FP64 pipe (two lanes a clock and SM), which bounds
// every kernel that refines: ten and seven integer operations cost a sixth of
// one conversion.  What is not a normal number of both types goes by integers
// too: a conversion there would take its turn in the pipe in every warp,
// predicated off or not.
static __device__ __noinline__ float narrow_rare(unsigned hi, unsigned lo) {
    const unsigned e = (hi >> 20) & 0x7ffu;
    const unsigned long long m = ((unsigned long long)((hi & 0xfffffu) | 0x100000u) << 32) | lo;
    unsigned r = 0;
    if (e >= 1151u) {
        if (e == 2047u && (m & 0xfffffffffffffull)) return __uint_as_float(0x7fffffffu);
        r = 0x7f800000u;
    } else if (e >= 873u) {   // a subnormal: units of 2^-149
        const unsigned shift = 926u - e;
        r = (unsigned)((m + ((1ull << (shift - 1)) - 1) + ((m >> shift) & 1)) >> shift);
    }
    return __uint_as_float(r | (hi & 0x80000000u));
}
__device__ __forceinline__ float narrow(double x) {
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    if (((hi >> 20) & 0x7ffu) - 897u > 253u) return narrow_rare(hi, lo);
    const unsigned long long t = (((unsigned long long)hi << 32) | lo) + (0x0fffffffu + ((lo >> 29) & 1u));
    const unsigned u = __funnelshift_l((unsigned)t, (unsigned)(t >> 32), 3) - 0xc0000000u;
    return __uint_as_float((u & 0x7fffffffu) | (hi & 0x80000000u));
}
static __device__ __noinline__ double widen_rare(unsigned u) {
    const unsigned m = u & 0x7fffffffu, sign = u & 0x80000000u;
    if (m == 0) return __hiloint2double((int)sign, 0);
    if (m >= 0x7f800000u) return __hiloint2double((int)(sign | 0x7ff00000u | ((m & 0x7fffffu) >> 3)), (int)(u << 29));
    const unsigned shift = __clz(m) - 8, f = (m << shift) & 0x7fffffu;
    return __hiloint2double((int)(sign | ((897u - shift) << 20) | (f >> 3)), (int)(f << 29));
}
__device__ __forceinline__ double widen(float x) {
    const unsigned u = __float_as_uint(x), m = u & 0x7fffffffu;
    if (m - 0x00800000u >= 0x7f000000u) return widen_rare(u);
    return __hiloint2double((int)((u & 0x80000000u) | ((m >> 3) + 0x38000000u)), (int)(u << 29));
}
__device__ __forceinline__ double widen(double x) { return x; }
template <typename T>
__device__ __forceinline__ T rounded(float x) {
    return (T)x;
}
template <typename T>
__device__ __forceinline__ T rounded(double x) {
    if constexpr (sizeof(T) == 4) return narrow(x);
    else return x;
}

// 2 x, in FP64 by the exponent (outside the FP64 pipe, as narrow and widen).
static __device__ __noinline__ double twice_rare(double x) { return 2.0 * x; }
__device__ __forceinline__ float twice(float x) { return 2.0f * x; }
__device__ __forceinline__ double twice(double x) {
    const unsigned hi = (unsigned)__double2hiint(x);
    if (((hi >> 20) & 0x7ffu) - 1u > 2044u) return twice_rare(x);
    return __hiloint2double((int)(hi + 0x100000u), __double2loint(x));
}

// 1 / d to 2^-44 outside the FP64 pipe, for positive d with an exponent of at most
// 480 either way (recip_fits): the upper 24 bits of the mantissa by rcp.approx,
// whose remainder against all 47 bits, in FP32, gives the rest; joined in integers.
__device__ __forceinline__ bool recip_fits(double d) {
    return (unsigned)__double2hiint(d) - ((1023u - 480u) << 20) < (960u << 20);
}
__device__ __forceinline__ double recip_start(double d) {
    const unsigned hi = (unsigned)__double2hiint(d), lo = (unsigned)__double2loint(d);
    const float dh = __uint_as_float(0x3f800000u | ((hi << 3) & 0x7fffffu) | (lo >> 29));   // 1 .. 2
    const float dl = __uint_as_float(0x34000000u | ((lo >> 6) & 0x7fffffu)) - 0x1p-23f;
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(dh));
    const float e = fmaf(-dl, r, fmaf(-dh, r, 1.0f));
    const int c = __float2int_rn(r * fmaf(e, e, e) * 0x1p52f);   // below 2^30
    // r is 1/2 .. 1, whose FP64 units are 2^-53 (c is not positive where r is 1)
    const long long bits = ((long long)__float_as_uint(r) << 29) + (896LL << 52) + ((long long)c << 1);
    return __longlong_as_double(bits - ((long long)((int)(hi >> 20) - 1023) << 52));
}

// 1 / d, in two operations of the FP64 pipe (an IEEE division is nine).
static __device__ __noinline__ double recip_rare(double d) { return 1.0 / d; }
__device__ __forceinline__ float recip_set(float d) { return 1.0f / d; }
__device__ __forceinline__ double recip_set(double d) {
    if (!recip_fits(d)) return recip_rare(d);
    const double r = recip_start(d);
    return fma(r, fma(-d, r, 1.0), r);
}

// Harmonic mean 2ab / (a + b) of two coefficients, the face between them.
// FP64: the divide of the FP64 pipe (a 58th of the FP32 rate) bounds the
// set-up of every operator, so the quotient takes three operations instead of
// nine: the start above, n r, and its correction by its own remainder
// (Markstein), correct to about 2^-88 before the last rounding: the IEEE quotient but
// for one in some 2^34 (2.1e9 random pairs, and as many reciprocals, met none).
// Measured against a start by rcp.approx.f64 and a Newton step in the pipe (two
// operations more, and IEEE 1 / D): 5304 FP64 samples of 64 x 64 7.79 -> 7.35 ms,
// 1000 mixed samples of 256 x 256 25.7 -> 25.2.
// (Any d: scaled where its reciprocal is no normal number.  By Newton steps, since a
// division in the callee takes registers from its callers: the 16 x 16 mixed kernel
// was 2% slower with one.)
static __device__ __noinline__ double quotient_rare(double n, double d) {
    const int e = (__double2hiint(d) >> 20) & 0x7ff;
    const double s = e > 2023 ? 0x1p-64 : e < 24 ? 0x1p128 : 1.0;
    n *= s;
    d *= s;
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(d));
    r = fma(r, fma(-d, r, 1.0), r);
    r = fma(r, fma(-d, r, 1.0), r);
    const double q = n * r;
    return fma(fma(-d, q, n), r, q);
}
__device__ __forceinline__ float harmonic_mean(float a, float b) { return 2.0f * a * b / (a + b); }
__device__ __forceinline__ double harmonic_mean(double a, double b) {
    const double n = twice(a) * b, d = a + b;
    if (!recip_fits(d)) return quotient_rare(n, d);
    const double r = recip_start(d), q = n * r;
    return fma(fma(-d, q, n), r, q);
}

// Geometric mean of four positive coefficients.  FP64: two square roots (25
// operations of the FP64 pipe, against 157 for four logarithms and an
// exponential) where no product leaves the range, else by logarithms.
__device__ __forceinline__ float geometric_mean4(float a, float b, float c, float d) {
    return expf(0.25f * (logf(a) + logf(b) + logf(c) + logf(d)));
}
__device__ __forceinline__ double geometric_mean4(double a, double b, double c, double d) {
    const double p = a * b, q = c * d;
    if (p > 1e-140 && p < 1e140 && q > 1e-140 && q < 1e140) return sqrt(sqrt(p * q));
    return exp(0.25 * (log(a) + log(b) + log(c) + log(d)));
}

// -x where flip, by the sign bit (a negation is an addition of the FP64 pipe).
__device__ __forceinline__ float flip_if(bool flip, float x) {
    return __uint_as_float(__float_as_uint(x) ^ (flip ? 0x80000000u : 0u));
}
__device__ __forceinline__ double flip_if(bool flip, double x) {
    return __hiloint2double((int)((unsigned)__double2hiint(x) ^ (flip ? 0x80000000u : 0u)), __double2loint(x));
}

// The bilinear cell-centred prolongation (9, 3, 3, 1) / 16 of four coarse
// values: own cell, its x neighbour, its y neighbour, the diagonal one.  The
// roundings are spelled out, so every kernel that prolongs rounds the same
// way (left to the compiler's contraction, one of the strip kernels did not).
template <typename U>
__device__ __forceinline__ U prolong_vals(U own, U nx, U ny, U nxy) {
    return mul_rn(add_rn(fma(U(3), ny, fma(U(9), own, mul_rn(U(3), nx))), nxy), U(0.0625));
}

// Restriction after red-black sweeps in FP64: a sweep ends on black, whose cells
// then satisfy their equations to rounding, so their residuals are taken as zero
// and half the residuals, three FP64 operations a cell, are never formed.  (In
// FP32 the rounding is not far below what the correction still has to resolve,
// and the pipe is not the bound: all four.)
template <typename T>
constexpr bool kRedOnly = sizeof(T) == 8;

// One smoothing call of the strip shape on grid n x n: hs half-sweeps
// (red first) on p_in -> p_out.
template <typename T>
struct StripCall {
    int n = 0;
    size_t S = 0;                      // samples of the batch
    int hs = 0;                        // half-sweeps: 2 nsweeps, or post- and pre-smoothing in one (strip_merges)
    bool fuse = false;                 // also the residual's restriction into bc
    const T *b = nullptr, *Te = nullptr, *Tn = nullptr, *D = nullptr;
    const T* rD = nullptr;             // 1 / D (FP64 only: the FP32 kernels form it)
    const T* p_in = nullptr;           // null: a zero iterate
    T* p_out = nullptr;
    const int32_t* active = nullptr;
    const T* ec = nullptr;             // coarse correction added to the iterate on load
    T *bc = nullptr, *pc = nullptr;    // fuse: coarse rhs, and (nullable) the coarse iterate to zero
    const int32_t* order = nullptr;    // list of the samples still iterating
    size_t busy = 0;                   // their count where the host knows it (0: all)
    const int32_t* dcount = nullptr;   // their count on the device (refinement loops inside a graph)
    int ns = 0;                        // Dirichlet north / south edges
};

template <typename T>
void strip_launch(fm_ctx* ctx, const StripCall<T>& c, cudaStream_t st);

// The strip shape runs 1 or 2 sweeps on even grids of at least 16 cells.
inline bool strip_fits(int n, int nu1, int nu2) {
    return n >= 16 && n % 2 == 0 && nu1 >= 1 && nu1 <= 2 && nu2 >= 1 && nu2 <= 2;
}

// The post-smoothing of one V-cycle and the pre-smoothing of the next run as
// one call of 2 (nu1 + nu2) half-sweeps (FP32, as many sweeps on both sides).
template <typename T>
inline bool strip_merges(int nu1, int nu2) {
    return sizeof(T) == 4 && nu1 == nu2;
}

// Kernel attributes on the current device, and occupancies.
template <typename T>
void strip_init(int sms);

}  // namespace fm
