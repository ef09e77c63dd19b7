// Counts of the values at which the library's short device functions differ from the
// functions they stand for (test_gpu_short_functions.py).
#include "fmg_strip_impl.cuh"
#include "fmg_warp.cuh"
#include "mlp_short.cuh"

using namespace fm;

// Out of line: the reference's own operations, not folded into the function under test.
static __device__ __noinline__ float ref_recip(float d) { return 1.0f / d; }
static __device__ __noinline__ double ref_div(double n, double d) { return n / d; }
static __device__ __noinline__ float ref_narrow(double x) { return (float)x; }
static __device__ __noinline__ double ref_widen(float x) { return (double)x; }

__device__ bool same(float a, float b) { return __float_as_uint(a) == __float_as_uint(b) || (isnan(a) && isnan(b)); }
__device__ bool same(double a, double b) {
    return __double_as_longlong(a) == __double_as_longlong(b) || (isnan(a) && isnan(b));
}
__device__ long long ulps(double a, double b) {
    const long long d = __double_as_longlong(a) - __double_as_longlong(b);
    return d < 0 ? -d : d;
}
__device__ uint64_t hash(uint64_t x) {   // splitmix64
    x += 0x9E3779B97F4A7C15ull;
    x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
    x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
    return x ^ (x >> 31);
}

enum { kGelu, kNormal, kWiden, kNarrow, kTwice, kStripRecip, kRecip, kDiagonal, kFace, kFaceFar, kCases };

// [0] values that differ, [1] values more than one ulp off.
template <int CASE>
__global__ void k_compare(uint64_t count, unsigned long long* bad) {
    unsigned long long n = 0, far = 0;
    for (uint64_t t = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; t < count; t += (uint64_t)gridDim.x * blockDim.x) {
        const uint32_t u = (uint32_t)t;
        const float f = __uint_as_float(u);
        const uint64_t h = hash(t), g = hash(t + (1ull << 40));
        if (CASE == kGelu) {   // each number beside another one
            const float o = __uint_as_float(u * 0x9E3779B1u + 12345u);
            n += gelu_bf16x2(f, o) != bf16x2_bits(gelu_f(f), gelu_f(o));
        }
        if (CASE == kNormal) {
            const uint32_t k = u & 0x7FFFFFu, o = (u * 0x9E3779B1u + 12345u) & 0x7FFFFFu;
            n += normal_bf16x2(k, o) != bf16x2_bits(normcdfinvf(word_uniform(k)), normcdfinvf(word_uniform(o)));
        }
        if (CASE == kWiden) n += !same(widen(f), ref_widen(f));
        if (CASE == kNarrow) {   // every FP32 number, the ties above it and their neighbours; and any FP64 number
            const long long b = __double_as_longlong(ref_widen(f));
            for (int q = 0; q < 4; ++q) {
                const double x = __longlong_as_double(b + (q ? 0x0FFFFFFFll + (q - 1) : 0));
                n += !same(narrow(x), ref_narrow(x));
            }
            const double x = __longlong_as_double((long long)h);
            n += !same(narrow(x), ref_narrow(x));
            const double y = __longlong_as_double((long long)((g & 0x800FFFFFFFFFFFFFull) | ((860 + (h >> 8) % 320) << 52)));
            n += !same(narrow(y), ref_narrow(y));   // exponents around both ends of FP32
        }
        if (CASE == kTwice) n += !same(twice(__longlong_as_double((long long)h)), __dmul_rn(2.0, __longlong_as_double((long long)h)));
        if (CASE == kStripRecip) {   // 2^-126 <= d < 2^126
            if (u >= 0x00800000u && u < 0x7E800000u) n += !same(strip_recip(f), ref_recip(f));
        }
        if (CASE == kRecip) n += !same(recip(f), ref_recip(f));
        if (CASE == kDiagonal) {   // exponents of both branches
            const double d = __longlong_as_double((long long)((h & 0x000FFFFFFFFFFFFFull) | ((uint64_t)(500 + (g >> 8) % 1046) << 52)));
            const double r = recip_set(d), e = ref_div(1.0, d);
            n += !same(r, e);
            far += ulps(r, e) > 1;
        }
        if (CASE == kFace || CASE == kFaceFar) {
            const int span = CASE == kFace ? 400 : 980;
            const double a = __longlong_as_double((long long)((h & 0x000FFFFFFFFFFFFFull) | ((uint64_t)(1023 - span / 2 + (g >> 8) % span) << 52)));
            const double b = __longlong_as_double((long long)((g & 0x000FFFFFFFFFFFFFull) | ((uint64_t)(1023 - span / 2 + (h >> 52) % span) << 52)));
            const double r = harmonic_mean(a, b), e = ref_div(__dmul_rn(__dmul_rn(2.0, a), b), __dadd_rn(a, b));
            n += !same(r, e);
            far += ulps(r, e) > 1;
        }
    }
    atomicAdd(bad, n);
    atomicAdd(bad + 1, far);
}

extern "C" int compare(int which, uint64_t count, unsigned long long* out) {
    unsigned long long* bad = nullptr;
    if (cudaMalloc((void**)&bad, 16) != cudaSuccess || cudaMemset(bad, 0, 16) != cudaSuccess) return 1;
    switch (which) {
        case kGelu: k_compare<kGelu><<<1216, 256>>>(count, bad); break;
        case kNormal: k_compare<kNormal><<<1216, 256>>>(count, bad); break;
        case kWiden: k_compare<kWiden><<<1216, 256>>>(count, bad); break;
        case kNarrow: k_compare<kNarrow><<<1216, 256>>>(count, bad); break;
        case kTwice: k_compare<kTwice><<<1216, 256>>>(count, bad); break;
        case kStripRecip: k_compare<kStripRecip><<<1216, 256>>>(count, bad); break;
        case kRecip: k_compare<kRecip><<<1216, 256>>>(count, bad); break;
        case kDiagonal: k_compare<kDiagonal><<<1216, 256>>>(count, bad); break;
        case kFace: k_compare<kFace><<<1216, 256>>>(count, bad); break;
        case kFaceFar: k_compare<kFaceFar><<<1216, 256>>>(count, bad); break;
        default: cudaFree(bad); return 2;
    }
    const int e = cudaMemcpy(out, bad, 16, cudaMemcpyDeviceToHost) != cudaSuccess;
    cudaFree(bad);
    return e;
}
