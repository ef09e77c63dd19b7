// FP64 KL field synthesis (Sec. 3.1) on the tensor cores:
//   K[s][c] = exp( sum_k B[c][k] xi[s][k] )
// by the error-free splitting of Ozaki, Ogita, Oishi & Rump (Numer. Algorithms
// 59, 2012).  A row of B (or xi) is scaled by a power of two to magnitudes
// below 1/2 and cut into nine signed digits of seven bits, |d| <= 64, which
// BF16 holds exactly (digit i as d 2^(-7 i)): 63 bits below the row's scale,
// where FP64 has 53 below each entry.  The product of two digits is at most
// 2^12 units, so the sum of the products of all digit pairs (i, j) with i + j
// = t over up to 512 modes stays within 2^24 units: the FP32 accumulators of
// the tensor cores hold it exactly, in whatever order they add.  Pairs with i +
// j <= 8 (from 0) are kept: t = 0 .. 7 in accumulators of their own, t = 8, whose
// place value is 2^-70 of the row scales, rounded into the eighth; the rest
// are below 2^-65.  The epilogue joins the accumulators in integers, rounds
// twice, and takes the exponential.  (Eight digits and t <= 7 would do for
// rows of even size; a row with one entry thousands of times the others,
// against a small coefficient, was then less accurate than the plain sum.)
//
// Bound: the FP64 pipe, two operations per clock and SM.  A contraction in it
// takes M operations per field value and its exponential 21; here the
// conversion takes 3 and the exponential 11 (fm_exp below), and the 45 M
// tensor-core products per value run beside it, a tile ahead.  2000 fields of
// 64 x 64 cells from 128 modes: 272 us (388 with a tile per CTA and two CTAs an
// SM, whose loads and products were not hidden), 2035 by the FP64 contraction (95% of that
// pipe), with errors against 128-bit arithmetic of 8.2e-17 (rms; at most
// 4.9e-16) against its 6.9e-16 (6.2e-15).  From 256 modes up the products bound
// it: 100 fields of 256 x 256 from 256 modes 336 us (3791 by the contraction), 500 of 64 x
// 64 from 512 modes 198 (2134).
//
// A tile is 128 cells x 32 samples: eight 128 x 32 accumulators in 256 columns
// of tensor memory, the digits of 32 modes per stage (64-byte swizzle, 90 KB).
// The basis is cut once, when it is installed; the coefficients are cut by four
// warps of every CTA, straight into the operand stage, so that a call keeps
// nothing: no buffer to size, to share between streams or to hold under a capture.
// Each tile cuts its 32 rows anew, in integers beside the FP64 pipe (a kernel of
// its own for them and their digits by TMA took 284 us for the first case above).
#include <cuda_bf16.h>
#include <cudaTypedefs.h>

#include <algorithm>

#include "common.cuh"
#include "tc.cuh"

namespace fm {

constexpr int kOzDigits = 9, kOzBits = 7, kOzAcc = 8;   // digits a row, bits a digit, accumulators
constexpr int kOzM = 128;      // cells per tile (MMA M)
constexpr int kOzN = 32;       // samples per tile (MMA N)
constexpr int kOzK = 32;       // modes per stage (one 64-byte swizzle row)
constexpr int kOzEpi = 256;          // threads that drain and store
constexpr int kOzCut = 128;          // threads that cut the coefficients
constexpr int kOzThreads = kOzEpi + 64 + kOzCut;
constexpr int kOzStages = 2;
constexpr unsigned kOzBand = 8;      // cell tiles of a band (4 .. 32 within 1% of one another)
constexpr int kOzMaxM = 512;   // 512 modes x 8 pairs x 2^12 = 2^24
constexpr uint32_t kOzABytes = kOzM * kOzK * 2, kOzBBytes = kOzN * kOzK * 2;
constexpr uint32_t kOzStage = kOzDigits * (kOzABytes + kOzBBytes);
constexpr int kOzRowSets = 4;  // tiles whose coefficient rows' scales are kept (see the cutting warps)
constexpr size_t kOzSmem = 1024 + kOzStages * kOzStage + 64 * 16 + kOzRowSets * kOzN * 4 + 192;
constexpr int kOzNoScale = -(1 << 28);   // exponent of a row that is not split (a value that is not finite, or far out)
// Largest sum of a pair's scale exponents that is split whatever the sum of its
// products.  What is left out is relative to the scales (below 2^-60 of their
// product), not to the sum, so a large entry that meets a zero coefficient would
// cost digits (2^40 against 0: 1e-6 of the field); up to this line it is under
// 2^-50 of the field.  The line is on the product of the two rows' largest
// magnitudes, whichever modes hold them.  Past it a pair is split where its sum g is
// as large as kOzSumBits allow: the part left out is then below half an ulp of g.
// (A constant of -120 in the logarithm takes every pair past the line: 2000 fields of
// 64 x 64 from 128 modes 4.02 ms by plain sums, 2.05 by the FP64 contraction, 0.28 so.)
constexpr int kOzMaxScale = 10, kOzSumBits = 6, kOzFarScale = 400;
constexpr size_t kOzMaxBytes = (size_t)4 << 30;   // most digits kept per level

// 2^(j / 64) as the sum of two doubles.
__device__ const double2 kExpTable[64] = {
    {0x1.0000000000000p+0, 0x0.0p+0}, {0x1.02c9a3e778061p+0, -0x1.19083535b085dp-56},
    {0x1.059b0d3158574p+0, 0x1.d73e2a475b465p-55}, {0x1.0874518759bc8p+0, 0x1.186be4bb284ffp-57},
    {0x1.0b5586cf9890fp+0, 0x1.8a62e4adc610bp-54}, {0x1.0e3ec32d3d1a2p+0, 0x1.03a1727c57b53p-59},
    {0x1.11301d0125b51p+0, -0x1.6c51039449b3ap-54}, {0x1.1429aaea92de0p+0, -0x1.32fbf9af1369ep-54},
    {0x1.172b83c7d517bp+0, -0x1.19041b9d78a76p-55}, {0x1.1a35beb6fcb75p+0, 0x1.e5b4c7b4968e4p-55},
    {0x1.1d4873168b9aap+0, 0x1.e016e00a2643cp-54}, {0x1.2063b88628cd6p+0, 0x1.dc775814a8495p-55},
    {0x1.2387a6e756238p+0, 0x1.9b07eb6c70573p-54}, {0x1.26b4565e27cddp+0, 0x1.2bd339940e9d9p-55},
    {0x1.29e9df51fdee1p+0, 0x1.612e8afad1255p-55}, {0x1.2d285a6e4030bp+0, 0x1.0024754db41d5p-54},
    {0x1.306fe0a31b715p+0, 0x1.6f46ad23182e4p-55}, {0x1.33c08b26416ffp+0, 0x1.32721843659a6p-54},
    {0x1.371a7373aa9cbp+0, -0x1.63aeabf42eae2p-54}, {0x1.3a7db34e59ff7p+0, -0x1.5e436d661f5e3p-56},
    {0x1.3dea64c123422p+0, 0x1.ada0911f09ebcp-55}, {0x1.4160a21f72e2ap+0, -0x1.ef3691c309278p-58},
    {0x1.44e086061892dp+0, 0x1.89b7a04ef80d0p-59}, {0x1.486a2b5c13cd0p+0, 0x1.3c1a3b69062f0p-56},
    {0x1.4bfdad5362a27p+0, 0x1.d4397afec42e2p-56}, {0x1.4f9b2769d2ca7p+0, -0x1.4b309d25957e3p-54},
    {0x1.5342b569d4f82p+0, -0x1.07abe1db13cadp-55}, {0x1.56f4736b527dap+0, 0x1.9bb2c011d93adp-54},
    {0x1.5ab07dd485429p+0, 0x1.6324c054647adp-54}, {0x1.5e76f15ad2148p+0, 0x1.ba6f93080e65ep-54},
    {0x1.6247eb03a5585p+0, -0x1.383c17e40b497p-54}, {0x1.6623882552225p+0, -0x1.bb60987591c34p-54},
    {0x1.6a09e667f3bcdp+0, -0x1.bdd3413b26456p-54}, {0x1.6dfb23c651a2fp+0, -0x1.bbe3a683c88abp-57},
    {0x1.71f75e8ec5f74p+0, -0x1.16e4786887a99p-55}, {0x1.75feb564267c9p+0, -0x1.0245957316dd3p-54},
    {0x1.7a11473eb0187p+0, -0x1.41577ee04992fp-55}, {0x1.7e2f336cf4e62p+0, 0x1.05d02ba15797ep-56},
    {0x1.82589994cce13p+0, -0x1.d4c1dd41532d8p-54}, {0x1.868d99b4492edp+0, -0x1.fc6f89bd4f6bap-54},
    {0x1.8ace5422aa0dbp+0, 0x1.6e9f156864b27p-54}, {0x1.8f1ae99157736p+0, 0x1.5cc13a2e3976cp-55},
    {0x1.93737b0cdc5e5p+0, -0x1.75fc781b57ebcp-57}, {0x1.97d829fde4e50p+0, -0x1.d185b7c1b85d1p-54},
    {0x1.9c49182a3f090p+0, 0x1.c7c46b071f2bep-56}, {0x1.a0c667b5de565p+0, -0x1.359495d1cd533p-54},
    {0x1.a5503b23e255dp+0, -0x1.d2f6edb8d41e1p-54}, {0x1.a9e6b5579fdbfp+0, 0x1.0fac90ef7fd31p-54},
    {0x1.ae89f995ad3adp+0, 0x1.7a1cd345dcc81p-54}, {0x1.b33a2b84f15fbp+0, -0x1.2805e3084d708p-57},
    {0x1.b7f76f2fb5e47p+0, -0x1.5584f7e54ac3bp-56}, {0x1.bcc1e904bc1d2p+0, 0x1.23dd07a2d9e84p-55},
    {0x1.c199bdd85529cp+0, 0x1.11065895048ddp-55}, {0x1.c67f12e57d14bp+0, 0x1.2884dff483cadp-54},
    {0x1.cb720dcef9069p+0, 0x1.503cbd1e949dbp-56}, {0x1.d072d4a07897cp+0, -0x1.cbc3743797a9cp-54},
    {0x1.d5818dcfba487p+0, 0x1.2ed02d75b3707p-55}, {0x1.da9e603db3285p+0, 0x1.c2300696db532p-54},
    {0x1.dfc97337b9b5fp+0, -0x1.1a5cd4f184b5cp-54}, {0x1.e502ee78b3ff6p+0, 0x1.39e8980a9cc8fp-55},
    {0x1.ea4afa2a490dap+0, -0x1.e9c23179c2893p-54}, {0x1.efa1bee615a27p+0, 0x1.dc7f486a4b6b0p-54},
    {0x1.f50765b6e4540p+0, 0x1.9d3e12dd8a18bp-54}, {0x1.fa7c1819e90d8p+0, 0x1.74853f3a5931ep-55},
};

// e^x to within 0.53 ulp (table-driven: Tang, ACM TOMS 15, 1989): x = n ln 2 / 64
// + r, e^x = 2^(n / 64) (1 + p(r)), |r| <= ln 2 / 128, p the Taylor polynomial
// of degree 5 (its remainder below 2^-54.6), the table value in two parts.
// Eleven FP64 operations; the exponent is added in integers.
__device__ __forceinline__ double fm_exp(double x, const double2* tab) {
    // (compared in integers: a comparison is an operation of the FP64 pipe too)
    if ((unsigned)(__double2hiint(x) & 0x7FFFFFFF) >= 0x4085E000u) return exp(x);   // |x| >= 700, NaN
    constexpr double kMagic = 6755399441055744.0;   // 1.5 2^52
    const double t = fma(x, 0x1.71547652b82fep+6, kMagic);
    const int n = __double2loint(t);
    const double tn = t - kMagic;
    const double r = fma(tn, -0x1.9ef35793c7673p-47, fma(tn, -0x1.62e42fefa2000p-7, x));
    const double r2 = r * r;
    double q = fma(r, 1.0 / 120, 1.0 / 24);
    q = fma(q, r, 1.0 / 6);
    q = fma(q, r, 0.5);
    const double p = fma(q, r2, r);
    const double2 e = tab[n & 63];
    const double v = e.x + fma(e.x, p, e.y);
    return __hiloint2double(__double2hiint(v) + ((n >> 6) << 20), __double2loint(v));
}

// The sum of the eight accumulators (of d d 2^(-7 t)), in units of 2^-14, scaled
// by 2^e.
__device__ __forceinline__ double oz_join(const uint32_t (&acc)[kOzAcc][8], int i, int e) {
    long long h = 0, l = 0;
#pragma unroll
    for (int t = 0; t < 4; ++t) {
        const float uh = __uint_as_float(acc[t][i]) * (float)(1LL << (kOzBits * t));
        const float ul = __uint_as_float(acc[t + 4][i]) * (float)(1LL << (kOzBits * (t + 4)));
        h += (long long)__float2int_rn(uh) * (1LL << (kOzBits * (3 - t)));
        l += (long long)__float2int_rn(ul) * (1LL << (kOzBits * (3 - t)));
    }
    // |h|, |l| < 2^51: the bits of 1.5 2^52 + h, less 1.5 2^52
    constexpr long long kBits = 0x4338000000000000LL;
    constexpr double kMagic = 6755399441055744.0;
    const double dh = __longlong_as_double(kBits + h) - kMagic, dl = __longlong_as_double(kBits + l) - kMagic;
    const double g = fma(dl, 0x1p-28, dh);
    const int hi = __double2hiint(g);
    // times 2^(e - 35) in the exponent field (g is 0 or between 2^-28 and 2^47)
    return (hi << 1) == 0 ? 0.0 : __hiloint2double(hi + ((e - 5 * kOzBits) << 20), __double2loint(g));
}

__device__ __forceinline__ void tmem_ld_32x32b_x8(uint32_t taddr, uint32_t (&r)[8]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr)
                 : "memory");
}

// Shared-memory matrix descriptor of a K-major tile written by TMA with
// 64-byte swizzling: rows of 64 B, 8-row groups 512 B apart.
__device__ __forceinline__ uint64_t sdesc_kmajor_sw64(uint32_t saddr) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);   // start address
    d |= (uint64_t)1 << 16;                     // leading-dimension offset (unused here)
    d |= (uint64_t)(512 >> 4) << 32;            // stride between 8-row groups
    d |= (uint64_t)1 << 46;                     // descriptor version of tcgen05
    d |= (uint64_t)4 << 61;                     // 64-byte swizzle
    return d;
}

// The scale exponent of a row whose largest biased exponent is top: 2^e is at
// least twice the largest magnitude.  Rows with values that are not finite, or
// with scales far from 1, are left to the plain sum (kOzNoScale).
__device__ __forceinline__ int row_scale(int top) {
    const int e = top - 1023 + 2;
    if (top == 0) return 0;
    return top != 0x7FF && e < 200 && e > -200 ? e : kOzNoScale;
}
// x below the scale 2^e as a 63-bit fixed-point number (units of 2^(e - 63)).
__device__ __forceinline__ long long row_fixed(double x, int e) {
    const long long bits = __double_as_longlong(x);
    const int be = (int)(bits >> 52) & 0x7FF;
    if (be == 0 || e == kOzNoScale) return 0;
    const long long m = (bits & 0xFFFFFFFFFFFFFLL) | (1LL << 52);   // at exponent be - 1075
    const int sh = be - 1075 - (e - kOzDigits * kOzBits);           // at most 9
    long long v = 0;
    if (sh >= 0) v = m << sh;
    else if (sh > -54) v = (m + (1LL << (-sh - 1))) >> -sh;
    return bits < 0 ? -v : v;
}
// Digit i of v, balanced, cut from the low end (i = kOzDigits - 1 first, 0 last),
// as the bits of the FP32 number d 2^(-7 i), whose upper half is its BF16.
__device__ __forceinline__ unsigned next_digit(long long& v, int i) {
    const int d = i > 0 ? ((int)(v + 64) & 127) - 64 : (int)v;
    v = (v - d) >> kOzBits;
    const float f = __uint_as_float(0x4B400000u + (unsigned)d) - 12582912.0f;   // 1.5 2^23 + d
    return __float_as_uint(f * (1.0f / (float)(1LL << (kOzBits * i))));
}

// Persistent: CTA b takes tiles b, b + gridDim.x, ...
// Warps 0 .. 7 drain, warp 8 (one thread) loads the basis digits, warp 9 (one
// thread) issues the products, warps 10 .. 13 cut the coefficients; two stages of
// operands and two sets of accumulators, so the next tile's products run under
// this one's epilogue.
__global__ void __launch_bounds__(kOzThreads, 1)
    k_kl_split(const __grid_constant__ CUtensorMap mapA, int cells, int S, int M, int Mpad,
               const int* __restrict__ ec, const double* __restrict__ B, const double* __restrict__ xi,
               double* __restrict__ K, int* __restrict__ err) {
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = tc::smem_u32(smem_raw);
    uint8_t* stage = smem_raw + ((1024 - (raw & 1023)) & 1023);   // per stage: A digits, then B digits
    double2* tab = reinterpret_cast<double2*>(stage + kOzStages * kOzStage);
    int* ex = reinterpret_cast<int*>(tab + 64);   // the coefficient rows' scales, by tile (kOzRowSets in turn)
    uint64_t* full = reinterpret_cast<uint64_t*>(ex + kOzRowSets * kOzN);   // basis digits in
    uint64_t* cut = full + kOzStages;             // coefficient digits in
    uint64_t* scaled = cut + kOzStages;           // a tile's scales in
    uint64_t* empty = scaled + kOzRowSets;
    uint64_t* tfull = empty + kOzStages;    // accumulators ready, by set
    uint64_t* tempty = tfull + 2;           // accumulators drained
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(tempty + 2);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const unsigned stiles = (unsigned)(S + kOzN - 1) / kOzN, ctiles = (unsigned)(cells + kOzM - 1) / kOzM;
    const unsigned tiles = stiles * ctiles;
    // Tile t: bands of kOzBand cell tiles, in a band the cell tiles of one sample tile
    // after the other.  CTAs that run side by side share operands and write runs of 8 KB
    // of a field.  Sample tiles fastest, they wrote 1 KB of every field at a stride of a
    // field: once tiles of unlike length (a last one of few samples) had set the CTAs
    // apart, 817 fields of 256 x 256 from 108 modes took 1.82 ms, 1.65 so.
    struct At {
        int s0, c0;
    };
    auto at = [&](unsigned t) {
        const unsigned band = t / (stiles * kOzBand), r = t - band * stiles * kOzBand;
        const unsigned w = min(kOzBand, ctiles - band * kOzBand);
        return At{(int)(r / w) * kOzN, (int)(band * kOzBand + r % w) * kOzM};
    };
    if (threadIdx.x < 64) tab[threadIdx.x] = kExpTable[threadIdx.x];
    if (threadIdx.x == 0) {
        for (int i = 0; i < kOzStages; ++i) {
            tc::mbar_init(&full[i], 1);
            tc::mbar_init(&cut[i], kOzCut / 32);
            tc::mbar_init(&empty[i], 1);
        }
        for (int i = 0; i < kOzRowSets; ++i) tc::mbar_init(&scaled[i], kOzN);
        for (int i = 0; i < 2; ++i) {
            tc::mbar_init(&tfull[i], 1);
            tc::mbar_init(&tempty[i], kOzEpi);
        }
        tc::fence_barrier_init();
        tc::prefetch_tensormap(&mapA);
    }
    if (warp == 0) tc::tmem_alloc(tmem_slot, 2 * kOzAcc * kOzN);
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem = *tmem_slot;
    const int kblocks = Mpad / kOzK;
    if (warp == 8) {
        if (lane == 0) {
            int q = 0;   // stage loads so far
            bool ok = true;
            for (unsigned tile = blockIdx.x; ok && tile < tiles; tile += gridDim.x) {
                const int c0 = at(tile).c0;
                for (int kb = 0; kb < kblocks; ++kb) {
                    const int st = q % kOzStages, round = q / kOzStages;
                    if (round > 0 && !(ok = tc::mbar_wait(&empty[st], (round - 1) & 1, err))) break;
                    uint8_t* a = stage + st * kOzStage;
                    tc::mbar_arrive_expect_tx(&full[st], kOzDigits * kOzABytes);
                    for (int i = 0; i < kOzDigits; ++i)
                        tc::tma_load_2d(a + i * kOzABytes, &mapA, &full[st], i * Mpad + kb * kOzK, c0);
                    ++q;
                }
            }
            tc::drain_loads(full, kOzStages, q, err);
        }
    } else if (warp == 9) {
        if (lane == 0) {
            constexpr uint32_t idesc = tc::idesc_bf16_f32(kOzM, kOzN);
            int q = 0, it = 0;
            bool ok = true;
            for (unsigned tile = blockIdx.x; ok && tile < tiles; tile += gridDim.x, ++it) {
                const int set = it & 1;
                if (it >= 2 && !(ok = tc::mbar_wait(&tempty[set], ((it >> 1) - 1) & 1, err))) break;
                tc::fence_after_sync();
                const uint32_t acc = tmem + set * (kOzAcc * kOzN);
                for (int kb = 0; kb < kblocks; ++kb, ++q) {
                    const int st = q % kOzStages;
                    if (!(ok = tc::mbar_wait(&full[st], (q / kOzStages) & 1, err))) break;
                    if (!(ok = tc::mbar_wait(&cut[st], (q / kOzStages) & 1, err))) break;
                    tc::fence_after_sync();
                    const uint32_t sa = tc::smem_u32(stage + st * kOzStage);
                    const uint64_t da = sdesc_kmajor_sw64(sa), db = sdesc_kmajor_sw64(sa + kOzDigits * kOzABytes);
                    // Unrolled, descriptors by constant steps: formed anew for every product,
                    // their instructions held the tensor cores up (one thread issues, in a warp
                    // beside three others of its scheduler): 100 fields of 256 x 256 from 256 modes
                    // 475 us, 351 so.
#pragma unroll
                    for (int i = 0; i < kOzDigits; ++i)
#pragma unroll
                        for (int j = 0; j < kOzDigits - i; ++j) {
                            const int t = i + j < kOzAcc ? i + j : kOzAcc - 1;
#pragma unroll
                            for (int k = 0; k < kOzK / 16; ++k)
                                tc::mma_bf16(acc + t * kOzN, da + (i * kOzABytes + 32 * k) / 16,
                                             db + (j * kOzBBytes + 32 * k) / 16, idesc,
                                             (kb | i | k) != 0 || j >= kOzAcc);
                        }
                    tc::mma_commit(&empty[st]);
                }
                tc::mma_commit(&tfull[set]);
            }
        }
    } else if (warp >= 10) {
        // Eight rows a warp.  The digits of modes 2 p, 2 p + 1 of two rows at a time: lane
        // 16 h + p has row h, its 4 bytes of the row's 64 at 4 p, whose 16-byte chunk the
        // swizzle exchanges by bits 7, 8 of the address (the row's bits 1, 2).
        const int r0 = 8 * (warp - 10), p = lane & 15, half = lane >> 4;
        int q = 0, it = 0;
        bool ok = true;
        for (unsigned tile = blockIdx.x; ok && tile < tiles; tile += gridDim.x, ++it) {
            const int s0 = at(tile).s0;
            const double* rows[8];   // rows past the batch: the last one's, cut to zero below and never stored
            int top[8];              // largest biased exponent of each row
#pragma unroll
            for (int r = 0; r < 8; ++r) {
                rows[r] = xi + (size_t)min(s0 + r0 + r, S - 1) * M;
                top[r] = 0;
            }
#pragma unroll 2
            for (int k = lane; k < M; k += 32) {   // (sixteen loads in flight)
#pragma unroll
                for (int r = 0; r < 8; ++r) top[r] = max(top[r], (__double2hiint(__ldcg(rows[r] + k)) >> 20) & 0x7FF);
            }
            int e_mine = 0;   // lane r: the scale of row r0 + r
#pragma unroll
            for (int r = 0; r < 8; ++r) {
                const int e = row_scale(__reduce_max_sync(0xffffffffu, top[r]));
                if (lane == r) e_mine = s0 + r0 + r < S ? e : 0;
            }
            for (int kb = 0; kb < kblocks; ++kb, ++q) {
                const int st = q % kOzStages, round = q / kOzStages, k = kb * kOzK + 2 * p;
                // cut before the stage is free: between the products that read it last and those
                // that read it next there are the stores alone
                unsigned dig[4][kOzDigits];
                {
                    double x[4][2];
#pragma unroll
                    for (int r2 = 0; r2 < 4; ++r2) {
                        const int s = s0 + r0 + 2 * r2 + half;
                        const double* row = xi + (size_t)s * M;
                        x[r2][0] = s < S && k < M ? __ldcg(row + k) : 0.0;
                        x[r2][1] = s < S && k + 1 < M ? __ldcg(row + k + 1) : 0.0;
                    }
#pragma unroll
                    for (int r2 = 0; r2 < 4; ++r2) {
                        const int e = __shfl_sync(0xffffffffu, e_mine, 2 * r2 + half);
                        long long v0 = row_fixed(x[r2][0], e), v1 = row_fixed(x[r2][1], e);
#pragma unroll
                        for (int i = kOzDigits - 1; i >= 0; --i) {
                            const unsigned d0 = next_digit(v0, i), d1 = next_digit(v1, i);
                            dig[r2][i] = __byte_perm(d0, d1, 0x7632);
                        }
                    }
                }
                if (round > 0) {
                    ok = __all_sync(0xffffffffu, tc::mbar_wait(&empty[st], (round - 1) & 1, err));
                    if (!ok) break;
                }
                // The set of scales of kOzRowSets tiles ago is free: this stage was last read
                // by products of a tile at most two before this one, and these began once
                // the tile two before theirs was drained.
                if (kb == 0 && lane < 8) {
                    ex[(it % kOzRowSets) * kOzN + r0 + lane] = e_mine;
                    tc::mbar_arrive(&scaled[it % kOzRowSets]);
                }
                uint8_t* b = stage + st * kOzStage + kOzDigits * kOzABytes;
#pragma unroll
                for (int r2 = 0; r2 < 4; ++r2) {
                    const int r = r0 + 2 * r2 + half;
                    uint8_t* dst = b + 64 * r + (((p >> 2) ^ ((r >> 1) & 3)) << 4) + 4 * (p & 3);
#pragma unroll
                    for (int i = 0; i < kOzDigits; ++i) *reinterpret_cast<unsigned*>(dst + i * kOzBBytes) = dig[r2][i];
                }
                tc::fence_proxy_async_smem();   // the stores are operands of the tensor cores
                __syncwarp();
                if (lane == 0) tc::mbar_arrive(&cut[st]);
            }
        }
    } else {
        int it = 0;
        for (unsigned tile = blockIdx.x; tile < tiles; tile += gridDim.x, ++it) {
            const int set = it & 1;
            const int s0 = at(tile).s0, c0 = at(tile).c0;
            const int c = c0 + 32 * (warp & 3) + lane;
            const int e_c = c < cells ? ec[c] : 0;
            // all lanes or none (the loads below are warp-wide)
            bool ok = __all_sync(0xffffffffu, tc::mbar_wait(&scaled[it % kOzRowSets], (it / kOzRowSets) & 1, err));
            if (!ok) break;
            const int e_row = ex[(it % kOzRowSets) * kOzN + lane];   // lane r: the scale of row r
            ok = __all_sync(0xffffffffu, tc::mbar_wait(&tfull[set], (it >> 1) & 1, err));
            if (!ok) break;
            tc::fence_after_sync();
            const uint32_t row = tmem + set * (kOzAcc * kOzN) + ((uint32_t)(32 * (warp & 3)) << 16);
#pragma unroll 1
            for (int h = 0; h < 2; ++h) {
                const int col = 16 * (warp >> 2) + 8 * h;
                uint32_t acc[kOzAcc][8];
#pragma unroll
                for (int t = 0; t < kOzAcc; ++t) tmem_ld_32x32b_x8(row + t * kOzN + col, acc[t]);
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                if (h == 1) {   // this thread has read the set
                    tc::fence_before_sync();
                    tc::mbar_arrive(&tempty[set]);
                }
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int s = s0 + col + i;
                    const int e = e_c + __shfl_sync(0xffffffffu, e_row, col + i);
                    if (c >= cells || s >= S) continue;
                    double g = 0.0;
                    bool split = e > -(1 << 20) && e <= kOzFarScale;
                    if (split) {
                        g = oz_join(acc, i, e);
                        split = e <= kOzMaxScale || e <= ((__double2hiint(g) >> 20) & 0x7FF) - 1023 + kOzSumBits;
                    }
                    if (!split) {   // a row or a pair that is not split: the plain sum
                        g = 0.0;
                        for (int k = 0; k < M; ++k) g = fma(xi[(size_t)s * M + k], B[(size_t)c * M + k], g);
                    }
                    __stcs(K + (size_t)s * cells + c, fm_exp(g, tab));   // streamed past the operands in L2
                }
            }
        }
    }
    tc::fence_before_sync();
    __syncthreads();
    if (warp == 0) tc::tmem_dealloc(tmem, 2 * kOzAcc * kOzN);
}

// Rows of x (FP64 [rows][M]) -> digits out [rows][9 Mpad] BF16, digit i of mode
// k at i Mpad + k (zero beyond M), and the rows' scale exponents: x = 2^(e - 7)
// sum_i d_i 2^(-7 i).  One warp per row.  In integers: the value below the scale
// as a 63-bit fixed-point number, cut from the low end into balanced digits.
__global__ void k_split_rows(size_t rows, int M, int Mpad, const double* __restrict__ x,
                             __nv_bfloat16* __restrict__ out, int* __restrict__ exps) {
    const size_t r = ((size_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (r >= rows) return;
    const double* row = x + r * M;
    int top = 0;   // largest biased exponent of the row
    for (int k = lane; k < M; k += 32) top = max(top, (__double2hiint(row[k]) >> 20) & 0x7FF);
    top = __reduce_max_sync(0xffffffffu, top);
    const int e = row_scale(top);
    if (lane == 0) exps[r] = e;
    __nv_bfloat16* o = out + r * (size_t)(kOzDigits * Mpad);
    for (int k = lane; k < Mpad; k += 32) {
        long long v = k < M ? row_fixed(row[k], e) : 0;
#pragma unroll
        for (int i = kOzDigits - 1; i >= 0; --i)
            o[(size_t)i * Mpad + k] = __ushort_as_bfloat16((unsigned short)(next_digit(v, i) >> 16));
    }
}

// ------------------------------------------------------------------ host
static bool oz_map(CUtensorMap* map, const void* ptr, uint64_t rows, uint64_t width, uint32_t box_rows) {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    if (!fn) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) !=
                cudaSuccess ||
            q != cudaDriverEntryPointSuccess)
            return false;
        fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    }
    cuuint64_t dims[2] = {width, rows};
    cuuint64_t strides[1] = {width * 2};
    cuuint32_t box[2] = {(cuuint32_t)kOzK, box_rows};
    cuuint32_t estr[2] = {1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(ptr), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

static unsigned warps_grid(size_t rows) { return (unsigned)((rows + 7) / 8); }

// Digits of the installed basis, level by level (levels whose digits would
// take more than kOzMaxBytes, and bases of more than 512 modes, keep the FP64
// contraction).
fm_status kl_split_install(fm_ctx* ctx) {
    const int M = ctx->cfg.M;
    OzState& z = ctx->oz;
    z.Mpad = (M + kOzK - 1) / kOzK * kOzK;
    for (int l = 0; l < ctx->cfg.n_levels; ++l) {
        const int n = grid_of_level(ctx, l);
        const size_t cells = (size_t)n * n, bytes = cells * kOzDigits * z.Mpad * 2;
        z.have[l] = false;
        if (M > kOzMaxM || bytes > kOzMaxBytes || cells > ((size_t)1 << 30)) continue;
        if (!z.basis[l] && (cudaMalloc(&z.basis[l], bytes) != cudaSuccess ||
                            cudaMalloc((void**)&z.ec[l], cells * sizeof(int)) != cudaSuccess)) {
            cudaGetLastError();   // no room for the digits: the FP64 contraction serves this level
            cudaFree(z.basis[l]);
            z.basis[l] = nullptr;
            continue;
        }
        k_split_rows<<<warps_grid(cells), 256>>>(cells, M, z.Mpad, ctx->d_basis[l], (__nv_bfloat16*)z.basis[l],
                                                 z.ec[l]);
        z.have[l] = oz_map(&z.mapA[l], z.basis[l], cells, (uint64_t)kOzDigits * z.Mpad, kOzM);
    }
    FM_CUDA_TRY(ctx, cudaDeviceSynchronize());
    return FM_OK;
}

void kl_split_free(fm_ctx* ctx) {
    for (int l = 0; l < FM_MAX_LEVELS; ++l) {
        cudaFree(ctx->oz.basis[l]);
        cudaFree(ctx->oz.ec[l]);
    }
}

// Fields of n samples of `level` into d_K; false: no digits of this level are
// installed, and the caller's FP64 contraction serves the call.
bool kl_split_field(fm_ctx* ctx, int level, uint32_t n, const double* d_xi, double* d_K, cudaStream_t st,
                    fm_status* status) {
    OzState& z = ctx->oz;
    *status = FM_OK;
    if (!z.have[level]) return false;
    const int N = grid_of_level(ctx, level), cells = N * N, M = ctx->cfg.M;
    const size_t tiles = (size_t)((n + kOzN - 1) / kOzN) * ((cells + kOzM - 1) / kOzM);
    const unsigned grid = (unsigned)std::min<size_t>(tiles, (size_t)std::max(ctx->sms, 1));
    FM_TIMED(ctx, kFamKlGemm, st, 8.0 * ((double)n * M + (double)cells * M + (double)n * cells),
             2.0 * n * (double)cells * M,
             k_kl_split<<<grid, kOzThreads, kOzSmem, st>>>(z.mapA[level], cells, (int)n, M, z.Mpad, z.ec[level],
                                                           ctx->d_basis[level], d_xi, d_K, ctx->tc.err));
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
        set_error(ctx, std::string("kl_field_batch: ") + cudaGetErrorString(e));
        *status = FM_ECUDA;
    }
    return true;
}

void kl_split_init_attributes() {
    cudaFuncSetAttribute(k_kl_split, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kOzSmem);
    cudaGetLastError();
}

}  // namespace fm
