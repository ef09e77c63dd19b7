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

// The bilinear cell-centred prolongation (9, 3, 3, 1) / 16 of four coarse
// values: own cell, its x neighbour, its y neighbour, the diagonal one.  The
// roundings are spelled out, so every kernel that prolongs rounds the same
// way (left to the compiler's contraction, one of the strip kernels did not).
template <typename U>
__device__ __forceinline__ U prolong_vals(U own, U nx, U ny, U nxy) {
    return mul_rn(add_rn(fma(U(3), ny, fma(U(9), own, mul_rn(U(3), nx))), nxy), U(0.0625));
}

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

// Kernel attributes and occupancies, once per process.
template <typename T>
void strip_init(int sms);

}  // namespace fm
