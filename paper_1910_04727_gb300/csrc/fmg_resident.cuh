// Arguments and work counts of the sample-resident FMG kernels.
#pragma once

#include "common.cuh"

namespace fm {

// A sample whose V-cycles left the finite numbers: its QoI until a second launch has
// solved it again by the shared-memory form (a payload no arithmetic makes).
constexpr long long kAgain = 0x7ff8000057313641ll;

struct ResidentArgs {
    int n_fine, n0;
    size_t S;
    const double* K;
    Ghost<double> bd;   // boundary data (Table 1)
    int nu0, nu1, nu2;
    int ir;   // V-cycles between residual tests of a converged stage
    int converged, max_cycles;
    double tol, qtol;
    double *qf, *qc, *p_out;
    int32_t* status;
    bool again;      // only the samples whose qf is kAgain
    double* flops;   // nullable (profiling): [0] solver flops, [1] their FP64 part, [2] model bytes
};

// Solver flops of one V(nu1, nu2) cycle from grid k down: per grid j >= 1,
// nu1 + nu2 sweeps of 10 flops a cell, residual + restriction 10, correction
// 8; the coarsest solve a dense 16 x 16 product.
__device__ __forceinline__ double vcycle_flops(int n0, int k, int nu1, int nu2) {
    double f = 2.0 * (n0 * n0) * (n0 * n0);
    for (int j = 1; j <= k; ++j) {
        const double c = (double)(n0 << j) * (n0 << j);
        f += c * (10.0 * (nu1 + nu2) + 18.0);
    }
    return f;
}

// Algorithmic bytes of the same cycle in the streaming byte model of the
// level-wise kernels (each sweep reads p, K, b and writes p: 16 B per cell in
// FP32; residual + restriction 13 B and prolongation + correction 9 B per
// fine cell; twice that in FP64), the yardstick the resident kernel's
// effective bandwidth is quoted against.
__device__ __forceinline__ double vcycle_bytes(int n0, int k, int nu1, int nu2, int ts) {
    double b = 0.0;
    for (int j = 1; j <= k; ++j) {
        const double c = (double)(n0 << j) * (n0 << j);
        b += c * (16.0 * (nu1 + nu2) + 22.0) * (ts / 4.0);
    }
    return b;
}

// The converged mixed form with grids in registers: 16 x 16, one sample per warp
// (fmg_warp16.cu), and 32 x 32, one per five warps (fmg_team32.cu), coarsest grid
// 4 x 4.  Samples that leave the finite numbers come back as kAgain in qf.
// (..._init: kernel attributes on the current device.)
void warp16_init();
void team32_init();
void launch_warp16(fm_ctx* ctx, const ResidentArgs& a, cudaStream_t st);
void launch_team32(fm_ctx* ctx, const ResidentArgs& a, cudaStream_t st);

// The level-wise V-cycle from the 32 x 32 correction grid down in registers
// (fmg_team32.cu): operators of the grids 8, 16, 32, the 4 x 4 inverse, the 32 x 32
// rhs and result; S CTAs, one a sample (listed by order, if given).
struct Tail32Args {
    int nu1, nu2, ns;
    const float *Te[3], *Tn[3], *D[3];
    const float *Ainv, *b;
    float* p;
    const int32_t *active, *order;
};
void launch_tail32(const Tail32Args& a, size_t S, cudaStream_t st);

}  // namespace fm
