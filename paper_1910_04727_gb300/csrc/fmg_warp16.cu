// Sample-resident FMG of 16 x 16 samples in the mixed form (the level-0 work of
// an estimate): the arithmetic of fmg_resident.cu, operation for operation, with
// one sample per warp and its grids in registers.
//
// Lane l holds, of the 16 x 16 grid, columns 2 (l mod 8), +1 of rows 4 (l / 8) ..
// +3: eight cells, four of each colour, whose colours are fixed by the unrolled
// row; of the 8 x 8 grid, the 2 x 2 block (l mod 4, l / 4 mod 4) (lanes 16 .. 31
// repeat lanes 0 .. 15), which is one cell of the 4 x 4 grid.  A half-sweep
// of the 16 x 16 grid is six shuffles and four independent updates of four FMAs
// and a product; residuals restrict within a lane; transfers between the grids
// are shuffles.  Shared memory (13.9 KB a warp, 16 warps an SM) holds the FP64 side
// (iterate, faces, diagonal of the refined grid, cell c on lane c mod 32) and the
// coarsest inverse.
//
// Bound: the FP64 pipe (2 lanes a clock and SM), 72 % of its rate: six operations a
// cell and residual, one an update, five a face.  Conversions, the norm of the
// residual and the flop counts stay out of it.  20000 samples:
// 5.1 ms by the shared-memory form (nine loads an update, one update after the
// other, 107000 instructions a sample), 2.7 ms with the grids in registers and
// everything inlined (instruction fetch), 1.3 ms so.
#include <algorithm>
#include <cmath>

#include "fmg_warp.cuh"

namespace fm {

constexpr int kW16Warps = 4;

__global__ void __launch_bounds__(32 * kW16Warps, 4) k_fmg_warp16(ResidentArgs a) {
    extern __shared__ __align__(16) unsigned char w16_smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    W16Smem& sm = reinterpret_cast<W16Smem*>(w16_smem)[warp];
    const Ghost<float> td{(float)a.bd.w, (float)a.bd.e, (float)a.bd.s, (float)a.bd.n, a.bd.ns};
    const Ghost<float> zero{0.0f, 0.0f, 0.0f, 0.0f, a.bd.ns};
    const size_t stride = (size_t)gridDim.x * kW16Warps;
#pragma unroll 1
    for (size_t s = (size_t)blockIdx.x * kW16Warps + warp; s < a.S; s += stride) {
        G8 g8;
        G16 g16;
        const Stages r = coarse_stages<4>(a, a.K + s * 256, g8, g16, sm, td, zero, lane);
        if (lane == 0) {
            if (a.flops && r.finite) {   // the counts of fmg_resident.cu
                const double c[2] = {64.0, 256.0};
                double work = 0.0, work64 = 0.0, model = 0.0;
                for (int st = 0; st < 2; ++st) {
                    const double updates = r.tests[st] ? r.tests[st] - 1.0 : 0.0;
                    work64 += c[st] * (14.0 * r.tests[st] + updates);
                    model += c[st] * 20.0 * r.tests[st] + r.cycles[st] * vcycle_bytes(4, 1 + st, a.nu1, a.nu2, 4);
                    work += r.cycles[st] * vcycle_flops(4, 1 + st, a.nu1, a.nu2);
                }
                atomicAdd(a.flops, work + work64);
                atomicAdd(a.flops + 1, work64);
                atomicAdd(a.flops + 2, model);
            }
            a.qf[s] = r.finite ? r.q[1] : __longlong_as_double(kAgain);
            if (a.qc) a.qc[s] = r.q[0];
            if (a.status) a.status[s] = r.ok ? FM_OK : FM_ENOTCONV;
        }
        if (a.p_out) {
            double* po = a.p_out + s * 256;
            for (int c = lane; c < 256; c += 32) po[c] = sm.p[c];
        }
        __syncwarp();
    }
}

void warp16_init() {
    constexpr size_t smem = kW16Warps * sizeof(W16Smem);
    cudaFuncSetAttribute(k_fmg_warp16, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
}

void launch_warp16(fm_ctx* ctx, const ResidentArgs& a, cudaStream_t st) {
    constexpr size_t smem = kW16Warps * sizeof(W16Smem);
    int per_sm = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_fmg_warp16, 32 * kW16Warps, smem);
    const size_t need = (a.S + kW16Warps - 1) / kW16Warps;
    const size_t grid = std::min<size_t>(need, (size_t)std::max(per_sm, 1) * std::max(ctx->sms, 1));
    k_fmg_warp16<<<(unsigned)grid, 32 * kW16Warps, smem, st>>>(a);
}

}  // namespace fm
