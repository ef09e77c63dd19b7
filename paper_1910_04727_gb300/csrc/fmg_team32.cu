// Sample-resident FMG of 32 x 32 samples in the converged mixed form, one sample
// per CTA of five warps: the arithmetic of fmg_resident.cu with grids in registers.
//
// Warps 0 .. 3 hold a band of eight rows of the 32 x 32 grid each, laid out as the
// 16 x 16 grid of a warp (fmg_warp.cuh): lane l has columns 2 (l mod 16), +1 of rows
// 4 (l / 16) .. +3.  Half-sweeps take border rows of the bands above and below from
// shared memory, one barrier each.  Warp 4 runs the stages up to 16 x 16 beside the
// set-up of the 32 x 32 stage, then the V-cycle from 16 x 16 down for every cycle.
// The FP64 side is in shared memory, a column a lane and eight rows a warp.
//
// Bound: the FP64 pipe, as for 16 x 16 (four times its work a sample).  8000 samples:
// 9.7 ms by the shared-memory form (nine loads and a divide an update on 128
// threads), 2.5 ms so; 1000 samples 1.73 and 0.47 ms.
#include <algorithm>
#include <cmath>

#include "fmg_warp.cuh"

namespace fm {

namespace {

constexpr int kTeam = 160;        // threads: four bands and the coarse grids
constexpr int kBandBarrier = 1;   // named barrier of the bands

struct Borders {
    float top[4][32], bot[4][32];   // border rows of the bands' iterates
    float c16[256];                 // the 16 x 16 grid's rhs, then its correction
};

struct Team32Smem : Borders {
    double p[1024], d[1024], te[1024], tn[1024];
    double tw[32], ts[32];
    double f[4][32];
    union {
        struct {
            float te[1024], tn[1024], tw[32], ts[32];
        } faces;
        float r[1024];            // residual, then correction
    };
    Stop stop;
    float rr[4];                    // partial norms
    double r2[4], q;
    int bad;
    W16Smem w16;
};

// A band of the 32 x 32 grid.
struct Band {
    float w[4], ei[4], ee[4], sf[2], nf[4][2];
    float d[4][2], rd[4][2], b[4][2], p[4][2];
};

__device__ __forceinline__ void band_sync() { asm volatile("bar.sync %0, %1;" ::"n"(kBandBarrier), "n"(128) : "memory"); }

__device__ __forceinline__ void all_sync() { asm volatile("bar.sync 0, %0;" ::"n"(kTeam) : "memory"); }

template <Form F, int C>
__device__ __forceinline__ void half_sweep32(Band& g, Borders& sm, int band, int lane) {
    const int cx = lane & 15;
    const bool up = lane >= 16;   // the band's upper four rows
    float nb[4];
#pragma unroll
    for (int y = 0; y < 4; ++y) nb[y] = ((y + C) & 1) == 0 ? up1(g.p[y][1]) : dn1(g.p[y][0]);
    float lo = __shfl_up_sync(kAll, g.p[3][C & 1], 16), hi = __shfl_down_sync(kAll, g.p[0][(3 + C) & 1], 16);
    if (!up) lo = band > 0 ? sm.top[band - 1][2 * cx + (C & 1)] : 0.0f;
    if (up) hi = band < 3 ? sm.bot[band + 1][2 * cx + ((3 + C) & 1)] : 0.0f;
#pragma unroll
    for (int y = 0; y < 4; ++y) {
        const int x = (y + C) & 1;
        float acc = g.b[y][x];
        acc = x == 0 ? fmaf(g.w[y], nb[y], acc) : fmaf(g.ei[y], g.p[y][0], acc);
        acc = x == 0 ? fmaf(g.ei[y], g.p[y][1], acc) : fmaf(g.ee[y], nb[y], acc);
        acc = y == 0 ? fmaf(g.sf[x], lo, acc) : fmaf(g.nf[y > 0 ? y - 1 : 0][x], g.p[y > 0 ? y - 1 : 0][x], acc);
        acc = y == 3 ? fmaf(g.nf[3][x], hi, acc) : fmaf(g.nf[y][x], g.p[y < 3 ? y + 1 : 3][x], acc);
        g.p[y][x] = F == kResident32 ? quotient(acc, g.d[y][x], g.rd[y][x]) : __fmul_rn(acc, g.rd[y][x]);
    }
    if (up) sm.top[band][2 * cx + ((3 + C) & 1)] = g.p[3][(3 + C) & 1];
    else sm.bot[band][2 * cx + (C & 1)] = g.p[0][C & 1];
    band_sync();
}

template <Form F>
__device__ __forceinline__ void sweeps32(Band& g, Borders& sm, int n, int band, int lane) {
#pragma unroll 1
    for (int s = 0; s < n; ++s) {
        half_sweep32<F, 0>(g, sm, band, lane);
        half_sweep32<F, 1>(g, sm, band, lane);
    }
}

// Both border rows, after the iterate changed as a whole.
__device__ __forceinline__ void publish(const Band& g, Borders& sm, int band, int lane) {
    const int cx = lane & 15;
    if (lane >= 16) *reinterpret_cast<float2*>(&sm.top[band][2 * cx]) = make_float2(g.p[3][0], g.p[3][1]);
    else *reinterpret_cast<float2*>(&sm.bot[band][2 * cx]) = make_float2(g.p[0][0], g.p[0][1]);
    band_sync();
}

// Residual restricted to the 16 x 16 rhs.
template <Form F>
__device__ __forceinline__ void restrict32(const Band& g, Borders& sm, int band, int lane) {
    const int cx = lane & 15;
    const bool up = lane >= 16;
    float W[4], E[4], S[2], N[2];
#pragma unroll
    for (int y = 0; y < 4; ++y) {
        W[y] = up1(g.p[y][1]);
        E[y] = dn1(g.p[y][0]);
    }
#pragma unroll
    for (int x = 0; x < 2; ++x) {
        S[x] = __shfl_up_sync(kAll, g.p[3][x], 16);
        N[x] = __shfl_down_sync(kAll, g.p[0][x], 16);
        if (!up) S[x] = band > 0 ? sm.top[band - 1][2 * cx + x] : 0.0f;
        if (up) N[x] = band < 3 ? sm.bot[band + 1][2 * cx + x] : 0.0f;
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        float r[2][2];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int y = 2 * h + q, ys = y > 0 ? y - 1 : 0, yn = y < 3 ? y + 1 : 3;
            r[q][0] = residual<F, 0>(g.d[y][0], g.p[y][0], g.b[y][0], g.w[y], W[y], g.ei[y], g.p[y][1],
                                  y == 0 ? g.sf[0] : g.nf[ys][0], y == 0 ? S[0] : g.p[ys][0], g.nf[y][0],
                                  y == 3 ? N[0] : g.p[yn][0]);
            r[q][1] = residual<F, 1>(g.d[y][1], g.p[y][1], g.b[y][1], g.ei[y], g.p[y][0], g.ee[y], E[y],
                                  y == 0 ? g.sf[1] : g.nf[ys][1], y == 0 ? S[1] : g.p[ys][1], g.nf[y][1],
                                  y == 3 ? N[1] : g.p[yn][1]);
        }
        sm.c16[16 * (4 * band + 2 * (lane >> 4) + h) + cx] = r[0][0] + r[0][1] + r[1][0] + r[1][1];
    }
}

// p (+)= P u from the 16 x 16 values in sm.c16 (add: black cells alone where
// post-smoothing replaces the red ones).
__device__ __forceinline__ void prolong32(Band& g, const Borders& sm, const Ghost<float>& gh, bool add, bool all,
                                          int band, int lane) {
    const int I = lane & 15, J0 = 4 * band + 2 * (lane >> 4);
    float o[4], l[4], r[4];   // coarse rows J0 - 1 .. J0 + 2
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int J = min(max(J0 - 1 + q, 0), 15);
        const float* u = sm.c16 + 16 * J + I;
        o[q] = u[0];
        l[q] = I > 0 ? u[-1] : fmaf(2.0f, gh.w, -o[q]);
        r[q] = I < 15 ? u[1] : fmaf(2.0f, gh.e, -o[q]);
    }
    if (gh.ns && J0 == 0) {
        o[0] = fmaf(2.0f, gh.s, -o[0]);
        l[0] = fmaf(2.0f, gh.s, -l[0]);
        r[0] = fmaf(2.0f, gh.s, -r[0]);
    }
    if (gh.ns && J0 == 14) {
        o[3] = fmaf(2.0f, gh.n, -o[3]);
        l[3] = fmaf(2.0f, gh.n, -l[3]);
        r[3] = fmaf(2.0f, gh.n, -r[3]);
    }
#pragma unroll
    for (int y = 0; y < 4; ++y) {
        const int J = 1 + (y >> 1), K = (y & 1) ? J + 1 : J - 1, x = (y + 1) & 1;   // x: the black column
        const float vb = x == 0 ? prolong_vals(o[J], l[J], o[K], l[K]) : prolong_vals(o[J], r[J], o[K], r[K]);
        g.p[y][x] = add ? __fadd_rn(g.p[y][x], vb) : vb;
    }
    if (!all) return;
#pragma unroll
    for (int y = 0; y < 4; ++y) {
        const int J = 1 + (y >> 1), K = (y & 1) ? J + 1 : J - 1, x = y & 1;
        const float vr = x == 0 ? prolong_vals(o[J], l[J], o[K], l[K]) : prolong_vals(o[J], r[J], o[K], r[K]);
        g.p[y][x] = add ? __fadd_rn(g.p[y][x], vr) : vr;
    }
}

// One V-cycle on the 32 x 32 grid: the bands' part and the fifth warp's.
template <Form F>
__device__ __forceinline__ void band_vcycle(Band& g, Borders& sm, int nu1, int nu2, const Ghost<float>& zero, int band,
                                            int lane) {
#pragma unroll 1
    for (int h = 0; h < 2; ++h) {
        if (h) {
            restrict32<F>(g, sm, band, lane);
            all_sync();
            all_sync();   // the correction from 16 x 16 is in
            prolong32(g, sm, zero, true, nu2 == 0, band, lane);
            publish(g, sm, band, lane);
        }
        sweeps32<F>(g, sm, h ? nu2 : nu1, band, lane);
    }
}

template <Form F>
__device__ __forceinline__ void coarse_vcycle(G16& g16, G8& g8, Borders& sm, CoarseSmem& cs, int nu1, int nu2,
                                              const Ghost<float>& zero, int lane) {
    float* const c16 = sm.c16 + 16 * 4 * (lane >> 3) + 2 * (lane & 7);   // the lane's cells
    all_sync();   // the restricted residual is in
#pragma unroll
    for (int y = 0; y < 4; ++y) {
        const float2 r = *reinterpret_cast<const float2*>(c16 + 16 * y);
        g16.b[y][0] = r.x;
        g16.b[y][1] = r.y;
        g16.p[y][0] = g16.p[y][1] = 0.0f;
    }
    vcycle<F>(true, g16, g8, cs, nu1, nu2, zero, lane);
#pragma unroll
    for (int y = 0; y < 4; ++y) *reinterpret_cast<float2*>(c16 + 16 * y) = make_float2(g16.p[y][0], g16.p[y][1]);
    all_sync();
}

// FP64 faces of a band's rows and their FP32 copies; the edges' faces are 2K (or 0).
__device__ __forceinline__ void band_faces(const double* __restrict__ K, int ns, Team32Smem& sm, int band, int lane) {
    const int i = lane;
#pragma unroll 1
    for (int j = 8 * band; j < 8 * band + 8; ++j) {
        const double* f = K + 32 * j + i;
        const double k = __ldg(f);
        const int c = 32 * j + i;
        const double te = harmonic_mean(k, __ldg(f + (i < 31 ? 1 : 0)));
        if (i < 31) sm.te[c] = te;
        if (j < 31) sm.tn[c] = harmonic_mean(k, __ldg(f + 32));
    }
    if (lane < 8) {
        const int j = 8 * band + lane;
        sm.tw[j] = 2.0 * __ldg(K + 32 * j);
        sm.te[32 * j + 31] = 2.0 * __ldg(K + 32 * j + 31);
    }
    if (band == 0) sm.ts[lane] = ns ? 2.0 * __ldg(K + lane) : 0.0;
    if (band == 3) sm.tn[992 + lane] = ns ? 2.0 * __ldg(K + 992 + lane) : 0.0;
    band_sync();
#pragma unroll 1
    for (int j = 8 * band; j < 8 * band + 8; ++j) {
        const int c = 32 * j + i;
        const double te = sm.te[c], tn = sm.tn[c];
        const double tw = *(i > 0 ? sm.te + c - 1 : sm.tw + j), ts = *(j > 0 ? sm.tn + c - 32 : sm.ts + i);
        sm.d[c] = tw + te + ts + tn;
        sm.faces.te[c] = narrow(te);
        sm.faces.tn[c] = narrow(tn);
    }
    if (band == 0) {
        sm.faces.tw[lane] = narrow(sm.tw[lane]);
        sm.faces.ts[lane] = narrow(sm.ts[lane]);
    }
    band_sync();
}

__device__ __forceinline__ void band_load(const Team32Smem& sm, Band& g, int band, int lane) {
    const int cx = lane & 15;
    const auto& f = sm.faces;
#pragma unroll
    for (int y = 0; y < 4; ++y) {
        const int j = 8 * band + 4 * (lane >> 4) + y, c = 32 * j + 2 * cx;
        const float2 e = *reinterpret_cast<const float2*>(f.te + c), t = *reinterpret_cast<const float2*>(f.tn + c);
        const float w = *(cx > 0 ? f.te + c - 1 : f.tw + j);
        const float2 s = *reinterpret_cast<const float2*>(j > 0 ? f.tn + c - 32 : f.ts + 2 * cx);
        g.d[y][0] = w + e.x + s.x + t.x;
        g.d[y][1] = e.x + e.y + s.y + t.y;
        g.rd[y][0] = recip(g.d[y][0]);
        g.rd[y][1] = recip(g.d[y][1]);
        // no cells past the edges
        g.w[y] = cx > 0 ? w : 0.0f;
        g.ei[y] = e.x;
        g.ee[y] = cx < 15 ? e.y : 0.0f;
        g.nf[y][0] = j < 31 ? t.x : 0.0f;
        g.nf[y][1] = j < 31 ? t.y : 0.0f;
        if (y == 0) {
            g.sf[0] = j > 0 ? s.x : 0.0f;
            g.sf[1] = j > 0 ? s.y : 0.0f;
        }
    }
}

// The FP64 start of a band: the refined 16 x 16 solution interpolated.
__device__ __forceinline__ void band_interpolate(Team32Smem& sm, const Ghost<double>& bd, int band, int lane) {
    const int i = lane, I = i >> 1, x = (i & 1) ? 1 : -1;
    const double* u = sm.w16.p;
    const bool xe = I + x < 0 || I + x > 15;
    const double gx = 2.0 * (i == 0 ? bd.w : bd.e);
#pragma unroll 1
    for (int j = 8 * band; j < 8 * band + 8; ++j) {
        const int J = j >> 1, y = (j & 1) ? 1 : -1;
        const bool ye = J + y < 0 || J + y > 15;
        const double* row = u + 16 * J + I;
        const double* oth = ye ? row : row + 16 * y;
        const double o = row[0];
        double nx = xe ? o : row[x], ny = oth[0], nxy = xe ? oth[0] : oth[x];
        if (xe) {
            nx = gx - nx;
            nxy = gx - nxy;
        }
        if (ye && bd.ns) {
            const double gy = 2.0 * (j == 0 ? bd.s : bd.n);
            ny = gy - ny;
            nxy = gy - nxy;
        }
        sm.p[32 * j + i] = prolong_vals(o, nx, ny, nxy);
    }
}

// A band's residuals, rounded into sm.r; their FP32 norm.
__device__ __forceinline__ float band_residual(Team32Smem& sm, int ns, int band, int lane) {
    float rr = 0.0f;
#pragma unroll 2
    for (int c = 256 * band + lane; c < 256 * band + 256; c += 32) {
        const float r = narrow(residual64(sm, 5, c, ns));
        sm.r[c] = r;
        rr = fmaf(r, r, rr);
    }
    return warp_sum(rr);
}

// The residual test of pass `it`, the same in every warp; true where the stage ends.
// Its barriers are met by both roles.
struct Loop {
    double q_prev, q;
    int tests;
    bool ok;
};

template <typename Exact>
__device__ __forceinline__ bool stage_done(Team32Smem& sm, const ResidentArgs& a, int it, Loop& l, Exact exact) {
    all_sync();   // norms and QoI are in
    const Stop stop = sm.stop;
    const float rr = (sm.rr[0] + sm.rr[1]) + (sm.rr[2] + sm.rr[3]);
    l.q = sm.q;
    ++l.tests;
    bool done = rr < stop.below;
    if (!done && !(rr > stop.above)) {   // next to the limit: the FP64 sum
        exact();
        all_sync();
        done = (sm.r2[0] + sm.r2[1]) + (sm.r2[2] + sm.r2[3]) <= stop.limit;
    }
    if (done || (a.qtol > 0 && fabs(l.q - l.q_prev) <= a.qtol * fabs(l.q))) return true;
    l.q_prev = l.q;
    l.ok = it < a.max_cycles;
    return !l.ok;
}

__device__ __forceinline__ void band_role(const ResidentArgs& a, size_t s, const Ghost<float>& td,
                                          const Ghost<float>& zero, Team32Smem& sm, int warp, int lane) {
    const double* K = a.K + s * 1024;
    const int cx = lane & 15, row0 = 8 * warp + 4 * (lane >> 4);
    Band g;
    if (threadIdx.x == 0) sm.bad = 0;
    band_faces(K, a.bd.ns, sm, warp, lane);
    band_load(sm, g, warp, lane);
    if (warp == 0) {
        const Stop stop = stage_limit(sm, 32, a.bd, a.tol, lane);
        if (lane == 0) sm.stop = stop;
    }
    all_sync();   // the 16 x 16 solution is there
    if (a.qc != nullptr) {
        band_interpolate(sm, a.bd, warp, lane);
    } else {
        prolong32(g, sm, td, false, true, warp, lane);
#pragma unroll
        for (int y = 0; y < 4; ++y)
#pragma unroll
            for (int x = 0; x < 2; ++x) sm.p[32 * (row0 + y) + 2 * cx + x] = widen(g.p[y][x]);
    }
    all_sync();
    Loop l{NAN, NAN, 0, true};
    // FP64 residual -> FP32 V-cycles on the correction -> FP64 update
#pragma unroll 1
    for (int it = 0; !sm.bad; ++it) {
        const float rr = band_residual(sm, a.bd.ns, warp, lane);
        if (lane == 0) sm.rr[warp] = rr;
        const bool done = stage_done(sm, a, it, l, [&] {
            double r2 = 0.0;
#pragma unroll 1
            for (int c = 256 * warp + lane; c < 256 * warp + 256; c += 32) {
                const double v = residual64(sm, 5, c, a.bd.ns);
                r2 = fma(v, v, r2);
            }
            r2 = warp_sum(r2);
            if (lane == 0) sm.r2[warp] = r2;
        });
        if (done) break;
#pragma unroll
        for (int y = 0; y < 4; ++y) {
            const float2 v = *reinterpret_cast<const float2*>(sm.r + 32 * (row0 + y) + 2 * cx);
            g.b[y][0] = v.x;
            g.b[y][1] = v.y;
            g.p[y][0] = g.p[y][1] = 0.0f;
        }
        publish(g, sm, warp, lane);
#pragma unroll 1
        for (int v = 0; v < a.ir; ++v) band_vcycle<kResident32>(g, sm, a.nu1, a.nu2, zero, warp, lane);
        bool finite = true;
#pragma unroll
        for (int y = 0; y < 4; ++y) {
            finite = finite && isfinite(g.p[y][0]) && isfinite(g.p[y][1]);
            *reinterpret_cast<float2*>(sm.r + 32 * (row0 + y) + 2 * cx) = make_float2(g.p[y][0], g.p[y][1]);
        }
        if (!finite) sm.bad = 1;
        __syncwarp();
#pragma unroll 2
        for (int c = 256 * warp + lane; c < 256 * warp + 256; c += 32) sm.p[c] += widen(sm.r[c]);
        all_sync();
    }
    if (a.p_out)
        for (int c = threadIdx.x; c < 1024; c += 128) a.p_out[s * 1024 + c] = sm.p[c];
}

__device__ __forceinline__ void coarse_role(const ResidentArgs& a, size_t s, const Ghost<float>& td,
                                            const Ghost<float>& zero, Team32Smem& sm, int lane) {
    const double* K = a.K + s * 1024;
    G8 g8;
    G16 g16;
    const Stages low = coarse_stages<5>(a, K, g8, g16, sm.w16, td, zero, lane);
    if (a.qc == nullptr) {
#pragma unroll
        for (int y = 0; y < 4; ++y)
            *reinterpret_cast<float2*>(sm.c16 + 16 * (4 * (lane >> 3) + y) + 2 * (lane & 7)) =
                make_float2(g16.p[y][0], g16.p[y][1]);
    }
    all_sync();
    if (lane == 0 && !low.finite) sm.bad = 1;
    // from here on the 16 x 16 grid carries corrections
    faces32<5>(K, 4, true, a.bd.ns, sm.w16, reinterpret_cast<float*>(sm.w16.te), lane);
    load16(sm.w16.faces, g16, sm.w16, lane);
    all_sync();
    Loop l{NAN, NAN, 0, true};
    int cycles = 0;
#pragma unroll 1
    for (int it = 0; !sm.bad; ++it) {
        const double v = qoi(sm, 32, a.bd, lane);
        if (lane == 0) sm.q = v;
        if (stage_done(sm, a, it, l, [] {})) break;
        cycles += a.ir;
#pragma unroll 1
        for (int v = 0; v < a.ir; ++v) coarse_vcycle<kResident32>(g16, g8, sm, sm.w16, a.nu1, a.nu2, zero, lane);
        all_sync();   // the update is done
    }
    if (lane == 0) {
        const bool bad = sm.bad != 0;
        if (a.flops && !bad) {   // the counts of fmg_resident.cu
            const int t[3] = {low.tests[0], low.tests[1], l.tests}, n[3] = {low.cycles[0], low.cycles[1], cycles};
            double work = 0.0, work64 = 0.0, model = 0.0;
            for (int k = 0; k < 3; ++k) {
                const double c = 64 << 2 * k, updates = t[k] ? t[k] - 1.0 : 0.0;
                work64 += c * (14.0 * t[k] + updates);
                model += c * 20.0 * t[k] + n[k] * vcycle_bytes(4, 1 + k, a.nu1, a.nu2, 4);
                work += n[k] * vcycle_flops(4, 1 + k, a.nu1, a.nu2);
            }
            atomicAdd(a.flops, work + work64);
            atomicAdd(a.flops + 1, work64);
            atomicAdd(a.flops + 2, model);
        }
        a.qf[s] = bad ? __longlong_as_double(kAgain) : l.q;
        if (a.qc) a.qc[s] = low.q[1];
        if (a.status) a.status[s] = l.ok && low.ok ? FM_OK : FM_ENOTCONV;
    }
}

struct Tail32Smem : Borders {
    CoarseSmem coarse;
};

// A correction operator in memory -> the 16 x 16 and 8 x 8 grids' registers.
__device__ __forceinline__ void operator16(const float* __restrict__ Te, const float* __restrict__ Tn,
                                           const float* __restrict__ D, G16& g, CoarseSmem& sm, int lane) {
    const int cx = lane & 7, ry = lane >> 3;
#pragma unroll
    for (int y = 0; y < 4; ++y) {
        const int j = 4 * ry + y, c = 16 * j + 2 * cx;
        const float2 e = *reinterpret_cast<const float2*>(Te + c), t = *reinterpret_cast<const float2*>(Tn + c);
        const float2 d = *reinterpret_cast<const float2*>(D + c);
        const float w = up1(e.y);
        sm.df[2 * y][lane] = d.x;
        sm.df[2 * y + 1][lane] = d.y;
        g.rd[y][0] = recip(d.x);
        g.rd[y][1] = recip(d.y);
        g.w[y] = cx > 0 ? w : 0.0f;
        g.ei[y] = e.x;
        g.ee[y] = cx < 7 ? e.y : 0.0f;
        g.nf[y][0] = j < 15 ? t.x : 0.0f;
        g.nf[y][1] = j < 15 ? t.y : 0.0f;
    }
#pragma unroll
    for (int x = 0; x < 2; ++x) {
        const float s = __shfl_up_sync(kAll, g.nf[3][x], 8);
        g.sf[x] = ry > 0 ? s : 0.0f;
    }
}

__device__ __forceinline__ void operator8(const float* __restrict__ Te, const float* __restrict__ Tn,
                                          const float* __restrict__ D, G8& g, int lane) {
    const int bx = lane & 3, by = (lane >> 2) & 3;
    float t[2][2];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const int c = 8 * (2 * by + q) + 2 * bx;
        const float2 e = *reinterpret_cast<const float2*>(Te + c), n = *reinterpret_cast<const float2*>(Tn + c);
        const float2 d = *reinterpret_cast<const float2*>(D + c);
        const float w = lf(e.y);
        g.w[q] = bx > 0 ? w : 0.0f;
        g.ei[q] = e.x;
        g.ee[q] = bx < 3 ? e.y : 0.0f;
        t[q][0] = n.x;
        t[q][1] = n.y;
        g.d[q][0] = d.x;
        g.d[q][1] = d.y;
        g.rd[q][0] = recip(d.x);
        g.rd[q][1] = recip(d.y);
    }
#pragma unroll
    for (int x = 0; x < 2; ++x) {
        const float s = be(t[1][x]);
        g.sf[x] = by > 0 ? s : 0.0f;
        g.ni[x] = t[0][x];
        g.nn[x] = by < 3 ? t[1][x] : 0.0f;
    }
}

}  // namespace

__global__ void __launch_bounds__(kTeam, 3) k_fmg_team32(ResidentArgs a) {
    extern __shared__ __align__(16) unsigned char team_smem[];
    Team32Smem& sm = *reinterpret_cast<Team32Smem*>(team_smem);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const Ghost<float> td{(float)a.bd.w, (float)a.bd.e, (float)a.bd.s, (float)a.bd.n, a.bd.ns};
    const Ghost<float> zero{0.0f, 0.0f, 0.0f, 0.0f, a.bd.ns};
    if (warp < 4) {
#pragma unroll 1
        for (size_t s = blockIdx.x; s < a.S; s += gridDim.x) {
            band_role(a, s, td, zero, sm, warp, lane);
            all_sync();
        }
    } else {
#pragma unroll 1
        for (size_t s = blockIdx.x; s < a.S; s += gridDim.x) {
            coarse_role(a, s, td, zero, sm, lane);
            all_sync();
        }
    }
}

// The V-cycle of the level-wise schedule from a 32 x 32 correction grid down to
// 4 x 4, from a zero iterate: k_vcycle_tail's arithmetic, one sample a CTA.  Bound by
// the chain of half-sweeps (eight of 32 x 32 at a barrier each, as many of each grid
// below in one warp); the shared-memory form issues nine loads an update.  A solve
// of 1000 samples of 256 x 256: 62 launches of 25.7 us on average, now 12.5.
__global__ void __launch_bounds__(kTeam, 3) k_vcycle_tail32(Tail32Args a) {
    __shared__ Tail32Smem sm;
    const size_t s = a.order ? (size_t)a.order[blockIdx.x] : blockIdx.x;
    if (a.active && !a.active[s]) return;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const Ghost<float> zero{0.0f, 0.0f, 0.0f, 0.0f, a.ns};
    if (warp == 4) {
        G8 g8;
        G16 g16;
        const float* A = a.Ainv + s * 256;
#pragma unroll
        for (int q = 0; q < 2; ++q) {   // 16 rows of 16
            const int e = 4 * (lane + 32 * q);
            *reinterpret_cast<float4*>(&sm.coarse.ainv[e >> 4][e & 15]) = *reinterpret_cast<const float4*>(A + e);
        }
        operator8(a.Te[0] + s * 64, a.Tn[0] + s * 64, a.D[0] + s * 64, g8, lane);
        operator16(a.Te[1] + s * 256, a.Tn[1] + s * 256, a.D[1] + s * 256, g16, sm.coarse, lane);
        __syncwarp();
        coarse_vcycle<kLevelwise>(g16, g8, sm, sm.coarse, a.nu1, a.nu2, zero, lane);
        return;
    }
    const int cx = lane & 15, row0 = 8 * warp + 4 * (lane >> 4);
    const float* te = a.Te[2] + s * 1024;
    const float* tn = a.Tn[2] + s * 1024;
    const float* dd = a.D[2] + s * 1024;
    Band g;
#pragma unroll
    for (int y = 0; y < 4; ++y) {
        const int j = row0 + y, c = 32 * j + 2 * cx;
        const float2 e = *reinterpret_cast<const float2*>(te + c), t = *reinterpret_cast<const float2*>(tn + c);
        const float2 d = *reinterpret_cast<const float2*>(dd + c);
        const float2 b = *reinterpret_cast<const float2*>(a.b + s * 1024 + c);
        const float w = up1(e.y);
        g.d[y][0] = d.x;
        g.d[y][1] = d.y;
        g.rd[y][0] = recip(d.x);
        g.rd[y][1] = recip(d.y);
        g.b[y][0] = b.x;
        g.b[y][1] = b.y;
        g.p[y][0] = g.p[y][1] = 0.0f;
        g.w[y] = cx > 0 ? w : 0.0f;
        g.ei[y] = e.x;
        g.ee[y] = cx < 15 ? e.y : 0.0f;
        g.nf[y][0] = j < 31 ? t.x : 0.0f;
        g.nf[y][1] = j < 31 ? t.y : 0.0f;
        if (y == 0) {
            const float2 u = j > 0 ? *reinterpret_cast<const float2*>(tn + c - 32) : make_float2(0.0f, 0.0f);
            g.sf[0] = u.x;
            g.sf[1] = u.y;
        }
    }
    publish(g, sm, warp, lane);
    band_vcycle<kLevelwise>(g, sm, a.nu1, a.nu2, zero, warp, lane);
#pragma unroll
    for (int y = 0; y < 4; ++y)
        *reinterpret_cast<float2*>(a.p + s * 1024 + 32 * (row0 + y) + 2 * cx) = make_float2(g.p[y][0], g.p[y][1]);
}

void launch_tail32(const Tail32Args& a, size_t S, cudaStream_t st) {
    k_vcycle_tail32<<<(unsigned)S, kTeam, 0, st>>>(a);
}

void team32_init() {
    constexpr size_t smem = sizeof(Team32Smem);
    cudaFuncSetAttribute(k_fmg_team32, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
}

void launch_team32(fm_ctx* ctx, const ResidentArgs& a, cudaStream_t st) {
    constexpr size_t smem = sizeof(Team32Smem);
    int per_sm = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_fmg_team32, kTeam, smem);
    const size_t grid = std::min<size_t>(a.S, (size_t)std::max(per_sm, 1) * std::max(ctx->sms, 1));
    k_fmg_team32<<<(unsigned)grid, kTeam, smem, st>>>(a);
}

}  // namespace fm
