// The column-strip smoother's kernel and its launch (instantiated per
// arithmetic in fmg_strip_f32.cu and fmg_strip_f64.cu).
//
// nsweeps red-black sweeps (HS = 2 nsweeps half-sweeps) marching up the rows
// of one sample.  A warp covers 64 columns: lane l owns columns 2l, 2l+1, so
// in every row it holds one cell of each colour; W / E neighbours in other
// lanes come by warp shuffles, N / S neighbours from the rows the lane keeps
// in registers.  At step y the warp takes in row y and runs half-sweep k on
// row y - k for k = 1 .. HS: row y - k + 1 has just had half-sweep k - 1 and
// row y - k - 1 had half-sweep k one step earlier, so every update sees the
// values the sweep order prescribes, and row y - HS is final and is written.
// The HS + 2 rows in flight stay in registers (a ring whose slots are fixed
// by the unrolled step index); the rows ahead arrive through a per-warp
// shared-memory ring of as many rows filled by cp.async (each lane copies
// and reads back only its own pairs, so its slot index is a constant too).
//
// Columns: a group of W = 1 .. 4 warps covers 64 W adjacent columns and
// steps in lockstep (one named barrier a row); the columns on both sides of
// a warp border are exchanged through shared memory after every row, so a
// grid of up to 256 columns is covered exactly once, with no halo.  Wider
// grids take several overlapping windows (XH halo columns on inner sides).
// Grids of 16 and 32 columns pack 64 / n samples into a warp.  Without the
// groups a 128-column grid cost three 64-column windows and a 64-column one
// two: half to a third of the lanes did nothing that was kept.
//
// Halo cells (window and segment edges) are updated with whatever their
// missing neighbours read as; what is wrong moves one cell per half-sweep,
// so it never reaches the cells written.  At domain edges the face is zero.
// No update is masked: a half-sweep is one shuffle, four FMAs, one product.
//
// Arithmetic as in the colour kernel: p = (b + W + E + S + N) (1 / D) with
// the reciprocal of D (FP32: rcp.approx and one Newton step, which gives the
// correctly rounded 1 / D for every D from 2^-126 up to 2^126, as
// tests/test_gpu_short_functions.py walks through; FP64: read from rD, formed
// once at set-up, since an FP64 reciprocal costs more than a half-sweep's five
// FP64 operations), so the sweeps are bit-identical to the other shapes (FP32 diagonals
// outside that range, where 1 / D is no normal number, or D none, excepted).
//
// FUSE: the warp also forms the residual b - A p of each final row once the
// row above it is final, and its restriction: the lane's column pair is one
// coarse column, so it sums four fine residuals over two rows in
// k_residual_restrict's order and writes b_c.  D of that row comes from a
// shared-memory ring twice as deep.  EC: the iterate is p_in + P ec, the
// coarse row that a fine row needs coming through a ring of its own.
// EC + FUSE with HS = 8 is the post-smoothing of one V-cycle and the
// pre-smoothing of the next in one pass over memory.
//
// Bound and measured, 1000 FP32 samples (GB300, in a converged solve):
//   256 x 256: pre-smoothing from zero 266 us (5.4 TB/s; with three to five
//     overlapping one-warp windows, the zero iterate read and an IEEE
//     division per cell it took 607), post-smoothing 291 (453; 5.6 TB/s),
//     both in one pass 560, against 600 one after the other: HBM bounds the
//     first two, instruction issue (256 a row of 64 columns) the merged one;
//   128 x 128: 76 (193), 85 (169) and 144; 64 x 64: 25 (61) and 23 (55).
// The merged kernel needs 207 registers: held to 168 (three CTAs an SM) it
// spilled and took 384 us where it takes 144.
#pragma once

#include <algorithm>
#include <cmath>

#include "fmg_strip.cuh"

namespace fm {

constexpr int kStripMaxWarps = 4;

template <typename T>
struct Pair;
template <>
struct Pair<float> {
    using type = float2;
};
template <>
struct Pair<double> {
    using type = double2;
};

// Asynchronous global -> shared copies of B = 4, 8 or 16 bytes (cp.async, both
// addresses B-aligned), commit groups, and the wait until at most N groups
// of this thread are still in flight.
template <int B>
__device__ __forceinline__ void cp_async(void* smem, const void* gmem) {
    static_assert(B == 4 || B == 8 || B == 16, "cp.async of 4, 8 or 16 bytes");
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"((uint32_t)__cvta_generic_to_shared(smem)),
                 "l"(gmem), "n"(B)
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// 1 / d, correctly rounded where 1 / d is a normal number (see above).
__device__ __forceinline__ float strip_recip(float d) {
    float r;
    asm("rcp.approx.f32 %0, %1;" : "=f"(r) : "f"(d));
    return fmaf(r, fmaf(-d, r, 1.0f), r);
}

template <typename T>
struct StripArgs {
    int n, W, nwin, seg, segs, resident;   // resident: groups in flight on the whole GPU
    int lgn;                               // PACK: log2 n
    size_t S;
    size_t head;                           // packs in segments of seg rows; those after them in segments of seg2
    int seg2, segs2;
    const T *b, *Te, *Tn, *D, *rD, *p_in;
    T* p_out;
    const int32_t* active;
    const T* ec;
    T *bc, *pc;
    const int32_t* order;
    const int32_t* dcount;
    int ns;
};

// Halo columns and rows (even: rows and columns go in pairs).
__host__ __device__ constexpr int strip_halo(int HS, bool fuse) { return fuse ? HS + 2 : HS; }

// Rows of the shortest segments (even, at least 16 or the grid) with which
// `units` strips of n rows still go into one wave of `resident` groups.
__host__ __device__ inline int strip_fill(int n, size_t units, size_t resident) {
    const int k = (int)(resident / (units > 0 ? units : 1));
    const int seg = k > 1 ? ((n + k - 1) / k + 1) / 2 * 2 : n;
    return seg < 16 ? (n < 16 ? n : 16) : seg < n ? seg : n;
}

// Shared memory of one warp.
template <typename T, int HS, bool FUSE, bool EC>
struct StripSmem {
    using V2 = typename Pair<T>::type;
    static constexpr int R = HS + 2;
    static constexpr bool kF32 = sizeof(T) == 4;
    V2 ring[R][4][32];                                   // p, b, Te, Tn
    V2 dring[kF32 ? (FUSE ? 2 * R : R) : (FUSE ? 2 * R : 1)][32];   // D
    V2 rring[kF32 ? 1 : R][32];                          // FP64: 1 / D
    T cring[EC ? R / 2 : 1][36];                         // coarse rows: [0] left of lane 0, [1 + l], [33]
    T wring[R];                                          // the west face of lane 0's left cell
    T xch[2][2][HS + 2];                                 // [side][buffer]: the border column's rows
};

template <typename T, int HS, bool FUSE, bool EC>
__host__ __device__ constexpr int strip_min_blocks() {
    return sizeof(T) == 4 ? (HS <= 4 ? (FUSE && EC ? 3 : 4) : 2) : 2;
}

template <typename T, int HS, bool FUSE, bool EC, bool PACK>
__global__ void __launch_bounds__(32 * kStripMaxWarps, (strip_min_blocks<T, HS, FUSE, EC>()))
    k_rbgs_strip(const StripArgs<T> a) {
    using V2 = typename Pair<T>::type;
    using SM = StripSmem<T, HS, FUSE, EC>;
    constexpr int R = HS + 2;
    constexpr int XH = strip_halo(HS, FUSE);
    constexpr bool kF32 = sizeof(T) == 4;
    constexpr unsigned kAll = 0xffffffffu;
    static_assert(HS % 2 == 0 && XH % 2 == 0, "even half-sweep count and halos");
    extern __shared__ __align__(16) unsigned char strip_smem[];
    SM* const smem = reinterpret_cast<SM*>(strip_smem);

    const int n = a.n, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int W = PACK ? 1 : a.W, grp = warp / W, wig = warp - grp * W;
    SM& sm = smem[warp];
    // the samples enumerated and their row segments: as launched, or (dcount:
    // inside a device-side refinement loop) the count of listed samples the
    // last residual test left, with segments short enough to fill one wave
    // of groups when those samples are few
    const int pk = PACK ? 64 >> a.lgn : 1;
    size_t S = a.S, head = a.head;
    int seg = a.seg, segs = a.segs;
    if (a.dcount) S = (size_t)*a.dcount;
    const size_t packs = (S + pk - 1) / pk;
    if (a.dcount) {
        head = packs;
        if (packs > 0 && packs * a.nwin < (size_t)a.resident) {
            seg = strip_fill(n, packs * a.nwin, (size_t)a.resident);
            segs = (n + seg - 1) / seg;
        }
    }
    const size_t unit = (size_t)blockIdx.x * (blockDim.x / (32 * W)) + grp;
    const int win = (int)(unit % a.nwin);
    size_t rest = unit / a.nwin, pack0 = 0;   // unit of the window's row of packs and segments
    if (rest >= head * (size_t)segs) {
        rest -= head * (size_t)segs;
        pack0 = head;
        seg = a.seg2;
        segs = a.segs2;
        if (rest >= (packs - head) * (size_t)segs) return;
    }
    const int sy = (int)(rest % segs);
    const int gw = 64 * W;                              // columns of the group's window
    const int wx = win * (gw - 2 * XH);                 // its first column
    const int gx = PACK ? (2 * lane) & (n - 1) : wx + 64 * wig + 2 * lane;   // the lane's first column
    const size_t si = PACK ? (pack0 + rest / segs) * pk + ((2 * lane) >> a.lgn) : pack0 + rest / segs;
    bool in_x = gx < n;
    size_t s = 0;
    if (PACK) {
        in_x = si < S;
        if (in_x) s = a.order ? (size_t)a.order[si] : si;
        if (in_x && a.active && !a.active[s]) in_x = false;
    } else {
        s = a.order ? (size_t)a.order[si] : si;
        if (a.active && !a.active[s]) return;
    }
    const int oy = sy * seg, oye = min(oy + seg, n);
    const int ys = max(oy - XH, 0), ye = min(oye + XH, n);   // rows taken in; ys even
    const int ox = win == 0 ? 0 : wx + XH, oxe = wx + gw >= n ? n : wx + gw - XH;
    const bool out_x = in_x && (PACK || (gx >= ox && gx < oxe));
    const bool first = gx == 0;                              // no west face
    const bool last = gx + 1 >= n - 1;                       // no east face
    const bool left = !PACK && lane == 0 && wig > 0;         // west neighbour in the group's warp to the left
    const bool right = !PACK && lane == 31 && wig < W - 1;
    const size_t base = s * (size_t)n * n + gx;
    const int nc = n / 2, I = gx >> 1;                       // the lane's coarse column
    const T* const ecs = EC ? a.ec + s * (size_t)nc * nc + I : nullptr;
    const bool has_p = a.p_in != nullptr;

    // neutral operands (a zero iterate, no faces, D = 1): columns outside the
    // domain keep them, rows above the segment get them when their turn comes
    auto neutral = [&](int slot, int dslot) {
        const V2 z{T(0), T(0)}, o{T(1), T(1)};
#pragma unroll
        for (int q = 0; q < 4; ++q) sm.ring[slot][q][lane] = z;
        if (kF32 || FUSE) sm.dring[dslot][lane] = o;
        if (!kF32) sm.rring[slot][lane] = o;
        if (left) sm.wring[slot] = T(0);
    };
    // row y into ring slot `slot` (D: dslot), with EC on odd y coarse row
    // min((y + 1) / 2, nc - 1), the highest one fine rows y and y + 1 need;
    // every step commits one group
    auto fetch = [&](int y, int slot, int dslot, bool odd) {
        if (y < ye) {
            if (in_x) {
                const size_t g = base + (size_t)(unsigned)y * (unsigned)n;
                constexpr int B = (int)sizeof(V2);
                if (has_p) cp_async<B>(&sm.ring[slot][0][lane], a.p_in + g);
                cp_async<B>(&sm.ring[slot][1][lane], a.b + g);
                cp_async<B>(&sm.ring[slot][2][lane], a.Te + g);
                cp_async<B>(&sm.ring[slot][3][lane], a.Tn + g);
                if (kF32 || FUSE) cp_async<B>(&sm.dring[dslot][lane], a.D + g);
                if (!kF32) cp_async<B>(&sm.rring[slot][lane], a.rD + g);
                if (left) cp_async<(int)sizeof(T)>(&sm.wring[slot], a.Te + g - 1);
            }
            if (EC && odd) {
                const T* crow = ecs + (size_t)min((y + 1) >> 1, nc - 1) * nc;
                T* cr = sm.cring[slot >> 1];
                if (in_x) cp_async<(int)sizeof(T)>(&cr[1 + lane], crow);
                if (!PACK && in_x && lane == 0 && I > 0) cp_async<(int)sizeof(T)>(&cr[0], crow - 1);
                if (!PACK && in_x && lane == 31 && I + 1 < nc) cp_async<(int)sizeof(T)>(&cr[33], crow + 1);
            }
        } else if (in_x) {
            neutral(slot, dslot);
        }
        cp_async_commit();
    };
    // EC: own, left and right values of coarse rows y / 2 - 1, y / 2 and
    // (y + 1) / 2 with the error's ghosts: -own across the west and east
    // Dirichlet edges; past the south / north edge the edge row itself across a
    // no-flow edge, its negative across a Dirichlet one (ns)
    T cm[3] = {T(0), T(0), T(0)}, c0[3] = {T(0), T(0), T(0)}, cp[3] = {T(0), T(0), T(0)};
    const bool sg = a.ns != 0;
    auto coarse3 = [&](T own, T lf, T rt, T (&dst)[3]) {
        dst[0] = own;
        dst[1] = I == 0 ? flip_if(true, own) : lf;
        dst[2] = I == nc - 1 ? flip_if(true, own) : rt;
    };
    if (EC && in_x) {   // coarse rows ys / 2 - 1 and ys / 2 around fine row ys
        const T* crow = ecs + (size_t)(ys / 2) * nc;
        coarse3(crow[0], I > 0 ? crow[-1] : T(0), I + 1 < nc ? crow[1] : T(0), c0);
#pragma unroll
        for (int q = 0; q < 3; ++q) cm[q] = flip_if(sg, c0[q]);
        if (ys > 0) {
            crow -= nc;
            coarse3(crow[0], I > 0 ? crow[-1] : T(0), I + 1 < nc ? crow[1] : T(0), cm);
        }
    }
    T p[R][2], bb[R][2], rr[R][2], ee[R][2], nf[R][2], wl[R];
#pragma unroll
    for (int c = 0; c < R; ++c) {
        p[c][0] = p[c][1] = bb[c][0] = bb[c][1] = ee[c][0] = ee[c][1] = nf[c][0] = nf[c][1] = wl[c] = T(0);
        rr[c][0] = rr[c][1] = T(0);
    }
    // FUSE: the row leaving the ring (p and north faces) and the partial coarse sum
    T pq[2] = {T(0), T(0)}, nq[2] = {T(0), T(0)}, rsum = T(0);
    if (!in_x) {
#pragma unroll
        for (int q = 0; q < R; ++q) {
            neutral(q, q);
            if (FUSE) neutral(q, R + q);
        }
    } else if (!has_p) {
#pragma unroll
        for (int q = 0; q < R; ++q) sm.ring[q][0][lane] = V2{T(0), T(0)};
    }
#pragma unroll
    for (int q = 0; q < R; ++q) fetch(ys + q, q, q, q & 1);
    if (W > 1) {   // the rows below the first one read as zero on both sides
        if (lane < HS + 2) {
#pragma unroll
            for (int q = 0; q < 4; ++q) sm.xch[q >> 1][q & 1][lane] = T(0);
        }
        asm volatile("bar.sync %0, %1;" ::"r"(grp + 1), "r"(32 * W) : "memory");
    }
    const SM& sl = smem[warp - (wig > 0 ? 1 : 0)];
    const SM& sr = smem[warp + (wig < W - 1 ? 1 : 0)];
    const int yend = ye + HS + (FUSE ? 1 : 0);
    int half = 0;   // the half of the D ring that holds rows y0 .. y0 + R - 1
    for (int y0 = ys; y0 < yend; y0 += R, half ^= 1) {
#pragma unroll
        for (int J = 0; J < R; ++J) {
            const int y = y0 + J;
            if (y >= yend) break;
            // The neighbours in other lanes, all shuffled before the first update: the
            // half-sweeps of a step change one colour and read the other, so what
            // they take from other lanes is what the previous step left.  Only
            // the north neighbour of each update is new, a chain of one FMA and
            // one product per half-sweep.  Border columns of the neighbouring
            // warps as published after step y - 1.
            const T* const xl = sl.xch[1][((y - 1) >> 1) & 1];
            const T* const xr = sr.xch[0][((y - 1) >> 1) & 1];
            T side[HS];
#pragma unroll
            for (int k = 1; k <= HS; ++k) {
                const int c = (J - k + 4 * R) % R;
                if (J & 1) {
                    side[k - 1] = __shfl_up_sync(kAll, p[c][1], 1);
                    if (left) side[k - 1] = xl[k - 1];
                    if (PACK && first) side[k - 1] = T(0);   // the left lane holds another sample
                } else {
                    side[k - 1] = __shfl_down_sync(kAll, p[c][0], 1);
                    if (right) side[k - 1] = xr[k - 1];
                    if (PACK && last) side[k - 1] = T(0);
                }
            }
            // FUSE: both neighbours of row q = y - HS - 1, final since step y - 1; the
            // side that step y - 1 did not change was published after step y - 2
            T qw = T(0), qe = T(0);
            if (FUSE) {
                const int c = (J - HS - 1 + 4 * R) % R;
                qw = __shfl_up_sync(kAll, p[c][1], 1);
                qe = __shfl_down_sync(kAll, p[c][0], 1);
                if (left) qw = (J & 1) ? xl[HS] : sl.xch[1][((y - 2) >> 1) & 1][HS - 1];
                if (right) qe = (J & 1) ? sr.xch[0][((y - 2) >> 1) & 1][HS - 1] : xr[HS];
                if (PACK && first) qw = T(0);
                if (PACK && last) qe = T(0);
            }
            if (FUSE) {   // keep row y - R (the S neighbour of the residual row y - HS - 1)
                pq[0] = p[J][0];
                pq[1] = p[J][1];
                nq[0] = nf[J][0];
                nq[1] = nf[J][1];
            }
            {   // take in row y (register slot J), then start the copy of row y + R
                cp_async_wait<R - 1>();   // this lane's copies of row y have landed
                const V2 fp = sm.ring[J][0][lane], fb = sm.ring[J][1][lane];
                const V2 fe = sm.ring[J][2][lane], fn = sm.ring[J][3][lane];
                T a0 = fp.x, a1 = fp.y;
                if (EC) {   // the coarse-grid correction p + (P e) as k_prolong forms it
                    if (J & 1) {
                        __syncwarp();   // the neighbouring lanes' coarse copies have landed too
                        const T* cr = sm.cring[J >> 1];
                        coarse3(cr[1 + lane], cr[lane], cr[2 + lane], cp);
                        __syncwarp();   // every lane has read the slot before it is refilled
                        if (y == n - 1) {
#pragma unroll
                            for (int q = 0; q < 3; ++q) cp[q] = flip_if(sg, c0[q]);
                        }
                    }
                    // fine row y: coarse row y / 2 and its y neighbour, one row down for
                    // even y, one up for odd y.  Black cells only: the first half-sweep
                    // replaces the red ones from their black neighbours.
                    if (in_x && y < ye) {
                        if (J & 1) a0 = add_rn(a0, prolong_vals(c0[0], c0[1], cp[0], cp[1]));
                        else a1 = add_rn(a1, prolong_vals(c0[0], c0[2], cm[0], cm[2]));
                    }
                    if (J & 1) {
#pragma unroll
                        for (int q = 0; q < 3; ++q) {
                            cm[q] = c0[q];
                            c0[q] = cp[q];
                        }
                    }
                }
                p[J][0] = a0;
                p[J][1] = a1;
                bb[J][0] = fb.x;
                bb[J][1] = fb.y;
                if constexpr (kF32) {
                    const V2 fd = sm.dring[FUSE ? half * R + J : J][lane];
                    rr[J][0] = strip_recip(fd.x);
                    rr[J][1] = strip_recip(fd.y);
                } else {
                    const V2 fr = sm.rring[J][lane];
                    rr[J][0] = fr.x;
                    rr[J][1] = fr.y;
                }
                ee[J][0] = fe.x;
                ee[J][1] = last ? T(0) : fe.y;
                nf[J][0] = y < n - 1 ? fn.x : T(0);
                nf[J][1] = y < n - 1 ? fn.y : T(0);
                wl[J] = __shfl_up_sync(kAll, fe.y, 1);   // W face: the left cell's east face
                if (left) wl[J] = sm.wring[J];
                if (first) wl[J] = T(0);
                fetch(y + R, J, FUSE ? (half ^ 1) * R + J : J, J & 1);
            }
#pragma unroll
            for (int k = 1; k <= HS; ++k) {
                // half-sweep k (colour (k - 1) & 1) on row r = y - k: the left cell
                // (even column) has that colour iff y is odd
                const int c = (J - k + 4 * R) % R, lo = (J - k - 1 + 4 * R) % R, hi = (J - k + 1 + 4 * R) % R;
                if (J & 1) {
                    T acc = bb[c][0];
                    acc = fma(wl[c], side[k - 1], acc);
                    acc = fma(ee[c][0], p[c][1], acc);
                    acc = fma(nf[lo][0], p[lo][0], acc);
                    acc = fma(nf[c][0], p[hi][0], acc);
                    p[c][0] = mul_rn(acc, rr[c][0]);
                } else {
                    T acc = bb[c][1];
                    acc = fma(ee[c][0], p[c][0], acc);
                    acc = fma(ee[c][1], side[k - 1], acc);
                    acc = fma(nf[lo][1], p[lo][1], acc);
                    acc = fma(nf[c][1], p[hi][1], acc);
                    p[c][1] = mul_rn(acc, rr[c][1]);
                }
            }
            {
                const int r = y - HS;
                if (out_x && r >= oy && r < oye) {
                    const int c = (J - HS + 4 * R) % R;
                    *reinterpret_cast<V2*>(a.p_out + base + (size_t)(unsigned)r * (unsigned)n) = V2{p[c][0], p[c][1]};
                }
            }
            if (FUSE) {
                // residual of row q = y - HS - 1 (rows q - 1, q + 1 final), as residual_at forms it
                const int q = y - HS - 1;
                const int c = (J - HS - 1 + 4 * R) % R, hi = (J - HS + 4 * R) % R;
                if (out_x && q >= oy && q < oye) {
                    const V2 dq = sm.dring[(J + 1 < R ? (half ^ 1) * R : half * R) + (J + 1) % R][lane];
                    // FP64: red cells only, a row's left one on even q (kRedOnly)
                    T r0 = T(0), r1 = T(0);
                    if (!kRedOnly<T> || (J & 1)) {
                        T v0 = mul_rn(dq.x, p[c][0]);
                        v0 = fma(-wl[c], qw, v0);
                        v0 = fma(-ee[c][0], p[c][1], v0);
                        v0 = fma(-nq[0], pq[0], v0);
                        v0 = fma(-nf[c][0], p[hi][0], v0);
                        r0 = bb[c][0] - v0;
                    }
                    if (!kRedOnly<T> || !(J & 1)) {
                        T v1 = mul_rn(dq.y, p[c][1]);
                        v1 = fma(-ee[c][0], p[c][0], v1);
                        v1 = fma(-ee[c][1], qe, v1);
                        v1 = fma(-nq[1], pq[1], v1);
                        v1 = fma(-nf[c][1], p[hi][1], v1);
                        r1 = bb[c][1] - v1;
                    }
                    if ((J & 1) == 0) {   // q odd: the coarse cell's upper row
                        const size_t cc = s * (size_t)nc * nc + (size_t)(q / 2) * nc + I;
                        a.bc[cc] = kRedOnly<T> ? rsum + r1 : rsum + r0 + r1;
                        if (a.pc) a.pc[cc] = T(0);
                    } else {
                        rsum = kRedOnly<T> ? r0 : r0 + r1;
                    }
                }
            }
            if (W > 1) {   // publish the border columns of rows y .. y - HS, then one barrier
                const int buf = (y >> 1) & 1;
                if (J & 1) {
                    if (lane == 0 && wig > 0) {
#pragma unroll
                        for (int k = 0; k <= HS; ++k) sm.xch[0][buf][k] = p[(J - k + 4 * R) % R][0];
                    }
                } else {
                    if (lane == 31 && wig < W - 1) {
#pragma unroll
                        for (int k = 0; k <= HS; ++k) sm.xch[1][buf][k] = p[(J - k + 4 * R) % R][1];
                    }
                }
                asm volatile("bar.sync %0, %1;" ::"r"(grp + 1), "r"(32 * W) : "memory");
            }
        }
    }
    cp_async_wait<0>();
}

// ------------------------------------------------------------------ launch
// Window geometry of grid n: W warps a group, nwin windows a row, the
// fewest warps a row (ties: fewer warps a group).
inline void strip_windows(int n, int XH, int* W, int* nwin) {
    int best = 1 << 30;
    for (int w = 1; w <= kStripMaxWarps; ++w) {
        const int gw = 64 * w, k = n <= gw ? 1 : 1 + (n - gw + gw - 2 * XH - 1) / (gw - 2 * XH);
        if (k * w < best) {
            best = k * w;
            *W = w;
            *nwin = k;
        }
    }
}

// How `packs` strips-of-samples of nwin windows are cut into row segments: all into
// the power-of-two fraction of n (at least 16 rows) that minimises the waves of
// units over the resident groups times the steps of one unit (segment plus halo
// rows plus the steps that drain the wavefront), or, where that is less, whole
// waves of uncut strips and one wave of the rest in segments that just fill it.
// 1000 samples of 256 x 256, 304 groups resident: four waves of 265 steps, against
// three and one of 117 (88 samples in three segments); the solve's eight-half-sweep
// passes 8.4 -> 7.7 ms.
struct StripCut {
    size_t head;     // packs in segments of seg rows; the rest in segments of seg2
    int seg, seg2;
};

inline StripCut strip_cut(int n, size_t packs, int nwin, int HS, int VH, int resident) {
    auto steps = [&](int seg) { return std::min(seg + (seg < n ? 2 * VH : 0), n) + HS + 1; };
    const size_t units1 = packs * nwin, R = (size_t)std::max(1, resident);
    StripCut best{packs, n, n};
    double best_cost = 1e300;
    for (int seg = n; seg >= 16; seg /= 2) {
        const size_t units = units1 * ((n + seg - 1) / seg);
        const double cost = std::ceil((double)units / (double)R) * steps(seg);
        if (cost < best_cost * 0.999) {
            best_cost = cost;
            best = {packs, seg, seg};
        }
        if (seg % 4) break;   // segments start on even rows
    }
    const size_t waves = units1 / R, head = std::min(packs, waves * R / nwin), rest = packs - head;
    if (rest > 0 && rest * nwin <= R) {
        const int seg2 = strip_fill(n, rest * nwin, R);
        if (waves * (double)steps(n) + steps(seg2) < best_cost * 0.98) best = {head, n, seg2};
    }
    return best;
}

// Groups per CTA: four warps, or three for W = 3.
inline int strip_groups(int W) { return W == 3 ? 1 : kStripMaxWarps / W; }

template <typename T, int HS, bool FUSE, bool EC, bool PACK>
struct StripVariant {
    static int resident[kStripMaxWarps + 1];   // groups in flight on the GPU, by W
    static size_t smem(int W) { return (size_t)W * strip_groups(W) * sizeof(StripSmem<T, HS, FUSE, EC>); }
    static void init(int sms) {
        auto k = k_rbgs_strip<T, HS, FUSE, EC, PACK>;
        cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem(4));
        for (int W = 1; W <= kStripMaxWarps; ++W) {
            int blocks = 0;
            if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, k, 32 * W * strip_groups(W), smem(W)) !=
                cudaSuccess)
                blocks = 1;
            // (the first device's count serves all: the library is built for one kind)
            if (!resident[W]) resident[W] = std::max(1, blocks) * strip_groups(W) * std::max(1, sms);
        }
    }
    static void launch(fm_ctx* ctx, const StripCall<T>& c, cudaStream_t st) {
        constexpr int VH = strip_halo(HS, FUSE);
        StripArgs<T> a{};
        a.n = c.n;
        strip_windows(c.n, VH, &a.W, &a.nwin);
        int pk = 1;
        if (PACK) {
            a.W = a.nwin = 1;
            while ((1 << a.lgn) < c.n) ++a.lgn;
            pk = 64 / c.n;
        }
        a.resident = resident[a.W];
        // with the host's count of active samples and their list, enumerate only
        // those; with a device-side count (dcount, refinement loops inside a
        // graph) the kernel enumerates the listed samples itself, and the grid
        // covers the most units it can form (all samples, or one wave)
        const bool dev = c.dcount && c.order;
        const bool listed = !dev && c.order && c.busy > 0 && c.busy < c.S;
        a.S = listed ? c.busy : c.S;
        const size_t packs = (a.S + pk - 1) / pk;
        const StripCut cut = strip_cut(c.n, packs, a.nwin, HS, VH, a.resident);
        a.head = cut.head;
        a.seg = cut.seg;
        a.segs = (c.n + a.seg - 1) / a.seg;
        a.seg2 = cut.seg2;
        a.segs2 = (c.n + a.seg2 - 1) / a.seg2;
        size_t units = (a.head * a.segs + (packs - a.head) * a.segs2) * (size_t)a.nwin;
        if (dev) units = std::max(units, (size_t)a.resident);
        a.b = c.b;
        a.Te = c.Te;
        a.Tn = c.Tn;
        a.D = c.D;
        a.rD = c.rD;
        a.p_in = c.p_in;
        a.p_out = c.p_out;
        a.active = c.active;
        a.ec = c.ec;
        a.bc = c.bc;
        a.pc = c.pc;
        a.order = (listed || dev) ? c.order : nullptr;
        a.dcount = dev ? c.dcount : nullptr;
        a.ns = c.ns;
        const int G = strip_groups(a.W);
        const unsigned grid = (unsigned)((units + G - 1) / G);
        const double cells = (double)a.S * c.n * c.n;
        const double ops = (c.p_in ? 6.0 : 5.0) + (FUSE ? 0.25 : 0.0) + (EC ? 0.25 : 0.0);
        FM_TIMED(ctx, kFamSmootherStrip, st, ops * sizeof(T) * cells, (5.0 * HS + (FUSE ? 12.0 : 0.0)) * cells,
                 k_rbgs_strip<T, HS, FUSE, EC, PACK><<<grid, 32 * a.W * G, smem(a.W), st>>>(a));
    }
};
template <typename T, int HS, bool FUSE, bool EC, bool PACK>
int StripVariant<T, HS, FUSE, EC, PACK>::resident[kStripMaxWarps + 1] = {};

// f(variant) for the variant of a call, or for every one (all).
template <typename T, int HS, bool FUSE, bool EC, typename F>
inline void strip_pick(bool pack, bool all, F f) {
    if (all || pack) f(StripVariant<T, HS, FUSE, EC, true>());
    if (all || !pack) f(StripVariant<T, HS, FUSE, EC, false>());
}
template <typename T, typename F>
inline void strip_for(int hs, bool fuse, bool ec, bool pack, bool all, F f) {
    if (all || (hs == 2 && fuse && !ec)) strip_pick<T, 2, true, false>(pack, all, f);
    if (all || (hs == 4 && fuse && !ec)) strip_pick<T, 4, true, false>(pack, all, f);
    if (all || (hs == 2 && !fuse && ec)) strip_pick<T, 2, false, true>(pack, all, f);
    if (all || (hs == 4 && !fuse && ec)) strip_pick<T, 4, false, true>(pack, all, f);
    if (all || (hs == 2 && !fuse && !ec)) strip_pick<T, 2, false, false>(pack, all, f);
    if (all || (hs == 4 && !fuse && !ec)) strip_pick<T, 4, false, false>(pack, all, f);
    if constexpr (sizeof(T) == 4) {
        if (all || (hs == 4 && fuse && ec)) strip_pick<T, 4, true, true>(pack, all, f);
        if (all || (hs == 8 && fuse && ec)) strip_pick<T, 8, true, true>(pack, all, f);
        if (all || (hs == 8 && fuse && !ec)) strip_pick<T, 8, true, false>(pack, all, f);
    }
}

template <typename T>
void strip_launch(fm_ctx* ctx, const StripCall<T>& c, cudaStream_t st) {
    const bool pack = c.n <= 32 && (c.n & (c.n - 1)) == 0;
    strip_for<T>(c.hs, c.fuse, c.ec != nullptr, pack, false, [&](auto v) { v.launch(ctx, c, st); });
}

template <typename T>
void strip_init(int sms) {
    strip_for<T>(0, false, false, false, true, [&](auto v) { v.init(sms); });
}

}  // namespace fm
