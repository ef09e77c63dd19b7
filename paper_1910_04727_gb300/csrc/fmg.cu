// Batched full multigrid for the Case II Darcy problem (Eq. 1, Table 1,
// Sec. 2.5), level-wise schedule: one FMG hierarchy per sample, all samples
// of a batch advanced together, every kernel covering every cell of every
// (active) sample of one grid, x fastest so a warp touches consecutive cells
// of one row.  Used for grids whose hierarchy does not fit in one CTA's
// shared memory (n > 64); smaller grids take the resident schedule.
//
// Per grid k (n_k = n_coarsest << k) and sample the scratch holds
//   K   FP64 coefficients (injected from the finer grid; the finest is the input)
//   Te  east-face transmissibility of each cell (2K on the east edge)
//   Tn  north-face transmissibility (0 on the north edge)
//   D   diagonal: sum of the four face transmissibilities (2K on the west edge)
//   p   iterate, b right-hand side
// in the V-cycle type T (FP64, or FP32 in the mixed form), and for the
// coarsest grid the inverse of its dense operator, so each exact solve is a
// small matrix-vector product.  The mixed form adds FP64 p, Te, Tn, D on the
// two refined grids (n/2 and n, which give Q^c and Q^f).
#include <algorithm>
#include <cmath>
#include <mutex>

#include "common.cuh"
#include "fmg_resident.cuh"
#include "fmg_strip.cuh"
#include "once_per_device.h"

namespace fm {

constexpr int kBlock = 256;

inline unsigned blocks_for(size_t threads) { return (unsigned)((threads + kBlock - 1) / kBlock); }


// Sample of a flat thread index and whether it still iterates.
__device__ __forceinline__ bool inactive(const int32_t* active, size_t s) { return active && !active[s]; }

// Sample, cell and column / row of a flat index over n x n grids.  By shifts
// where n is a power of two: the four divisions (64-bit ones for the sample) took
// longer than the arithmetic of the kernels that move a few bytes a cell.
struct CellAt {
    size_t s;
    int c, i, j;
};
__device__ __forceinline__ CellAt cell_at(size_t t, int n) {
    CellAt a;
    if ((n & (n - 1)) == 0) {
        const int lg = __ffs(n) - 1;
        a.s = t >> (2 * lg);
        a.c = (int)t & (n * n - 1);
        a.i = a.c & (n - 1);
        a.j = a.c >> lg;
    } else {
        const size_t cells = (size_t)n * n;
        a.s = t / cells;
        a.c = (int)(t % cells);
        a.i = a.c % n;
        a.j = a.c / n;
    }
    return a;
}

// K_c[J][I] = K_f[2J][2I] (Sec. 2.5, the lower-left child in 0-indexed form).
__global__ void k_inject(int nc, size_t S, const double* __restrict__ Kf, double* __restrict__ Kc) {
    const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    const size_t cells = (size_t)nc * nc;
    if (t >= S * cells) return;
    const CellAt at = cell_at(t, nc);
    const size_t s = at.s;
    const int I = at.i, J = at.j, nf = 2 * nc;
    Kc[t] = Kf[s * (size_t)nf * nf + (size_t)(2 * J) * nf + 2 * I];
}

// Correction-grid coefficients: K_c[J][I] = geometric mean of the four
// children K_f[2J+dj][2I+di] on the injected grid one level finer, computed
// in C (FP32 for the FP32 correction operators of the mixed form: they steer
// the iteration only, the refined stage operators stay FP64).
template <typename C>
__global__ void k_child_geomean(int nc, size_t S, const double* __restrict__ Kf, double* __restrict__ Kc) {
    const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    const size_t cells = (size_t)nc * nc;
    if (t >= S * cells) return;
    const CellAt at = cell_at(t, nc);
    const size_t s = at.s;
    const int I = at.i, J = at.j, nf = 2 * nc;
    const double* k = Kf + s * (size_t)nf * nf + (size_t)(2 * J) * nf + 2 * I;
    Kc[t] = widen(geometric_mean4(rounded<C>(k[0]), rounded<C>(k[1]), rounded<C>(k[nf]), rounded<C>(k[nf + 1])));
}

// Face transmissibilities: harmonic mean inside, 2K on the Dirichlet edges
// (west / east; north / south too when ns, Table 1 Case I), none on the
// no-flow edges, in arithmetic C; optional FP64 copies for refined grids
// (which take C = double).  Te of the east column and Tn of the north row
// hold the boundary faces: every kernel couples neighbours only across
// interior faces, so these enter through D alone.  Each face is formed once
// (the east and north faces of its cell); k_diagonal then sums them.
template <typename T, typename C>
__global__ void k_faces(int n, size_t S, int ns, const double* __restrict__ K, T* __restrict__ Te,
                        T* __restrict__ Tn, double* __restrict__ Te64, double* __restrict__ Tn64) {
    const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    const size_t cells = (size_t)n * n;
    if (t >= S * cells) return;
    const CellAt at = cell_at(t, n);
    const int i = at.i, j = at.j;
    const C k = rounded<C>(K[t]);
    // formed everywhere (of k with itself past an edge) and replaced by integers at
    // the edges: an FP64 product there would take its turn in every warp
    const C he = harmonic_mean(k, rounded<C>(K[i < n - 1 ? t + 1 : t]));
    const C hn = harmonic_mean(k, rounded<C>(K[j < n - 1 ? t + n : t]));
    const C te = (i < n - 1) ? he : twice(k);
    const C tn = (j < n - 1) ? hn : (ns ? twice(k) : C(0));
    Te[t] = rounded<T>(te);
    Tn[t] = rounded<T>(tn);
    if (Te64) {
        Te64[t] = (double)te;
        Tn64[t] = (double)tn;
    }
}

// D = tw + te + ts + tn from the faces in their arithmetic C (the FP64 copies
// where they exist): the west face of a cell is its west neighbour's east
// face, the same harmonic mean of the same two values, so D equals the sum
// of four freshly formed faces bit for bit.  Boundary faces: 2K west, 2K
// south when ns, else 0.  rD (FP64 grids): 1 / D for the smoothers, formed
// once here (may be K's own buffer: a cell reads its K before it writes).
template <typename T, typename C>
__global__ void k_diagonal(int n, size_t S, int ns, const double* K, const T* __restrict__ Te,
                           const T* __restrict__ Tn, const double* __restrict__ Te64,
                           const double* __restrict__ Tn64, T* __restrict__ D, double* __restrict__ D64, T* rD) {
    const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    const size_t cells = (size_t)n * n;
    if (t >= S * cells) return;
    const CellAt at = cell_at(t, n);
    const int i = at.i, j = at.j;
    // (a test for the copies here converted every face, in the FP64 pipe: 0.6 ms
    // where 0.3 do, 1000 grids of 256 x 256)
    auto face = [&](const T* f, const double* f64, size_t u) {
        if constexpr (sizeof(C) != sizeof(T)) return f64[u];
        else return f[u];
    };
    auto fe = [&](size_t u) { return face(Te, Te64, u); };
    auto fn = [&](size_t u) { return face(Tn, Tn64, u); };
    auto edge = [&] { return twice(rounded<C>(K[t])); };
    const C tw = (i > 0) ? fe(t - 1) : edge();
    const C ts = (j > 0) ? fn(t - n) : (ns ? edge() : C(0));
    const C d = tw + fe(t) + ts + fn(t);
    D[t] = rounded<T>(d);
    if (D64) D64[t] = (double)d;
    if (rD) rD[t] = recip_set((T)d);
}

// Cell o of the edge of an n x n grid (4 (n - 1) cells).
__device__ __forceinline__ void ring_cell(int o, int n, int& i, int& j) {
    const int q = o / (n - 1), e = o % (n - 1);   // side, position along it
    i = q == 0 ? e : q == 1 ? n - 1 : q == 2 ? n - 1 - e : 0;
    j = q == 0 ? 0 : q == 1 ? e : q == 2 ? n - 1 : n - 1 - e;
}
// Threads for S grids' cells and, after them, their edge cells once more.
inline size_t ring_threads(size_t S, int n) { return S * ((size_t)n * n + 4 * (size_t)(n - 1)); }

// Right-hand side of a stage problem: the Dirichlet data moved to the rhs.  Zero,
// without a read of K, off the edges; edge cells on threads of their own (in one
// pass their FP64 products took their turn in every warp: 288 us for the stages of
// 5000 FP64 samples of 64 x 64).
template <typename T>
__global__ void k_stage_rhs(int n, size_t S, const double* __restrict__ K, Bnd bd, T* __restrict__ b) {
    const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    const size_t cells = (size_t)n * n;
    if (t < S * cells) {
        const CellAt at = cell_at(t, n);
        if (at.i > 0 && at.i < n - 1 && at.j > 0 && at.j < n - 1) b[t] = T(0);
        return;
    }
    const int ring = 4 * (n - 1);
    const size_t u = t - S * cells, s = u / ring;
    if (s >= S) return;
    int i, j;
    ring_cell((int)(u % ring), n, i, j);
    const size_t g = s * cells + (size_t)j * n + i;
    const bool edge = i == 0 || i == n - 1 || bd.ns;
    b[g] = edge ? (T)dirichlet_rhs(bd, n, i, j, K[g]) : T(0);
}

// One colour of a red-black Gauss-Seidel sweep: cells with (i + j) % 2 == color.
template <typename T>
__global__ void k_rbgs_color(int n, size_t S, int color, const T* __restrict__ b, const T* __restrict__ Te,
                             const T* __restrict__ Tn, const T* __restrict__ D, const T* __restrict__ rD,
                             T* __restrict__ p, const int32_t* __restrict__ active) {
    const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    const size_t half = (size_t)n * n / 2;
    if (t >= S * half) return;
    const size_t s = t / half;
    if (inactive(active, s)) return;
    const int h = (int)(t % half);
    const int j = h / (n / 2);
    const int i = 2 * (h % (n / 2)) + ((j + color) & 1);
    const size_t c = s * (size_t)n * n + (size_t)j * n + i;
    T acc = b[c];
    if (i > 0) acc += Te[c - 1] * p[c - 1];
    if (i < n - 1) acc += Te[c] * p[c + 1];
    if (j > 0) acc += Tn[c - n] * p[c - n];
    if (j < n - 1) acc += Tn[c] * p[c + n];
    p[c] = acc * (rD ? rD[c] : T(1) / D[c]);
}

// (P u_c) at fine cell (i, j): bilinear cell-centred (9, 3, 3, 1) / 16
// (prolong_vals, one expression for every kernel that prolongs), with ghosts
// 2g - u across the Dirichlet edges (g = 0 for an error) and the edge value
// mirrored across the no-flow edges; a corner ghost takes the x rule on the
// y ghost.  The ghosts are formed only where a cell needs them: formed for
// every cell and selected, they were two thirds of an FP64 prolongation.
template <typename U>
__device__ __forceinline__ U prolong_at(int nc, const U* u, int i, int j, const Ghost<U>& g) {
    const int I = i >> 1, J = j >> 1;
    const int Ix = (i & 1) ? I + 1 : I - 1;
    const int Jy = (j & 1) ? J + 1 : J - 1;
    const bool xe = Ix < 0 || Ix > nc - 1, ye = Jy < 0 || Jy > nc - 1;
    const int Ic = xe ? I : Ix, Jc = ye ? J : Jy;
    const U* row = u + (size_t)J * nc;
    const U* other = u + (size_t)Jc * nc;
    U nx = row[Ic], ny = other[I], nxy = other[Ic];
    if (xe) {
        const U b = Ix < 0 ? g.w : g.e;
        nx = fma(U(2), b, -nx);
        nxy = fma(U(2), b, -nxy);
    }
    if (ye && g.ns) {
        const U b = Jy < 0 ? g.s : g.n;
        ny = fma(U(2), b, -ny);
        nxy = fma(U(2), b, -nxy);
    }
    return prolong_vals(row[I], nx, ny, nxy);
}
// The same of an error, whose boundary data are zero: the ghosts change sign.
template <typename U>
__device__ __forceinline__ U prolong_err(int nc, const U* u, int i, int j, int ns) {
    const int I = i >> 1, J = j >> 1;
    const int Ix = (i & 1) ? I + 1 : I - 1;
    const int Jy = (j & 1) ? J + 1 : J - 1;
    const bool xe = Ix < 0 || Ix > nc - 1, ye = Jy < 0 || Jy > nc - 1, fy = ye && ns;
    const int Ic = xe ? I : Ix;
    const U* row = u + (size_t)J * nc;
    const U* other = u + (size_t)(ye ? J : Jy) * nc;
    return prolong_vals(row[I], flip_if(xe, row[Ic]), flip_if(fy, other[I]), flip_if(xe != fy, other[Ic]));
}

// nsweeps red-black sweeps (colour 0 then 1) on tiles of TI x TI cells of
// one sample, staged in shared memory with a halo of hh = 2 nsweeps cells:
// each half-sweep leaves one more ring at the halo's edge stale, so after
// 2 nsweeps half-sweeps exactly the interior is current.  Every cell update
// is the colour kernel's, in the same order, so the result is bit-identical
// to 2 nsweeps k_rbgs_color launches while p, b and the coefficients cross
// HBM once.  The iterate is read from p_in and written to p_out (another
// buffer): a tile's halo is its neighbours' interior, which must still hold
// the values from before the call whatever order the CTAs run in.  Grid:
// S * tiles^2 CTAs, tile index fastest; inactive samples are not written.
template <typename T>
__global__ void __launch_bounds__(256) k_rbgs_tile(int n, size_t S, int TI, int hh, int nsweeps,
                                                   const T* __restrict__ b, const T* __restrict__ Te,
                                                   const T* __restrict__ Tn, const T* __restrict__ D,
                                                   const T* __restrict__ rD, const T* __restrict__ p_in,
                                                   T* __restrict__ p_out, const int32_t* __restrict__ active,
                                                   const T* __restrict__ ec, int ns) {
    extern __shared__ __align__(16) unsigned char tile_smem[];
    const int tiles = (n + TI - 1) / TI;
    const size_t s = blockIdx.x / ((unsigned)tiles * tiles);
    if (s >= S || inactive(active, s)) return;
    const int tid = (int)(blockIdx.x % ((unsigned)tiles * tiles));
    const int ti = tid % tiles, tj = tid / tiles;
    const int xa = max(ti * TI - hh, 0), ya = max(tj * TI - hh, 0);
    const int xb = min(ti * TI + TI + hh, n), yb = min(tj * TI + TI + hh, n);
    const int RW = xb - xa, RH = yb - ya, R = RW * RH;
    T* sp = reinterpret_cast<T*>(tile_smem);
    T* sb = sp + R;
    T* se = sb + R;
    T* sn = se + R;
    T* sd = sn + R;
    const size_t base = s * (size_t)n * n;
    for (int e = threadIdx.x; e < R; e += blockDim.x) {
        const int r = e / RW, q = e % RW;
        const size_t g = base + (size_t)(ya + r) * n + xa + q;
        // with ec: the coarse-grid correction p + (P e) as k_prolong forms it, on black
        // cells only (the first half-sweep replaces the red ones)
        const bool corr = ec && ((xa + q + ya + r) & 1);
        sp[e] = corr ? p_in[g] + prolong_err(n / 2, ec + s * (size_t)(n / 2) * (n / 2), xa + q, ya + r, ns)
                     : p_in[g];
        sb[e] = b[g];
        se[e] = Te[g];
        sn[e] = Tn[g];
        sd[e] = rD ? rD[g] : T(1) / D[g];
    }
    __syncthreads();
    const int W2 = (RW + 1) / 2;
    for (int hs = 0; hs < 2 * nsweeps; ++hs) {
        const int color = hs & 1;
        for (int h = threadIdx.x; h < RH * W2; h += blockDim.x) {
            const int r = h / W2;
            const int q = 2 * (h % W2) + ((color + xa + ya + r) & 1);
            if (q >= RW) continue;
            const int i = xa + q, j = ya + r;
            // a cell whose in-domain neighbour lies outside the region is not updated
            if ((i > 0 && q == 0) || (i < n - 1 && q == RW - 1) || (j > 0 && r == 0) || (j < n - 1 && r == RH - 1))
                continue;
            const int e = r * RW + q;
            T acc = sb[e];
            if (i > 0) acc += se[e - 1] * sp[e - 1];
            if (i < n - 1) acc += se[e] * sp[e + 1];
            if (j > 0) acc += sn[e - RW] * sp[e - RW];
            if (j < n - 1) acc += sn[e] * sp[e + RW];
            sp[e] = acc * sd[e];
        }
        __syncthreads();
    }
    const int x0 = ti * TI, y0 = tj * TI;
    const int IW = min(TI, n - x0), IH = min(TI, n - y0);
    for (int e = threadIdx.x; e < IW * IH; e += blockDim.x) {
        const int r = e / IW, q = e % IW;
        p_out[base + (size_t)(y0 + r) * n + x0 + q] = sp[(y0 - ya + r) * RW + (x0 - xa + q)];
    }
}

// The tile smoother with every operand but the iterate in registers.  Thread
// (c, g) owns the column pair 2c, 2c+1 and rows g RPT .. g RPT + RPT - 1 of an
// R x R region (tile interior plus halo, clipped at the domain edge) for all
// sweeps: in every row one of its two cells has the colour being updated, so
// every lane updates RPT cells per half-sweep with no divergence.  b, 1/D and
// the four faces of its cells are loaded once (a face that does not exist is
// zero, and the zero-padded shared array keeps every neighbour read in
// bounds); only p goes through shared memory, and neighbours inside the
// thread's own cells come from registers.  Same halo argument, same update
// order and reciprocal as the colour kernel: bit-identical sweeps (a missing
// face adds an exact zero).
template <typename T, int R, int RPT>
__global__ void __launch_bounds__((R / 2) * (R / RPT)) k_rbgs_tile_reg(int n, size_t S, int TI, int hh, int nsweeps,
                                                                      const T* __restrict__ b,
                                                                      const T* __restrict__ Te,
                                                                      const T* __restrict__ Tn,
                                                                      const T* __restrict__ D,
                                                                      const T* __restrict__ rD,
                                                                      const T* __restrict__ p_in, T* __restrict__ p_out,
                                                                      const int32_t* __restrict__ active,
                                                                      const T* __restrict__ ec, int ns) {
    static_assert(R % 2 == 0 && R % RPT == 0, "region must split into column pairs and row strips");
    constexpr int C = R / 2, P = R + 2;   // column pairs; padded row pitch
    __shared__ T sp[P * P];
    const int tiles = (n + TI - 1) / TI;
    const size_t s = blockIdx.x / ((unsigned)tiles * tiles);
    if (s >= S || inactive(active, s)) return;
    const int tid = (int)(blockIdx.x % ((unsigned)tiles * tiles));
    const int ti = tid % tiles, tj = tid / tiles;
    const int xa = max(ti * TI - hh, 0), ya = max(tj * TI - hh, 0);
    const int RW = min(ti * TI + TI + hh, n) - xa, RH = min(tj * TI + TI + hh, n) - ya;
    const int c = threadIdx.x % C, y0 = (threadIdx.x / C) * RPT;
    const size_t base = s * (size_t)n * n;
    for (int e = threadIdx.x; e < P * P; e += blockDim.x) sp[e] = T(0);
    __syncthreads();
    T rb[RPT][2], rr[RPT][2], re[RPT][2], rw[RPT][2], rn[RPT][2], rs[RPT][2], rp[RPT][2];
    bool up[RPT][2];
#pragma unroll
    for (int k = 0; k < RPT; ++k) {
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const int x = 2 * c + j, y = y0 + k, gx = xa + x, gy = ya + y;
            rb[k][j] = rr[k][j] = re[k][j] = rw[k][j] = rn[k][j] = rs[k][j] = rp[k][j] = T(0);
            up[k][j] = false;
            if (x < RW && y < RH) {
                const size_t g = base + (size_t)gy * n + gx;
                // with ec: the coarse-grid correction p + (P e) as k_prolong forms it, on
                // black cells only (the first half-sweep replaces the red ones)
                rp[k][j] = ec && ((gx + gy) & 1)
                               ? p_in[g] + prolong_err(n / 2, ec + s * (size_t)(n / 2) * (n / 2), gx, gy, ns)
                               : p_in[g];
                rb[k][j] = b[g];
                rr[k][j] = rD ? rD[g] : T(1) / D[g];
                if (gx < n - 1) re[k][j] = Te[g];
                if (gy < n - 1) rn[k][j] = Tn[g];
                if (gx > 0) rw[k][j] = Te[g - 1];
                if (gy > 0) rs[k][j] = Tn[g - n];
                // a cell whose in-domain neighbour lies outside the region is not updated
                up[k][j] = !((gx > 0 && x == 0) || (gx < n - 1 && x == RW - 1) || (gy > 0 && y == 0) ||
                             (gy < n - 1 && y == RH - 1));
                sp[(y + 1) * P + x + 1] = rp[k][j];
            }
        }
    }
    __syncthreads();
    for (int hs = 0; hs < 2 * nsweeps; ++hs) {
        const int color = hs & 1;
#pragma unroll
        for (int k = 0; k < RPT; ++k) {
            const int y = y0 + k;
            // the cell of this colour in row y: column 2c + j (selects, so the
            // register arrays are never indexed at run time)
            const bool j = ((color + xa + ya + y) & 1) != 0;
            const int x = 2 * c + (j ? 1 : 0);
            const T* row = sp + (y + 1) * P + x + 1;
            const T p0 = rp[k][0], p1 = rp[k][1];
            const T pw = j ? p0 : row[-1];
            const T pe = j ? row[1] : p1;
            const T ps = k > 0 ? (j ? rp[k - 1][1] : rp[k - 1][0]) : row[-P];
            const T pn = k < RPT - 1 ? (j ? rp[k + 1][1] : rp[k + 1][0]) : row[P];
            T acc = j ? rb[k][1] : rb[k][0];
            acc += (j ? rw[k][1] : rw[k][0]) * pw;
            acc += (j ? re[k][1] : re[k][0]) * pe;
            acc += (j ? rs[k][1] : rs[k][0]) * ps;
            acc += (j ? rn[k][1] : rn[k][0]) * pn;
            const bool u = j ? up[k][1] : up[k][0];
            const T v = u ? acc * (j ? rr[k][1] : rr[k][0]) : (j ? p1 : p0);
            if (j) rp[k][1] = v;
            else rp[k][0] = v;
            if (x < RW && y < RH) sp[(y + 1) * P + x + 1] = v;
        }
        __syncthreads();
    }
    const int x0 = ti * TI, y0i = tj * TI;
#pragma unroll
    for (int k = 0; k < RPT; ++k) {
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const int x = 2 * c + j, y = y0 + k, gx = xa + x, gy = ya + y;
            if (x < RW && y < RH && gx >= x0 && gx < min(x0 + TI, n) && gy >= y0i && gy < min(y0i + TI, n))
                p_out[base + (size_t)gy * n + gx] = rp[k][j];
        }
    }
}

// r = b - A p at cell c: D p rounded, then one fused multiply-add per face
// (W, E, S, N), spelled out so that every kernel forming a residual rounds
// the same way whatever the compiler would contract.
template <typename T>
__device__ __forceinline__ T residual_at(int n, size_t c, int i, int j, const T* b, const T* Te, const T* Tn,
                                         const T* D, const T* p) {
    T v = mul_rn(D[c], p[c]);
    if (i > 0) v = fma(-Te[c - 1], p[c - 1], v);
    if (i < n - 1) v = fma(-Te[c], p[c + 1], v);
    if (j > 0) v = fma(-Tn[c - n], p[c - n], v);
    if (j < n - 1) v = fma(-Tn[c], p[c + n], v);
    return b[c] - v;
}

// Residuals of the four children of coarse cell (I, J), summed (kRedOnly: smoothed
// = the last half-sweep has zeroed the black ones').
template <typename T>
__device__ __forceinline__ T restricted_at(int nf, size_t c00, int I, int J, const T* b, const T* Te, const T* Tn,
                                           const T* D, const T* p, bool smoothed) {
    const int i = 2 * I, j = 2 * J;
    const T r00 = residual_at(nf, c00, i, j, b, Te, Tn, D, p);
    if (kRedOnly<T> && smoothed) return r00 + residual_at(nf, c00 + nf + 1, i + 1, j + 1, b, Te, Tn, D, p);
    const T r10 = residual_at(nf, c00 + 1, i + 1, j, b, Te, Tn, D, p);
    const T r01 = residual_at(nf, c00 + nf, i, j + 1, b, Te, Tn, D, p);
    const T r11 = residual_at(nf, c00 + nf + 1, i + 1, j + 1, b, Te, Tn, D, p);
    return r00 + r10 + r01 + r11;
}

// Fused residual + restriction: b_c = sum of the four fine residuals; p_c = 0.
template <typename T>
__global__ void k_residual_restrict(int nc, size_t S, const T* __restrict__ bf, const T* __restrict__ Te,
                                    const T* __restrict__ Tn, const T* __restrict__ D, const T* __restrict__ pf,
                                    T* __restrict__ bc, T* __restrict__ pc, const int32_t* __restrict__ active,
                                    int smoothed) {
    const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    const size_t cells = (size_t)nc * nc;
    if (t >= S * cells) return;
    const CellAt at = cell_at(t, nc);
    if (inactive(active, at.s)) return;
    const int nf = 2 * nc;
    const size_t c00 = at.s * (size_t)nf * nf + (size_t)(2 * at.j) * nf + 2 * at.i;
    bc[t] = restricted_at(nf, c00, at.i, at.j, bf, Te, Tn, D, pf, smoothed != 0);
    pc[t] = T(0);
}

// p_f += P e_c (add = 1, boundary values 0) or p_f = P u_c (add = 0, FMG start,
// the Dirichlet data as ghost values).  Cells off the edges first, then the edge
// cells on threads of their own: the ghosts' FP64 operations take the FP64 pipe
// from every warp that holds them, predicated off or not (1000 grids of
// 256 x 256: nine operations a cell for five).
template <typename U>
__global__ void k_prolong(int nc, size_t S, const U* __restrict__ uc, Ghost<U> gh, int add, U* __restrict__ pf,
                          const int32_t* __restrict__ active) {
    const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int nf = 2 * nc, ring = 4 * (nf - 1);
    const size_t cells = (size_t)nf * nf;
    size_t s;
    int i, j;
    U v;
    if (t < S * cells) {
        const CellAt at = cell_at(t, nf);
        s = at.s;
        i = at.i;
        j = at.j;
        if (i == 0 || i == nf - 1 || j == 0 || j == nf - 1 || inactive(active, s)) return;
        const U* row = uc + s * (size_t)nc * nc + (size_t)(j >> 1) * nc + (i >> 1);
        const int x = (i & 1) ? 1 : -1, y = (j & 1) ? nc : -nc;
        v = prolong_vals(row[0], row[x], row[y], row[y + x]);
    } else {
        const size_t r = t - S * cells;
        s = r / ring;
        if (s >= S || inactive(active, s)) return;
        ring_cell((int)(r % ring), nf, i, j);
        v = prolong_at(nc, uc + s * (size_t)nc * nc, i, j, gh);
    }
    const size_t g = s * cells + (size_t)j * nf + i;
    pf[g] = add ? pf[g] + v : v;
}

// Three neighbouring values of a coarse row around column I: its own, west and
// east; past the Dirichlet edges the error's ghosts, minus its own.
template <typename T>
struct CoarseRow {
    T o, w, e;
};
template <typename T>
__device__ __forceinline__ CoarseRow<T> ghost_row(const CoarseRow<T>& r, int ns) {
    return CoarseRow<T>{flip_if(ns, r.o), flip_if(ns, r.w), flip_if(ns, r.e)};
}
// (P e) at the two fine columns of a coarse cell, in the fine row next to row `other`.
template <typename T, typename V2>
__device__ __forceinline__ V2 prolong_pair(const CoarseRow<T>& own, const CoarseRow<T>& other) {
    V2 d;
    d.x = prolong_vals(own.o, own.w, other.o, other.w);
    d.y = prolong_vals(own.o, own.e, other.o, other.e);
    return d;
}

template <typename T>
struct PairOf;
template <>
struct PairOf<float> {
    using type = float2;
};
template <>
struct PairOf<double> {
    using type = double2;
};

// Energy-optimal step of a coarse-grid correction: the correction d = P e_c
// is added as alpha d with alpha = (r, d) / (d, A d), r = b - A x the
// residual it answers, the exact line minimum of the energy error for the
// symmetric positive definite A (so a cycle never raises the energy error,
// whatever the correction operators).  Per (sample, chunk) of grid n: the
// partial sums of (r, d) and (d, A d) in FP64; entries 0 and 1 of the
// sample's 3-double slots in partial.
//
// A lane owns a coarse column (two fine ones) and walks up its band of rows:
// d of each cell is formed once, x and Tn of the row below stay in registers,
// and values of the next columns come by shuffle (windows of 30 columns with
// one more at each end, or 32 where the grid is no wider).  A thread per cell,
// forming d at the cell and its four neighbours, took 9.3 ms of a solve of seven
// fields of 1024 x 1024 (312 launches of 30 us on average); the walk takes 3.6
// (67 us on five fields of the finest grid, where the FP64 pipe's two FMAs a cell
// are 18 us and the instructions issued most of the rest).
template <typename T>
__global__ void __launch_bounds__(256) k_energy_partials(
    int n, size_t S, int chunks, const T* __restrict__ b, const T* __restrict__ Te, const T* __restrict__ Tn,
    const T* __restrict__ D, const T* __restrict__ x, const T* __restrict__ ec, const int32_t* __restrict__ active,
    const int32_t* __restrict__ order, double* __restrict__ partial, int ns) {
    using V2 = typename PairOf<T>::type;
    constexpr unsigned all = 0xffffffffu;
    __shared__ double red[2][32];
    if (blockIdx.x / chunks >= S) return;   // S: the samples enumerated (listed by order, if given)
    const size_t s = order ? (size_t)order[blockIdx.x / chunks] : blockIdx.x / chunks;
    const int ch = (int)(blockIdx.x % chunks);
    if (inactive(active, s)) return;
    const int nc = n / 2, lane = threadIdx.x & 31, warps = (int)(blockDim.x >> 5);
    const size_t base = s * (size_t)n * n;
    const T* e = ec + s * (size_t)nc * nc;
    // the chunk's coarse rows, as tasks of (window, part of the rows)
    const int cr = (nc + chunks - 1) / chunks, J0 = min(nc, ch * cr), J1 = min(nc, J0 + cr);
    const bool whole = nc <= 32;
    const int windows = whole ? 1 : (nc + 29) / 30;
    const int parts = max(1, min(cr, warps / windows)), pr = (cr + parts - 1) / parts;
    double rd = 0.0, dad = 0.0;
    for (int t = (int)(threadIdx.x >> 5); t < windows * parts; t += warps) {
        const int I = whole ? lane : 30 * (t % windows) - 1 + lane, Ic = min(max(I, 0), nc - 1);
        const bool mine = I >= 0 && I < nc && (whole || (lane >= 1 && lane <= 30));
        const int Ja = J0 + (t / windows) * pr, Jb = min(J1, Ja + pr);
        if (Ja >= Jb) continue;
        auto coarse = [&](int J) {
            CoarseRow<T> r;
            r.o = e[(size_t)J * nc + Ic];
            r.w = __shfl_up_sync(all, r.o, 1);
            r.e = __shfl_down_sync(all, r.o, 1);
            if (I <= 0) r.w = flip_if(true, r.o);
            if (I >= nc - 1) r.e = flip_if(true, r.o);
            return r;
        };
        auto fine = [&](const T* a, int j) { return *reinterpret_cast<const V2*>(a + base + (size_t)j * n + 2 * Ic); };
        CoarseRow<T> cur = coarse(Ja);
        const CoarseRow<T> below = Ja > 0 ? coarse(Ja - 1) : ghost_row(cur, ns);
        V2 dm = prolong_pair<T, V2>(below, cur), dc = prolong_pair<T, V2>(cur, below);
        const int jm = max(2 * Ja - 1, 0);
        V2 xm = fine(x, jm), tm = fine(Tn, jm), xc = fine(x, 2 * Ja);
        // row j: its values, those of the rows below and above
        auto row = [&](int j, const V2& dl, const V2& d, const V2& dh, const V2& xl, const V2& xv, const V2& xh,
                       const V2& tl, const V2& tn) {
            const V2 bv = fine(b, j), te = fine(Te, j), dd = fine(D, j);
            const T tw = __shfl_up_sync(all, te.y, 1);
            const T xw = __shfl_up_sync(all, xv.y, 1), xe = __shfl_down_sync(all, xv.x, 1);
            const T dw = __shfl_up_sync(all, d.y, 1), de = __shfl_down_sync(all, d.x, 1);
            const bool in_w = I > 0, in_e = I < nc - 1, in_s = j > 0, in_n = j < n - 1;
            auto apply = [&](T diag, T c, T fw, T vw, bool w, T fe, T ve, bool ee, T fs, T vs, T fn, T vn) {
                T v = mul_rn(diag, c);   // as residual_at forms A x
                if (w) v = fma(-fw, vw, v);
                if (ee) v = fma(-fe, ve, v);
                if (in_s) v = fma(-fs, vs, v);
                if (in_n) v = fma(-fn, vn, v);
                return v;
            };
            const T r0 = bv.x - apply(dd.x, xv.x, tw, xw, in_w, te.x, xv.y, true, tl.x, xl.x, tn.x, xh.x);
            const T r1 = bv.y - apply(dd.y, xv.y, te.x, xv.x, true, te.y, xe, in_e, tl.y, xl.y, tn.y, xh.y);
            const T a0 = apply(dd.x, d.x, tw, dw, in_w, te.x, d.y, true, tl.x, dl.x, tn.x, dh.x);
            const T a1 = apply(dd.y, d.y, te.x, d.x, true, te.y, de, in_e, tl.y, dl.y, tn.y, dh.y);
            if (mine) {
                const double d0 = widen(d.x), d1 = widen(d.y);
                rd = fma(widen(r0), d0, rd);
                dad = fma(d0, widen(a0), dad);
                rd = fma(widen(r1), d1, rd);
                dad = fma(d1, widen(a1), dad);
            }
        };
#pragma unroll 1
        for (int J = Ja; J < Jb; ++J) {
            const CoarseRow<T> up = J + 1 < nc ? coarse(J + 1) : ghost_row(cur, ns);
            const int j = 2 * J;
            const V2 d1 = prolong_pair<T, V2>(cur, up), d2 = prolong_pair<T, V2>(up, cur);
            const V2 x1 = fine(x, j + 1), x2 = fine(x, min(j + 2, n - 1));
            const V2 t0 = fine(Tn, j), t1 = fine(Tn, j + 1);
            row(j, dm, dc, d1, xm, xc, x1, tm, t0);
            row(j + 1, dc, d1, d2, xc, x1, x2, t0, t1);
            dm = d1;
            dc = d2;
            xm = x1;
            xc = x2;
            tm = t1;
            cur = up;
        }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        rd += __shfl_down_sync(all, rd, off);
        dad += __shfl_down_sync(all, dad, off);
    }
    if (lane == 0) {
        red[0][threadIdx.x >> 5] = rd;
        red[1][threadIdx.x >> 5] = dad;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double a = 0.0, q = 0.0;
        for (int w = 0; w < warps; ++w) {
            a += red[0][w];
            q += red[1][w];
        }
        double* out = partial + ((size_t)s * chunks + ch) * 3;
        out[0] = a;
        out[1] = q;
    }
}

// p_f += alpha P e_c, the stepped correction (in FP64, rounded once to T), with
// alpha = (r, d) / (d, A d) of the sample from its chunks' partial sums (0 when
// d = 0), summed by the first warp of each block: a launch of its own cost 4 us
// a cycle and grid.  Threads take coarse cells, so four fine cells share the nine
// coarse values (seven fields of 1024 x 1024: 3.5 ms a solve for both, now 2.4);
// S, order as in k_energy_partials.
constexpr int kStepCells = 4;   // coarse cells a thread
template <typename T>
__global__ void __launch_bounds__(256) k_energy_apply(int nc, size_t S, int chunks, int blocks,
                                                      const T* __restrict__ uc, const double* __restrict__ partial,
                                                      T* __restrict__ pf, const int32_t* __restrict__ active,
                                                      const int32_t* __restrict__ order, int ns) {
    using V2 = typename PairOf<T>::type;
    __shared__ double alpha_s;
    if (blockIdx.x / blocks >= S) return;
    const size_t s = order ? (size_t)order[blockIdx.x / blocks] : blockIdx.x / blocks;
    if (inactive(active, s)) return;
    if (threadIdx.x < 32) {
        double rd = 0.0, dad = 0.0;
        for (int ch = (int)threadIdx.x; ch < chunks; ch += 32) {
            rd += partial[((size_t)s * chunks + ch) * 3];
            dad += partial[((size_t)s * chunks + ch) * 3 + 1];
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            rd += __shfl_down_sync(0xffffffffu, rd, off);
            dad += __shfl_down_sync(0xffffffffu, dad, off);
        }
        if (threadIdx.x == 0) alpha_s = dad > 0.0 ? rd / dad : 0.0;
    }
    __syncthreads();
    const double alpha = alpha_s;
    const int nf = 2 * nc, cells = nc * nc;
    const T* u = uc + s * (size_t)cells;
    T* p = pf + s * (size_t)nf * nf;
    for (int c = (int)(blockIdx.x % blocks) * 256 + (int)threadIdx.x; c < cells; c += blocks * 256) {
        const int I = c % nc, J = c / nc;
        auto coarse = [&](int j) {
            const T* r = u + (size_t)j * nc + I;
            CoarseRow<T> v;
            v.o = r[0];
            v.w = I > 0 ? r[-1] : flip_if(true, v.o);
            v.e = I < nc - 1 ? r[1] : flip_if(true, v.o);
            return v;
        };
        const CoarseRow<T> own = coarse(J);
        const CoarseRow<T> lo = J > 0 ? coarse(J - 1) : ghost_row(own, ns);
        const CoarseRow<T> hi = J < nc - 1 ? coarse(J + 1) : ghost_row(own, ns);
#pragma unroll
        for (int y = 0; y < 2; ++y) {
            const V2 d = prolong_pair<T, V2>(own, y ? hi : lo);
            V2* q = reinterpret_cast<V2*>(p + (size_t)(2 * J + y) * nf + 2 * I);
            V2 v = *q;
            v.x = rounded<T>(fma(alpha, widen(d.x), widen(v.x)));
            v.y = rounded<T>(fma(alpha, widen(d.y), widen(v.y)));
            *q = v;
        }
    }
}

// The first colour (0) of post-smoothing fused with the coarse-grid
// correction p += P e: a red cell's update reads only its black neighbours,
// so they are read as p + (P e) on the fly and the red cell's own correction
// is never needed (its value is replaced); the next colour launch then
// replaces every black cell from the updated red ones.  Each corrected value
// is k_prolong's and each update k_rbgs_color's, so the sweep is
// bit-identical to a prolongation pass followed by the colour launches.
template <typename T>
__global__ void k_rbgs_color0_prolong(int n, size_t S, const T* __restrict__ b, const T* __restrict__ Te,
                                      const T* __restrict__ Tn, const T* __restrict__ D, const T* __restrict__ rD,
                                      T* __restrict__ p,
                                      const T* __restrict__ ec, const int32_t* __restrict__ active, int ns) {
    const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    const size_t half = (size_t)n * n / 2;
    if (t >= S * half) return;
    const size_t s = t / half;
    if (inactive(active, s)) return;
    const int h = (int)(t % half);
    const int j = h / (n / 2);
    const int i = 2 * (h % (n / 2)) + (j & 1);
    const size_t base = s * (size_t)n * n;
    const size_t c = base + (size_t)j * n + i;
    const int nc = n / 2;
    const T* e = ec + s * (size_t)nc * nc;
    T acc = b[c];
    if (i > 0) acc += Te[c - 1] * (p[c - 1] + prolong_err(nc, e, i - 1, j, ns));
    if (i < n - 1) acc += Te[c] * (p[c + 1] + prolong_err(nc, e, i + 1, j, ns));
    if (j > 0) acc += Tn[c - n] * (p[c - n] + prolong_err(nc, e, i, j - 1, ns));
    if (j < n - 1) acc += Tn[c] * (p[c + n] + prolong_err(nc, e, i, j + 1, ns));
    p[c] = acc * (rD ? rD[c] : T(1) / D[c]);
}

// Inverse of the operator of the coarsest grid (m = n0^2 <= 16 unknowns) in
// FP64, 32 samples per CTA: the faces by all threads, the banded L D L^T
// factors (half bandwidth n0) of a sample by one thread, then one column of
// the inverse per thread (forward and backward substitution of a unit
// vector).  Faces and factors lie in shared memory with the samples fastest,
// so a warp reads them without conflicts.  About 150 FP64 operations a column
// and 200 a sample, and chains of some 300 dependent ones; the dense
// Gauss-Jordan elimination of [A | I] by a warp per sample that this replaces
// took 83 us for 256 samples and 393 us for 5304.
constexpr int kInvSamples = 32;

template <typename T, int N0>
__global__ void __launch_bounds__(kInvSamples* N0* N0) k_coarse_inverse(size_t S, const double* __restrict__ K,
                                                                         T* __restrict__ Ainv, int ns) {
    constexpr int M = N0 * N0;
    __shared__ double se[M][kInvSamples], sn[M][kInvSamples];   // east and north faces
    __shared__ double sk[M][kInvSamples];                       // coefficients; then 1 / D(r)
    __shared__ double sl[M * N0][kInvSamples];                  // L(r, r - k) at r N0 + k - 1
    const int u = threadIdx.x % kInvSamples, c = threadIdx.x / kInvSamples;
    const size_t s = (size_t)blockIdx.x * kInvSamples + u;
    {   // cell c of sample u
        const double* k = K + s * M;
        const int i = c % N0, j = c / N0;
        const double kc = s < S ? k[c] : 1.0;
        const double ke = s < S && i < N0 - 1 ? k[c + 1] : kc, kn = s < S && j < N0 - 1 ? k[c + N0] : kc;
        sk[c][u] = kc;
        se[c][u] = i < N0 - 1 ? harmonic_mean(kc, ke) : 2.0 * kc;
        sn[c][u] = j < N0 - 1 ? harmonic_mean(kc, kn) : (ns ? 2.0 * kc : 0.0);
    }
    __syncthreads();
    if (threadIdx.x < kInvSamples) {
        double L[M][N0 + 1], rd[M];   // indexed by constants once unrolled
#pragma unroll
        for (int r = 0; r < M; ++r) {
            const int i = r % N0, j = r / N0;
            const double tw = i > 0 ? se[i > 0 ? r - 1 : r][u] : 2.0 * sk[r][u];
            const double ts = j > 0 ? sn[j > 0 ? r - N0 : r][u] : (ns ? 2.0 * sk[r][u] : 0.0);
            double d = tw + se[r][u] + ts + sn[r][u];
            double mr[N0 + 1];                // L(r, r - k) D(r - k)
#pragma unroll
            for (int q = N0; q >= 1; --q) {
                mr[q] = 0.0;
                L[r][q] = 0.0;
                if (r - q < 0) continue;
                double v = q == N0 ? -ts : ((q == 1 && i > 0) ? -tw : 0.0);
#pragma unroll
                for (int t = q + 1; t <= N0; ++t)
                    if (r - t >= 0) v = fma(-mr[t], L[r - q][t - q], v);
                mr[q] = v;
                L[r][q] = v * rd[r - q];
                d = fma(-v, L[r][q], d);
            }
            rd[r] = 1.0 / d;
#pragma unroll
            for (int q = 1; q <= N0; ++q) sl[r * N0 + q - 1][u] = L[r][q];
        }
#pragma unroll
        for (int r = 0; r < M; ++r) sk[r][u] = rd[r];
    }
    __syncthreads();
    if (s >= S) return;
    double x[M];
#pragma unroll
    for (int r = 0; r < M; ++r) {
        double v = r == c ? 1.0 : 0.0;
#pragma unroll
        for (int q = N0; q >= 1; --q)
            if (r - q >= 0) v = fma(-sl[r * N0 + q - 1][u], x[r - q], v);
        x[r] = v;
    }
#pragma unroll
    for (int r = M - 1; r >= 0; --r) {
        double v = x[r] * sk[r][u];
#pragma unroll
        for (int q = N0; q >= 1; --q)
            if (r + q < M) v = fma(-sl[(r + q) * N0 + q - 1][u], x[r + q], v);
        x[r] = v;
    }
    T* out = Ainv + (s * M + c) * M;   // column c as row c: the inverse is symmetric
#pragma unroll
    for (int r = 0; r < M; ++r) out[r] = (T)x[r];
}

template <typename T>
static void coarse_inverse(fm_ctx* ctx, int n0, size_t S, const double* K, T* Ainv, int ns, cudaStream_t st) {
    const int m = n0 * n0;
    const unsigned grid = (unsigned)((S + kInvSamples - 1) / kInvSamples);
    FM_TIMED(ctx, kFamCoarseInverse, st, (double)S * (8 * m + sizeof(T) * m * m), 2.0 * S * m * m * (2 * n0 + 1),
             if (n0 == 2) k_coarse_inverse<T, 2><<<grid, kInvSamples * m, 0, st>>>(S, K, Ainv, ns);
             else if (n0 == 3) k_coarse_inverse<T, 3><<<grid, kInvSamples * m, 0, st>>>(S, K, Ainv, ns);
             else k_coarse_inverse<T, 4><<<grid, kInvSamples * m, 0, st>>>(S, K, Ainv, ns));
}

// p = A^{-1} b on the coarsest grid; one thread per (sample, unknown).
template <typename T>
__global__ void k_coarse_solve(int m, size_t S, const T* __restrict__ Ainv, const T* __restrict__ b,
                               T* __restrict__ p, const int32_t* __restrict__ active) {
    const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= S * m) return;
    const size_t s = t / m;
    if (inactive(active, s)) return;
    const int r = (int)(t % m);
    const T* row = Ainv + s * (size_t)m * m + (size_t)r * m;
    const T* bs = b + s * m;
    T acc = T(0);
    for (int c = 0; c < m; ++c) acc += row[c] * bs[c];
    p[t] = acc;
}

// The QoI of Table 1, one warp per sample.  Case II: the east outflux
// Q = sum_j 2 K_(n-1,j) (p_(n-1,j) - pE), shuffle reduction.  Case I:
// u(0.5, 0.5), the mean of the four cells at the centre.
template <typename P>
__global__ void k_outflux(int n, size_t S, const double* __restrict__ K, const P* __restrict__ p, Bnd bd,
                          double* __restrict__ q) {
    const size_t warp = ((size_t)blockIdx.x * blockDim.x + threadIdx.x) / 32;
    const int lane = threadIdx.x & 31;
    if (warp >= S) return;
    if (bd.ns) {
        if (lane == 0) {
            const size_t c = warp * (size_t)n * n + (size_t)(n / 2 - 1) * n + n / 2 - 1;
            q[warp] = 0.25 * (((double)p[c] + (double)p[c + 1]) + ((double)p[c + n] + (double)p[c + n + 1]));
        }
        return;
    }
    const size_t base = warp * (size_t)n * n + (n - 1);
    double acc = 0.0;
    for (int j = lane; j < n; j += 32)
        acc += 2.0 * K[base + (size_t)j * n] * ((double)p[base + (size_t)j * n] - bd.g[1]);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, off);
    if (lane == 0) q[warp] = acc;
}

__global__ void k_fill(size_t count, double v, double* __restrict__ x) {
    const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t < count) x[t] = v;
}

// ------------------------------------------------------------------ refinement kernels
// Per-sample convergence test of the stage problem, split over `chunks`
// CTAs per sample (grid S * chunks, chunk index fastest): each CTA forms the
// residual of its band of rows and writes its partial sums of ||r||^2,
// ||b||^2 and the outflux to partial[(s * chunks + ch) * 3 + 0..2]; the
// mixed form (p64 != null) forms the residual in FP64 from the FP64 grid and
// writes it, rounded, into the FP32 rhs bT with the FP32 correction pT
// zeroed.  k_stage_decide then folds the partials in chunk order.  b / bT
// and p / pT are the same arrays, hence no __restrict__ on them.
// Threads walk rows (a column each, or several rows per pass on grids
// narrower than the block), so no cell index is divided.  The FP64 pipe (1/58 of
// the FP32 rate) bounds this kernel, so a cell off the Dirichlet edges, whose
// rhs is zero (r = -A p, no K load), takes six operations: the residual's
// product and four FMAs, and the square.  Cells on an edge, whose Dirichlet
// term and QoI share any warp that met one would wait for, come after them,
// one a thread.  An instruction of the FP64 pipe takes its turn also where its
// predicate is off for the whole warp, so there are none beside those six: 1000
// samples of 256 x 256 from 546 us a test on average to 319 (an eighth of the
// time: the sums across the warp).
template <typename T>
__global__ void k_stage_partials(int n, size_t S, int chunks, const double* __restrict__ K, Bnd bd,
                                 const T* b, const T* __restrict__ Te, const T* __restrict__ Tn,
                                 const T* __restrict__ D, const T* p, const double* __restrict__ p64,
                                 const double* __restrict__ Te64, const double* __restrict__ Tn64,
                                 const double* __restrict__ D64, T* bT, T* pT, const int32_t* __restrict__ active,
                                 double* __restrict__ partial, const int32_t* __restrict__ order) {
    __shared__ double red[3][32];
    // S: the samples enumerated (listed by order, if given)
    if (blockIdx.x / chunks >= S) return;
    const size_t s = order ? (size_t)order[blockIdx.x / chunks] : blockIdx.x / chunks;
    const int ch = (int)(blockIdx.x % chunks);
    if (inactive(active, s)) return;
    const size_t base = s * (size_t)n * n;
    const int rows = (n + chunks - 1) / chunks;
    const int j0 = ch * rows, j1 = min(n, j0 + rows);
    // thread -> first column i0 and row offset jo; a pass covers rpi rows
    const int nt = (int)blockDim.x;
    const bool wide = n >= nt;
    const int rpi = wide ? 1 : nt / n;
    const int i0 = wide ? (int)threadIdx.x : (int)threadIdx.x % n;
    const int jo = wide ? 0 : (int)threadIdx.x / n;
    const int istep = wide ? nt : n;
    double rr = 0.0, bb = 0.0, qq = 0.0;
    // the residual at cell (i, j) (interior: rhs zero), rounded into bT in the mixed form
    auto residual = [&](int i, int j, bool interior, double f) {
        const size_t g = base + (size_t)j * n + i;
        double r;
        if (p64) {
            double v = D64[g] * p64[g];
            if (interior || i > 0) v = fma(-Te64[g - 1], p64[g - 1], v);
            if (interior || i < n - 1) v = fma(-Te64[g], p64[g + 1], v);
            if (j > 0) v = fma(-Tn64[g - n], p64[g - n], v);
            if (j < n - 1) v = fma(-Tn64[g], p64[g + n], v);
            // (the sign changes in FP32: negated in FP64 it was an addition more a cell)
            r = interior ? v : f - v;
            bT[g] = interior ? -rounded<T>(r) : rounded<T>(r);
            if (pT) pT[g] = T(0);
        } else {
            r = widen(residual_at(n, g, i, j, b, Te, Tn, D, p));
        }
        rr = fma(r, r, rr);
    };
    const int ja = max(j0, bd.ns ? 1 : 0), jb = min(j1, bd.ns ? n - 1 : n);   // rows with interior cells
    if (jo < rpi) {
        for (int j = ja + jo; j < jb; j += rpi)
            for (int i = i0; i < n; i += istep)
                if (i > 0 && i < n - 1) residual(i, j, true, 0.0);
    }
    // the chunk's west and east columns, and in Case I what is left of its south and north rows
    const int cols = 2 * max(0, j1 - j0);
    const int south = bd.ns && j0 == 0 ? n - 2 : 0, north = bd.ns && j1 == n && j0 < n ? n - 2 : 0;
    for (int t = (int)threadIdx.x; t < cols + south + north; t += nt) {
        const int i = t < cols ? (t & 1) * (n - 1) : 1 + (t - cols) % (n - 2);
        const int j = t < cols ? j0 + (t >> 1) : (t - cols < south ? 0 : n - 1);
        const size_t g = base + (size_t)j * n + i;
        const double f = dirichlet_rhs(bd, n, i, j, K[g]);
        residual(i, j, false, f);
        bb = fma(f, f, bb);
        if (!bd.ns && i == n - 1) qq += 2.0 * K[g] * ((p64 ? p64[g] : widen(p[g])) - bd.g[1]);
    }
    if (bd.ns && threadIdx.x < 4) {   // Case I: the four centre cells
        const int i = n / 2 - 1 + (threadIdx.x & 1), j = n / 2 - 1 + (threadIdx.x >> 1);
        const size_t g = base + (size_t)j * n + i;
        if (j >= j0 && j < j1) qq = 0.25 * (p64 ? p64[g] : widen(p[g]));
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) rr += __shfl_down_sync(0xffffffffu, rr, off);
    // most warps met no edge (bits: an FP64 comparison costs as much as an addition)
    if (__any_sync(0xffffffffu, (__double_as_longlong(bb) | __double_as_longlong(qq)) != 0)) {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            bb += __shfl_down_sync(0xffffffffu, bb, off);
            qq += __shfl_down_sync(0xffffffffu, qq, off);
        }
    }
    if ((threadIdx.x & 31) == 0) {
        red[0][threadIdx.x >> 5] = rr;
        red[1][threadIdx.x >> 5] = bb;
        red[2][threadIdx.x >> 5] = qq;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double a = 0.0, b2 = 0.0, q = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
            a += red[0][w];
            b2 += red[1][w];
            q += red[2][w];
        }
        double* out = partial + ((size_t)s * chunks + ch) * 3;
        out[0] = a;
        out[1] = b2;
        out[2] = q;
    }
}

// The test itself, one warp per sample: active[s] = ||b - A p|| > tol ||b||
// and the last pass moved the outflux by more than qtol |Q|; counted in *left.
__global__ void k_stage_decide(size_t S, int chunks, const double* __restrict__ partial, double tol, double qtol,
                               double* __restrict__ qprev, int32_t* __restrict__ active, int32_t* __restrict__ left,
                               int32_t* __restrict__ order) {
    const size_t s = ((size_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (s >= S || inactive(active, s)) return;
    double a = 0.0, b2 = 0.0, q = 0.0;
    for (int ch = (int)(threadIdx.x & 31); ch < chunks; ch += 32) {
        const double* v = partial + ((size_t)s * chunks + ch) * 3;
        a += v[0];
        b2 += v[1];
        q += v[2];
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        a += __shfl_down_sync(0xffffffffu, a, off);
        b2 += __shfl_down_sync(0xffffffffu, b2, off);
        q += __shfl_down_sync(0xffffffffu, q, off);
    }
    if (threadIdx.x & 31) return;
    const bool done = a <= tol * tol * b2 || (qtol > 0 && fabs(q - qprev[s]) <= qtol * fabs(q));
    qprev[s] = q;
    active[s] = done ? 0 : 1;
    if (!done) {   // count it and list it (in no particular order) for launches over the active samples
        const int i = atomicAdd(left, 1);
        if (order) order[i] = (int32_t)s;
    }
}

// Mixed form: the FP64 refinement update p64 += e (the FP32 correction).
// Grid-stride over the enumerated cells: S samples (listed by order, if
// given), or with dcount (inside a graph's refinement loop) the count the
// last residual test left, so a launch sized for every sample does little
// work once few of them still iterate.  Cells go by pairs where a grid has an
// even number of them.
template <typename T>
__global__ void k_ir_update(int n, size_t S, const T* __restrict__ e, double* __restrict__ p64,
                            const int32_t* __restrict__ active, const int32_t* __restrict__ order,
                            const int32_t* __restrict__ dcount) {
    using V2 = typename PairOf<T>::type;
    const size_t cells = (size_t)n * n, total = (dcount ? (size_t)*dcount : S) * cells;
    const int w = cells % 2 == 0 ? 2 : 1;
    for (size_t t = ((size_t)blockIdx.x * blockDim.x + threadIdx.x) * w; t < total;
         t += (size_t)gridDim.x * blockDim.x * w) {
        const CellAt at = cell_at(t, n);
        const size_t s = order ? (size_t)order[at.s] : at.s;
        if (inactive(active, s)) continue;
        const size_t g = s * cells + at.c;
        if (w == 1) {
            p64[g] += widen(e[g]);
            continue;
        }
        const V2 v = *reinterpret_cast<const V2*>(e + g);
        double2 p = *reinterpret_cast<const double2*>(p64 + g);
        p.x += widen(v.x);
        p.y += widen(v.y);
        *reinterpret_cast<double2*>(p64 + g) = p;
    }
}

template <typename T>
__global__ void k_widen(size_t count, const T* __restrict__ x, double* __restrict__ y) {
    const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t < count) y[t] = widen(x[t]);
}

__global__ void k_status(size_t S, const int32_t* __restrict__ active, int32_t* __restrict__ status) {
    const size_t s = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (s < S && active[s]) status[s] = FM_ENOTCONV;
}

// ------------------------------------------------------------------ V-cycle tail
// The part of a level-wise V-cycle below a correction grid of at most 32 x 32
// cells, per sample in shared memory: pre-smoothing, residual and restriction
// down to the coarsest grid, its solve, then prolongation and post-smoothing
// back up.  One CTA per listed sample replaces the per-grid launches of those
// grids (several tiny launches per grid and cycle).  Every operation is the
// level-wise kernels' own, in their order and rounding: sweeps in colour
// order with the faces W, E, S, N fused into the accumulator and the
// reciprocal of D, residuals as residual_at forms them, restriction sums in
// k_residual_restrict's order, the coarse product as k_coarse_solve sums it,
// corrections as prolong_vals forms them; so the result is the per-grid
// schedule's bit for bit (up to the sign of a zero).
constexpr int kTailMaxN = 32;
constexpr int kTailThreads = 128;

template <typename T>
struct TailArgs {
    int kt, n0, nu1, nu2, ns;               // grids 0 .. kt, n_j = n0 << j; ns: Dirichlet north / south
    size_t S;                               // samples enumerated (the listed ones, with order)
    const T* Te[8];                         // correction operators of grids 0 .. kt
    const T* Tn[8];
    const T* D[8];
    const T* rD[8];                         // their reciprocals, where the hierarchy holds them (FP64)
    const T* b;                             // rhs of grid kt [..][n_kt^2]
    T* p;                                   // out: the correction on grid kt
    const T* Ainv;                          // coarsest correction operator's inverse [..][m][m]
    const int32_t* active;
    const int32_t* order;
};

template <typename T>
__host__ __device__ inline size_t tail_smem_bytes(int kt, int n0) {
    size_t cells = 0;
    for (int j = 0; j <= kt; ++j) cells += (size_t)(n0 << j) * (n0 << j);
    return (6 * cells + (size_t)n0 * n0 * n0 * n0) * sizeof(T);
}

// The largest tail footprint over every coarsest size (2, 3, 4) and the
// deepest correction grid of at most kTailMaxN cells a side above it.
template <typename T>
inline size_t tail_smem_max() {
    size_t m = 0;
    for (int n0 = 2; n0 <= 4; ++n0) {
        int kt = 0;
        while ((n0 << (kt + 1)) <= kTailMaxN) ++kt;
        m = std::max(m, tail_smem_bytes<T>(kt, n0));
    }
    return m;
}

template <typename T>
__global__ void __launch_bounds__(kTailThreads) k_vcycle_tail(TailArgs<T> a) {
    extern __shared__ __align__(16) unsigned char tail_smem[];
    const size_t u = blockIdx.x;
    if (u >= a.S) return;
    const size_t s = a.order ? (size_t)a.order[u] : u;
    if (inactive(a.active, s)) return;
    const int tid = threadIdx.x, nt = blockDim.x;
    // Grid j holds six arrays of n_j^2 = m0 4^j values (te, tn, d, 1/d, b, p)
    // from 6 m0 (4^j - 1) / 3 values into shared memory; the coarsest
    // operator's inverse follows the last grid.  Addresses are formed in
    // registers (no per-grid pointer tables in local memory).
    T* const sm = reinterpret_cast<T*>(tail_smem);
    const int m0 = a.n0 * a.n0;
    auto arr = [&](int j, int q) -> T* { return sm + 2 * m0 * ((1 << (2 * j)) - 1) + q * (m0 << (2 * j)); };
    for (int j = 0; j <= a.kt; ++j) {
        const int c = m0 << (2 * j);
        const T* gte = a.Te[j] + s * (size_t)c;
        const T* gtn = a.Tn[j] + s * (size_t)c;
        const T* gd = a.D[j] + s * (size_t)c;
        const T* gr = a.rD[j] ? a.rD[j] + s * (size_t)c : nullptr;
        T* te = arr(j, 0);
        T* tn = arr(j, 1);
        T* dd = arr(j, 2);
        T* rd = arr(j, 3);
#pragma unroll 4
        for (int e = tid; e < c; e += nt) {
            const T d = gd[e];
            te[e] = gte[e];
            tn[e] = gtn[e];
            dd[e] = d;
            rd[e] = gr ? gr[e] : T(1) / d;
        }
    }
    T* const ainv = arr(a.kt + 1, 0);
    {
        const int c = m0 << (2 * a.kt);
        const T* gb = a.b + s * (size_t)c;
        T* bt = arr(a.kt, 4);
        T* pt = arr(a.kt, 5);
#pragma unroll 4
        for (int e = tid; e < c; e += nt) {
            bt[e] = gb[e];
            pt[e] = T(0);   // the restriction left a zero correction
        }
        const T* gA = a.Ainv + s * (size_t)m0 * m0;
        for (int e = tid; e < m0 * m0; e += nt) ainv[e] = gA[e];
    }
    __syncthreads();
    // Red-black sweeps on grid j: thread -> column pair xh of rows y0, y0 + ry, ...
    // (zero: from a zero iterate, which the first red half-sweep need not read).
    auto sweeps = [&](int j, int nsw, bool zero) {
        const int n = a.n0 << j, hn = n >> 1, ry = nt / hn;
        const int xh = tid % hn, y0 = tid / hn;
        const T* te = arr(j, 0);
        const T* tn = arr(j, 1);
        const T* rd = arr(j, 3);
        const T* bb = arr(j, 4);
        T* pp = arr(j, 5);
        for (int it = 0; it < nsw; ++it)
            for (int color = 0; color < 2; ++color) {
                for (int y = y0; y < n && y0 < ry; y += ry) {
                    const int x = 2 * xh + ((y + color) & 1), c = y * n + x;
                    T acc = bb[c];
                    if (!(zero && it == 0 && color == 0)) {
                        if (x > 0) acc = fma(te[c - 1], pp[c - 1], acc);
                        if (x < n - 1) acc = fma(te[c], pp[c + 1], acc);
                        if (y > 0) acc = fma(tn[c - n], pp[c - n], acc);
                        if (y < n - 1) acc = fma(tn[c], pp[c + n], acc);
                    }
                    pp[c] = acc * rd[c];
                }
                __syncthreads();
            }
    };
    for (int j = a.kt; j >= 1; --j) {
        sweeps(j, a.nu1, true);
        const int nf = a.n0 << j, nc = nf / 2, rc = nt / nc;
        const int I = tid % nc, J0 = tid / nc;
        const T* te = arr(j, 0);
        const T* tn = arr(j, 1);
        const T* dd = arr(j, 2);
        const T* bf = arr(j, 4);
        const T* pf = arr(j, 5);
        T* bc = arr(j - 1, 4);
        T* pc = arr(j - 1, 5);
        for (int J = J0; J < nc && J0 < rc; J += rc) {
            bc[J * nc + I] = restricted_at(nf, (size_t)(2 * J) * nf + 2 * I, I, J, bf, te, tn, dd, pf, a.nu1 > 0);
            pc[J * nc + I] = T(0);
        }
        __syncthreads();
    }
    if (tid < m0) {
        const T* b0 = arr(0, 4);
        T acc = T(0);
        for (int c = 0; c < m0; ++c) acc = fma(ainv[tid * m0 + c], b0[c], acc);
        arr(0, 5)[tid] = acc;
    }
    __syncthreads();
    for (int j = 1; j <= a.kt; ++j) {
        // black cells (column pairs as in the sweeps), which post-smoothing starts
        // from; the red ones too where there is none
        const int nf = a.n0 << j, nc = nf / 2, ry = nt / nc;
        const int xh = tid % nc, y0 = tid / nc;
        const T* pc = arr(j - 1, 5);
        T* pf = arr(j, 5);
        for (int color = 1; color >= (a.nu2 > 0 ? 1 : 0); --color)
            for (int y = y0; y < nf && y0 < ry; y += ry) {
                const int x = 2 * xh + ((y + color) & 1);
                pf[y * nf + x] = pf[y * nf + x] + prolong_err(nc, pc, x, y, a.ns);
            }
        __syncthreads();
        sweeps(j, a.nu2, false);
    }
    const int c = m0 << (2 * a.kt);
    const T* pt = arr(a.kt, 5);
    T* gp = a.p + s * (size_t)c;
#pragma unroll 4
    for (int e = tid; e < c; e += nt) gp[e] = pt[e];
}

// ------------------------------------------------------------------ driver
template <typename T>
struct GridBufs {
    int n;
    const double* K;
    T *Te, *Tn, *D, *p, *b;
    T* p2;                             // second iterate buffer of the tile and strip smoothers
    double* Kc;                        // correction-grid coefficients (k < m)
    T *TeC, *TnC, *DC;                 // their faces and diagonal
    T *rD, *rDC;                       // FP64: reciprocals of D and DC (DC's takes the place of Kc, k >= 1)
    double *p64, *Te64, *Tn64, *D64;   // refined grids of the mixed form only
};

template <typename T>
struct Hierarchy {
    fm_ctx* ctx;
    int m;
    int n0;
    size_t S;
    GridBufs<T> g[FM_MAX_LEVELS + 8];
    T* Ainv;           // coarsest stage operator (injected K)
    T* AinvC;          // coarsest correction operator (child means)
    int32_t* active;   // per-sample iterate flags of converged stages
    int32_t* left;     // count of samples still iterating
    int32_t* iter;     // residual tests done in the current refined stage (graph loops)
    double* qprev;     // outflux of the previous iteration per sample
    double* partial;   // per-(sample, chunk) partial sums of the residual tests
    int32_t* order;    // the samples still iterating, as listed by the last residual test
    // Host-side count of the samples still iterating in a refined stage (the
    // host loop reads it after every test; S otherwise): the strip smoother
    // sizes its row segments for it, so that a launch with few active samples
    // does not march long columns.
    mutable size_t busy = 0;
    // Device-side count of the samples still iterating (the refinement loop
    // of a graph, where the host cannot read it): the strip smoother then
    // enumerates the listed samples itself.
    mutable const int32_t* dcount = nullptr;
    // launches may enumerate only the listed samples
    bool listed() const { return order && busy > 0 && busy < S; }
};

// CTAs per sample of a residual test on grid n (about 8192 cells each).
inline int check_chunks(int n) { return std::max(1, std::min(128, n * n / 8192)); }

// Chunks of a residual test (and of the energy step's sums): four times those,
// eight cells a thread, so that the last tests of a stage, with a few samples
// left, still spread over the SMs (200 fields of 128 x 128, 7 left: 78 us with 2
// chunks a sample).  48 more at most: hierarchy_bytes counts check_chunks and 1.8 KB
// a sample besides.
inline int test_chunks(int n) {
    return std::min(std::max(1, std::min(128, n * n / 2048)), check_chunks(n) + 48);
}

// Bytes of the reciprocal diagonals of one FP64 sample (grids below the
// finest; the finest grid's takes the room counted for its K, the input).
static size_t rdiag_bytes(int n_fine, int n0) {
    size_t total = 0;
    for (int n = n0; n < n_fine; n *= 2) total += (size_t)n * n * 8 + 256;
    return total;
}

static size_t hierarchy_bytes(int n_fine, int n0, size_t S, size_t tsize, bool mixed, bool converged) {
    size_t total = tsize == 8 ? rdiag_bytes(n_fine, n0) : 0;
    int m = 0;
    while ((n0 << m) < n_fine) ++m;
    for (int k = 0; k <= m; ++k) {
        const size_t c = (size_t)(n0 << k) * (n0 << k);
        total += c * (8 + 6 * tsize) + 6 * 256;
        if (k < m) total += c * (8 + 3 * tsize) + 4 * 256;
        if (mixed && k >= m - 1) total += c * 32 + 4 * 256;
    }
    total += 2 * ((size_t)n0 * n0 * n0 * n0 * tsize + 256);
    if (converged) total += 4 * 4 + 16 + (size_t)check_chunks(n_fine) * 24 + 7 * 256;
    return total * S + 4096;
}

int64_t batch_limit(const fm_ctx* ctx, int n) {
    const bool mixed = ctx->cfg.precision == FM_PREC_MIXED;
    const size_t per = hierarchy_bytes(n, std::max(ctx->cfg.n_coarsest, 4), 1, mixed ? 4 : 8, mixed, true) +
                       (size_t)n * n * sizeof(double) + (size_t)ctx->cfg.M * sizeof(double);
    const size_t budget = (size_t)8 << 30;   // 8 GiB of scratch per batch
    int64_t lim = (int64_t)(budget / per);
    if (ctx->cfg.max_batch > 0) lim = std::min<int64_t>(lim, ctx->cfg.max_batch);
    return std::max<int64_t>(lim, 1);
}

bool arena_holds(Arena& ar, size_t need) {
    if (ar.capacity >= need) return true;
    if (ar.base) cudaFree(ar.base);
    ar.base = nullptr;
    ar.capacity = 0;
    if (cudaMalloc((void**)&ar.base, need) != cudaSuccess) {
        cudaGetLastError();
        ar.base = nullptr;
        return false;
    }
    ar.capacity = need;
    return true;
}

// Scratch of a level-wise batch of S samples: grows `ar` when it is too small
// (never while a stream is being captured: callers size it first).
template <typename T>
static fm_status carve(fm_ctx* ctx, Arena& ar, Hierarchy<T>& H, int n_fine, int n0, size_t S, const double* d_K,
                       bool mixed, bool converged) {
    const size_t need = hierarchy_bytes(n_fine, n0, S, sizeof(T), mixed, converged);
    if (!arena_holds(ar, need)) {
        set_error(ctx, "fmg scratch allocation of " + std::to_string(need) + " bytes failed");
        return FM_ENOMEM;
    }
    char* cur = ar.base;
    auto take = [&](size_t bytes) {
        char* p = cur;
        cur += ((bytes + 255) / 256) * 256;
        return p;
    };
    H.ctx = ctx;
    H.n0 = n0;
    H.S = S;
    H.m = 0;
    while ((n0 << H.m) < n_fine) ++H.m;
    for (int k = 0; k <= H.m; ++k) {
        const int n = n0 << k;
        const size_t cnt = S * (size_t)n * n;
        GridBufs<T>& g = H.g[k];
        g.n = n;
        g.K = (k == H.m) ? d_K : (double*)take(cnt * 8);
        g.Te = (T*)take(cnt * sizeof(T));
        g.Tn = (T*)take(cnt * sizeof(T));
        g.D = (T*)take(cnt * sizeof(T));
        g.p = (T*)take(cnt * sizeof(T));
        g.b = (T*)take(cnt * sizeof(T));
        g.p2 = (T*)take(cnt * sizeof(T));
        g.Kc = nullptr;
        g.TeC = g.TnC = g.DC = nullptr;
        if (k < H.m) {
            g.Kc = (double*)take(cnt * 8);
            g.TeC = (T*)take(cnt * sizeof(T));
            g.TnC = (T*)take(cnt * sizeof(T));
            g.DC = (T*)take(cnt * sizeof(T));
        }
        g.rD = g.rDC = nullptr;
        if constexpr (sizeof(T) == 8) {
            g.rD = (T*)take(cnt * 8);
            if (k >= 1) g.rDC = (T*)g.Kc;
        }
        g.p64 = g.Te64 = g.Tn64 = g.D64 = nullptr;
        if (mixed && k >= H.m - 1) {
            g.p64 = (double*)take(cnt * 8);
            g.Te64 = (double*)take(cnt * 8);
            g.Tn64 = (double*)take(cnt * 8);
            g.D64 = (double*)take(cnt * 8);
        }
    }
    H.Ainv = (T*)take(S * (size_t)n0 * n0 * n0 * n0 * sizeof(T));
    H.AinvC = (T*)take(S * (size_t)n0 * n0 * n0 * n0 * sizeof(T));
    H.active = converged ? (int32_t*)take(S * 4) : nullptr;
    H.left = converged ? (int32_t*)take(4) : nullptr;
    H.iter = converged ? (int32_t*)take(4) : nullptr;
    H.qprev = converged ? (double*)take(S * 8) : nullptr;
    H.partial = converged ? (double*)take(S * (size_t)test_chunks(n_fine) * 24) : nullptr;
    H.order = converged ? (int32_t*)take(S * 4) : nullptr;
    return FM_OK;
}

constexpr size_t kMaxSmem = 200 * 1024;   // dynamic shared memory of the tile smoother

// Kernel attributes and occupancies, set once on every device before any launch
// or capture there.
void fmg_init_attributes(int device) {
    static OncePerDevice once;
    once.run(device, [&] {
        cudaFuncSetAttribute(k_rbgs_tile<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxSmem);
        cudaFuncSetAttribute(k_rbgs_tile<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxSmem);
        cudaFuncSetAttribute(k_vcycle_tail<float>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)tail_smem_max<float>());
        cudaFuncSetAttribute(k_vcycle_tail<double>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)tail_smem_max<double>());
        warp16_init();
        team32_init();
        int sms = 1;
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
        strip_init<float>(sms);
        strip_init<double>(sms);
        cudaGetLastError();
    });
}

// Launch shape code of the column-strip smoother (fmg_strip.cuh; tile codes are > 0, colour launches 0).
constexpr int kShapeStrip = -1;

static size_t tile_smem_bytes(int tile, int n, int nsweeps, size_t tsize) {
    const int TI = std::min(tile, n);
    const int hh = TI >= n ? 0 : 2 * nsweeps;
    const int RW = std::min(TI + 2 * hh, n);
    return 5 * (size_t)RW * RW * tsize;
}

// Launch shape `tile` (tile interior staged in shared memory, p_in -> p_out;
// 0: one launch per colour and sweep, in place on p_in) with `threads` per
// CTA.  Returns the buffer that holds the result.  With ec (tile shapes
// only), the iterate is p_in + P ec, the coarse-grid correction added as
// the tiles load.
template <typename T>
static T* smooth_with(fm_ctx* ctx, int tile, int threads, int n, size_t S, int nsweeps, const T* b, const T* Te,
                      const T* Tn, const T* D, const T* rD, T* p_in, T* p_out, const int32_t* active,
                      cudaStream_t st, const T* ec = nullptr, int ns = 0) {
    if (nsweeps <= 0) return p_in;
    const size_t cells = S * (size_t)n * n;
    if (tile > 0) {
        const int TI = std::min(tile, n);
        const int hh = TI >= n ? 0 : 2 * nsweeps;
        const int tiles = (n + TI - 1) / TI;
        const unsigned grid = (unsigned)(S * tiles * tiles);
        const double bytes = 6.0 * sizeof(T) * cells, flops = 10.0 * nsweeps * cells;
        // register-blocked regions (threads == 0): whole grids of 8, 16, 32
        // (and, FP32, 64) cells, or 32 (and, FP32, 64) interiors with a halo of
        // up to 4 (nsweeps <= 2); FP64 copies of the large regions would spill
        constexpr bool f32 = sizeof(T) == 4;
        if (threads == 0 && hh == 0 && (n == 8 || n == 16 || n == 32 || (f32 && n == 64))) {
            if (n == 8)
                FM_TIMED(ctx, kFamSmootherTile, st, bytes, flops, k_rbgs_tile_reg<T, 8, 1><<<grid, 4 * 8, 0, st>>>(
                    n, S, TI, hh, nsweeps, b, Te, Tn, D, rD, p_in, p_out, active, ec, ns));
            else if (n == 16)
                FM_TIMED(ctx, kFamSmootherTile, st, bytes, flops, k_rbgs_tile_reg<T, 16, 2><<<grid, 8 * 8, 0, st>>>(
                    n, S, TI, hh, nsweeps, b, Te, Tn, D, rD, p_in, p_out, active, ec, ns));
            else if (n == 32)
                FM_TIMED(ctx, kFamSmootherTile, st, bytes, flops, k_rbgs_tile_reg<T, 32, 4><<<grid, 16 * 8, 0, st>>>(
                    n, S, TI, hh, nsweeps, b, Te, Tn, D, rD, p_in, p_out, active, ec, ns));
            else if constexpr (f32)
                FM_TIMED(ctx, kFamSmootherTile, st, bytes, flops, k_rbgs_tile_reg<T, 64, 8><<<grid, 32 * 8, 0, st>>>(
                    n, S, TI, hh, nsweeps, b, Te, Tn, D, rD, p_in, p_out, active, ec, ns));
            return p_out;
        }
        if (threads == 0 && hh > 0 && hh <= 4 && (TI == 32 || (f32 && TI == 64))) {
            if (TI == 32)
                FM_TIMED(ctx, kFamSmootherTile, st, bytes, flops, k_rbgs_tile_reg<T, 40, 5><<<grid, 20 * 8, 0, st>>>(
                    n, S, TI, hh, nsweeps, b, Te, Tn, D, rD, p_in, p_out, active, ec, ns));
            else if constexpr (f32)
                FM_TIMED(ctx, kFamSmootherTile, st, bytes, flops, k_rbgs_tile_reg<T, 72, 9><<<grid, 36 * 8, 0, st>>>(
                    n, S, TI, hh, nsweeps, b, Te, Tn, D, rD, p_in, p_out, active, ec, ns));
            return p_out;
        }
        FM_TIMED(ctx, kFamSmootherTile, st, bytes, flops,
                 k_rbgs_tile<T><<<grid, threads > 0 ? threads : 256, tile_smem_bytes(tile, n, nsweeps, sizeof(T)),
                                  st>>>(n, S, TI, hh, nsweeps, b, Te, Tn, D, rD, p_in, p_out, active, ec, ns));
        return p_out;
    }
    T* p = p_in;
    const size_t half = cells / 2;
    for (int it = 0; it < nsweeps; ++it)
        for (int color = 0; color < 2; ++color)
            FM_TIMED(ctx, kFamSmoother, st, 3.0 * sizeof(T) * cells, 5.0 * cells,
                     k_rbgs_color<T><<<blocks_for(half), kBlock, 0, st>>>(n, S, color, b, Te, Tn, D, rD, p, active));
    return p;
}

static int tune_slot(int n) { return std::min(15, 31 - __builtin_clz((unsigned)n)); }

// Smoother launch shape of grid n.  Untuned defaults (fastest on GB300 for two
// sweeps): column strips from 64 x 64 (FP64 strips against one launch per colour,
// fixed schedule: 64 x 64, 5000 samples 12.0 / 14.0 ms; 128 x 128, 1000 samples 8.9 /
// 11.5; 256 x 256, 250 samples 9.2 / 11.8).  32 x 32 and 16 x 16 in FP32: strips too,
// with several samples in a warp (converged mixed solves, register-blocked regions
// / strips on both: 64 x 64, 1000 samples 3.88 / 3.47 ms, 5000 12.1 / 10.5; 32 x 32
// level-wise, 300 samples 1.97 / 1.69, 15000 14.6 / 8.9).  In FP64: one staged
// region a sample (fixed schedule, register-blocked / staged / strips: 32 x 32, 15000
// samples 5.00 / 4.72 / 5.03; 64 x 64, 5000 samples 6.25 / 6.12 / 6.40; converged 32 x
// 32, 15000 samples 28.7 / 26.5 / 28.5; level on a few hundred samples).  FP64 grids from 64 x 64
// of less than 2 Mi cells in the whole batch (1 Mi at 64 x 64): colour launches, since
// a strip marches its rows one after the other and few strips leave the SMs waiting
// (fixed schedule, strips / colours: one sample of 256 x 256 1.48 / 1.07 ms, 32 1.93 /
// 1.72, 64 level; one of 1024 x 1024 3.15 / 2.24, four 3.99 / 3.43 with strips on the
// finest 3.32; 160 of 64 x 64 0.77 / 0.73, 400 0.95 / 0.99).  Below, and
// where strips do not fit: one register-blocked region a sample.  An fm_autotune or
// fm_set_smoother_shape entry for this grid and precision replaces the
// default; the tuner times 64 Mi cells, so strips it has chosen give way to colour
// launches below the same lines, and those set by hand do not.  Tiles and strips need both smoothing phases of the V-cycle (so
// the iterate goes p -> p2 -> p); tiles need their staged region in shared
// memory, strips 1 or 2 sweeps.
template <typename T>
static void smooth_shape(const fm_ctx* ctx, int n, size_t S, const fm_solve_params& prm, int* tile, int* threads) {
    const int pi = sizeof(T) == 4 ? 1 : 0, slot = tune_slot(n);
    *threads = 0;
    *tile = n <= 32 ? 32 : kShapeStrip;   // 32: one region per sample, register-blocked
    if (n == 16 || n == 32) {
        if (sizeof(T) == 8) *threads = 8 * n;   // staged
        else if (strip_fits(n, prm.nu1, prm.nu2)) *tile = kShapeStrip;
    }
    const bool entry = ctx->tune.n[pi][slot] == n;
    if (entry) {
        *tile = ctx->tune.tile[pi][slot];
        *threads = ctx->tune.threads[pi][slot];
    }
    const bool by_hand = entry && ctx->tune.by_hand[pi][slot];
    if (sizeof(T) == 8 && n >= 64 && *tile == kShapeStrip && !by_hand &&
        S * n * n < ((size_t)1 << (n > 64 ? 21 : 20)))
        *tile = 0;
    if (*tile > 0 && (prm.nu1 < 1 || prm.nu2 < 1 ||
                      tile_smem_bytes(*tile, n, std::max(prm.nu1, prm.nu2), sizeof(T)) > kMaxSmem))
        *tile = 0;
    if (*tile == kShapeStrip && !strip_fits(n, prm.nu1, prm.nu2)) *tile = 0;
}

// The V-cycle below correction grid kt (<= 32 x 32) as one resident tail
// launch over the listed samples (k_vcycle_tail).
template <typename T>
static void vcycle_tail(const Hierarchy<T>& H, int kt, const fm_solve_params& prm, const int32_t* active,
                        cudaStream_t st) {
    fm_ctx* ctx = H.ctx;
    TailArgs<T> a{};
    a.kt = kt;
    a.n0 = H.n0;
    a.nu1 = prm.nu1;
    a.nu2 = prm.nu2;
    a.ns = prm.bc_case == FM_CASE_I ? 1 : 0;
    const bool listed = H.listed();
    a.S = listed ? H.busy : H.S;
    double cells = 0.0;
    for (int j = 0; j <= kt; ++j) {
        a.Te[j] = H.g[j].TeC;
        a.Tn[j] = H.g[j].TnC;
        a.D[j] = H.g[j].DC;
        a.rD[j] = H.g[j].rDC;
        cells += (double)H.g[j].n * H.g[j].n;
    }
    a.b = H.g[kt].b;
    a.p = H.g[kt].p;
    a.Ainv = H.AinvC;
    a.active = active;
    a.order = listed ? H.order : nullptr;
    const double top = (double)H.g[kt].n * H.g[kt].n;
    const double bytes = (3.0 * cells + 2.0 * top) * sizeof(T) * a.S;
    const double flops = (10.0 * (prm.nu1 + prm.nu2) + 18.0) * cells * a.S;
    if constexpr (sizeof(T) == 4) {
        if (kt == 3 && H.n0 == 4) {   // 4, 8, 16, 32: in registers
            Tail32Args t{};
            t.nu1 = a.nu1;
            t.nu2 = a.nu2;
            t.ns = a.ns;
            for (int j = 0; j < 3; ++j) {
                t.Te[j] = a.Te[j + 1];
                t.Tn[j] = a.Tn[j + 1];
                t.D[j] = a.D[j + 1];
            }
            t.Ainv = a.Ainv;
            t.b = a.b;
            t.p = a.p;
            t.active = a.active;
            t.order = a.order;
            FM_TIMED(ctx, kFamVcycleTail, st, bytes, flops, launch_tail32(t, a.S, st));
            return;
        }
    }
    FM_TIMED(ctx, kFamVcycleTail, st, bytes, flops,
             k_vcycle_tail<T><<<(unsigned)a.S, kTailThreads, tail_smem_bytes<T>(kt, H.n0), st>>>(a));
}

// Whether the smoother of correction grid k reads the zero iterate that the
// restriction leaves there: the coarsest solve, the tail and the strips don't.
template <typename T>
static bool reads_zero(const Hierarchy<T>& H, int k, const fm_solve_params& prm) {
    if (k == 0) return false;
    if (H.g[k].n <= H.ctx->tail_max && !prm.energy_step) return false;
    int tile, threads;
    smooth_shape<T>(H.ctx, H.g[k].n, H.S, prm, &tile, &threads);
    return tile != kShapeStrip;
}

// Where `count` V-cycles on grid k read their starting iterate: p, or p2
// where merged strips (see vcycles) pass through the two buffers an odd
// number of times; the result is always in p.
template <typename T>
static T* start_iterate(const Hierarchy<T>& H, int k, const fm_solve_params& prm, int count) {
    int tile, threads;
    smooth_shape<T>(H.ctx, H.g[k].n, H.S, prm, &tile, &threads);
    const bool merged = k > 0 && tile == kShapeStrip && count > 1 && strip_merges<T>(prm.nu1, prm.nu2);
    return merged && count % 2 == 0 ? H.g[k].p2 : H.g[k].p;
}

// The energy-optimal step of the correction on grid c.n onto iterate x of
// grid k: partial sums, then alpha and x += alpha P e_c.
template <typename T>
static void energy_step(const Hierarchy<T>& H, int k, const T* Te, const T* Tn, const T* D, T* x, const int32_t* active,
                        int ns, cudaStream_t st) {
    fm_ctx* ctx = H.ctx;
    const GridBufs<T>& g = H.g[k];
    const GridBufs<T>& c = H.g[k - 1];
    const double ts = sizeof(T);
    // bands of four coarse rows at least, as many as the sample's slots hold: few
    // large fields leave the coarser grids' launches with a few warps otherwise
    const int chunks = std::max(1, std::min(test_chunks(H.g[H.m].n), c.n / 4));
    const bool listed = H.listed();
    const size_t nl = listed ? H.busy : H.S;
    const int blocks = std::max(1, (int)(((size_t)c.n * c.n + 256 * kStepCells - 1) / (256 * kStepCells)));
    FM_TIMED(ctx, kFamProlong, st, (5.0 * ts + 1.25 * ts) * nl * g.n * g.n + 2.0 * ts * nl * g.n * g.n, 40.0 * nl * g.n * g.n,
             k_energy_partials<T><<<(unsigned)(nl * chunks), 256, 0, st>>>(
                 g.n, nl, chunks, g.b, Te, Tn, D, x, c.p, active, listed ? H.order : nullptr, H.partial, ns);
             k_energy_apply<T><<<(unsigned)(nl * blocks), 256, 0, st>>>(c.n, nl, chunks, blocks, c.p, H.partial, x,
                                                                        active, listed ? H.order : nullptr, ns));
}

// `count` V(nu1, nu2) cycles on grid k, from start_iterate (zero: from a zero
// iterate, which need not be in memory where the shape is the strip's) to
// g.p; grid `top` carries the stage operator (injected K), the grids below
// it the correction operators (child means).
//
// Strips with nu1 = nu2 run the post-smoothing of a cycle and the
// pre-smoothing of the next as one call (the same sweeps in the same order):
// count + 1 passes over the grid instead of 2 count.
template <typename T>
static void vcycles(const Hierarchy<T>& H, int k, int top, const fm_solve_params& prm, const int32_t* active,
                    cudaStream_t st, int count, bool zero) {
    fm_ctx* ctx = H.ctx;
    const size_t S = H.S;
    const GridBufs<T>& g = H.g[k];
    const double ts = sizeof(T);
    const bool stage_op = (k == top);
    const int ns = prm.bc_case == FM_CASE_I ? 1 : 0;   // Dirichlet north / south edges (Table 1, Case I)
    const T* Te = stage_op ? g.Te : g.TeC;
    const T* Tn = stage_op ? g.Tn : g.TnC;
    const T* D = stage_op ? g.D : g.DC;
    const T* rD = stage_op ? g.rD : g.rDC;
    if (k == 0) {
        const int m = H.n0 * H.n0;
        FM_TIMED(ctx, kFamCoarseSolve, st, (double)S * (m * m + 2 * m) * ts, 2.0 * S * m * m,
                 k_coarse_solve<T><<<blocks_for(S * m), kBlock, 0, st>>>(m, S, stage_op ? H.Ainv : H.AinvC, g.b,
                                                                         g.p, active));
        return;
    }
    const int n = g.n;
    const size_t cells = S * (size_t)n * n;
    const GridBufs<T>& c = H.g[k - 1];
    int tile, threads;
    smooth_shape<T>(ctx, n, S, prm, &tile, &threads);
    T* const pc = reads_zero(H, k - 1, prm) ? c.p : nullptr;   // the coarse iterate, where it must be zeroed
    // the V-cycle below: the resident tail for correction grids up to
    // ctx->tail_max, else grid by grid
    auto below = [&] {
        if (k - 1 >= 1 && c.n <= ctx->tail_max && !prm.energy_step && S > 0) vcycle_tail(H, k - 1, prm, active, st);
        else vcycles(H, k - 1, top, prm, active, st, 1, true);
    };
    if (tile == kShapeStrip) {
        const bool merge = count > 1 && strip_merges<T>(prm.nu1, prm.nu2);
        T* cur = start_iterate(H, k, prm, count);
        auto strip = [&](int sweeps, bool fuse, bool from_zero, bool correct) {
            StripCall<T> s;
            s.n = n;
            s.S = S;
            s.hs = 2 * sweeps;
            s.fuse = fuse;
            s.b = g.b;
            s.Te = Te;
            s.Tn = Tn;
            s.D = D;
            s.rD = rD;
            s.p_in = from_zero ? nullptr : cur;
            s.p_out = cur == g.p ? g.p2 : g.p;
            s.active = active;
            s.ec = correct ? c.p : nullptr;
            s.bc = c.b;
            s.pc = pc;
            s.order = H.order;
            s.busy = H.busy;
            s.dcount = H.dcount;
            s.ns = ns;
            strip_launch(ctx, s, st);
            cur = s.p_out;
        };
        for (int it = 0; it < count; ++it) {
            // pre-smoothing with the residual and its restriction in the same pass
            if (it == 0 || !merge) strip(prm.nu1, true, zero && it == 0, false);
            below();
            if (prm.energy_step) energy_step(H, k, Te, Tn, D, cur, active, ns, st);
            const bool next = merge && it + 1 < count;
            strip(next ? prm.nu1 + prm.nu2 : prm.nu2, next, false, !prm.energy_step);
        }
        return;
    }
    for (int it = 0; it < count; ++it) {
        // pre-smoothing p -> p2 (tiles) or in place; post-smoothing back into p
        T* cur = smooth_with<T>(ctx, tile, threads, n, S, prm.nu1, g.b, Te, Tn, D, rD, g.p, g.p2, active, st, nullptr, ns);
        FM_TIMED(ctx, kFamResidualRestrict, st, 5.5 * ts * cells, 10.0 * cells,
                 k_residual_restrict<T><<<blocks_for(S * (size_t)c.n * c.n), kBlock, 0, st>>>(
                     c.n, S, g.b, Te, Tn, D, cur, c.b, c.p, active, prm.nu1 > 0));
        below();
        if (prm.energy_step) {
            // the stepped correction (converged mode: partial sums in the hierarchy)
            energy_step(H, k, Te, Tn, D, cur, active, ns, st);
            smooth_with<T>(ctx, tile, threads, n, S, prm.nu2, g.b, Te, Tn, D, rD, cur, g.p, active, st, nullptr, ns);
        } else if (tile == 0 && prm.nu2 >= 1) {
            // colour launches: the correction rides in the first post-smoothing colour
            FM_TIMED(ctx, kFamSmoother, st, 3.0 * ts * cells + ts * S * c.n * c.n, 5.0 * cells,
                     k_rbgs_color0_prolong<T><<<blocks_for(cells / 2), kBlock, 0, st>>>(n, S, g.b, Te, Tn, D, rD,
                                                                                        cur, c.p, active, ns));
            FM_TIMED(ctx, kFamSmoother, st, 3.0 * ts * cells, 5.0 * cells,
                     k_rbgs_color<T><<<blocks_for(cells / 2), kBlock, 0, st>>>(n, S, 1, g.b, Te, Tn, D, rD, cur,
                                                                               active));
            smooth_with<T>(ctx, 0, 0, n, S, prm.nu2 - 1, g.b, Te, Tn, D, rD, cur, g.p, active, st);
        } else if (tile != 0 && prm.nu2 >= 1) {
            // tiles: the correction is added as they load the iterate
            smooth_with<T>(ctx, tile, threads, n, S, prm.nu2, g.b, Te, Tn, D, rD, cur, g.p, active, st, c.p, ns);
        } else {
            const Ghost<T> zg{T(0), T(0), T(0), T(0), ns};
            FM_TIMED(ctx, kFamProlong, st, 2.25 * ts * cells, 8.0 * cells,
                     k_prolong<T><<<blocks_for(ring_threads(S, n)), kBlock, 0, st>>>(c.n, S, c.p, zg, 1, cur,
                                                                                        active));
            smooth_with<T>(ctx, tile, threads, n, S, prm.nu2, g.b, Te, Tn, D, rD, cur, g.p, active, st, nullptr, ns);
        }
    }
}

template <typename P>
static void outflux(fm_ctx* ctx, int n, size_t S, const double* K, const P* p, const Bnd& bd, double* q,
                    cudaStream_t st) {
    FM_TIMED(ctx, kFamOutflux, st, 16.0 * S * n, 3.0 * S * n,
             k_outflux<P><<<blocks_for(S * 32), kBlock, 0, st>>>(n, S, K, p, bd, q));
}

// One residual test of the refined stage on grid k (partials, then the decision).
template <typename T>
static void stage_test(const Hierarchy<T>& H, int k, const fm_solve_params& prm, bool mixed, cudaStream_t st) {
    fm_ctx* ctx = H.ctx;
    const GridBufs<T>& g = H.g[k];
    const size_t S = H.S, cells = (size_t)g.n * g.n;
    const int chunks = test_chunks(g.n);
    const size_t ns = H.listed() ? H.busy : S;
    int tile, threads;
    smooth_shape<T>(ctx, g.n, S, prm, &tile, &threads);
    T* const pT = tile == kShapeStrip ? nullptr : g.p;   // strips start from zero without reading it
    FM_TIMED(ctx, kFamResidualRestrict, st, (mixed ? 48.0 : 40.0) * ns * cells, 12.0 * ns * cells,
             k_stage_partials<T><<<(unsigned)(ns * chunks), kBlock, 0, st>>>(
                 g.n, ns, chunks, g.K, bnd_of(prm), g.b, g.Te, g.Tn, g.D, g.p, g.p64, g.Te64, g.Tn64, g.D64, g.b,
                 pT, H.active, H.partial, H.listed() ? H.order : nullptr);
             k_stage_decide<<<blocks_for(S * 32), kBlock, 0, st>>>(S, chunks, H.partial, prm.tol, prm.qtol, H.qprev,
                                                              H.active, H.left, H.order));
}

// Blocks of a refinement update over `work` cells: enough to fill the GPU a
// few times over, the grid-stride loop takes the rest.
static unsigned ir_update_blocks(const fm_ctx* ctx, size_t work) {
    int sms = 152;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, ctx->device);
    return (unsigned)std::max<size_t>(1, std::min<size_t>(blocks_for(work), (size_t)sms * 16));
}

// Loop control of a refined stage inside a CUDA graph: after residual test
// number *it, another pass runs while a sample is still active and fewer than
// max_cycles tests have been made; the bound ends every loop.
__global__ void k_refine_cond(const int32_t* __restrict__ left, int32_t* __restrict__ it, int max_cycles,
                              cudaGraphConditionalHandle h) {
    const int i = *it;
    *it = i + 1;
    cudaGraphSetConditional(h, (*left > 0 && i < max_cycles) ? 1u : 0u);
}

// The refined stage as a device-side loop of the graph being captured on
// st: a residual test, then a conditional WHILE node whose body is nu0
// V-cycles (masked to the active samples), the FP64 update of the mixed form
// and the next test.  No host synchronisation; the same tests and updates in
// the same order as the host loop of refine_stage.
template <typename T>
static fm_status refine_stage_graph(const Hierarchy<T>& H, int k, const fm_solve_params& prm, bool mixed,
                                    int32_t* status, cudaStream_t st) {
    fm_ctx* ctx = H.ctx;
    const GridBufs<T>& g = H.g[k];
    const size_t S = H.S, cells = (size_t)g.n * g.n;
    cudaStreamCaptureStatus cs;
    cudaGraph_t graph = nullptr;
    const cudaGraphNode_t* deps = nullptr;
    size_t nd = 0;
    FM_CUDA_TRY(ctx, cudaStreamGetCaptureInfo(st, &cs, nullptr, &graph, &deps, nullptr, &nd));
    cudaGraphConditionalHandle h;
    FM_CUDA_TRY(ctx, cudaGraphConditionalHandleCreate(&h, graph, 0, cudaGraphCondAssignDefault));
    auto test = [&](cudaStream_t s) {
        cudaMemsetAsync(H.left, 0, sizeof(int32_t), s);
        stage_test(H, k, prm, mixed, s);
        k_refine_cond<<<1, 1, 0, s>>>(H.left, H.iter, prm.max_cycles, h);
    };
    FM_CUDA_TRY(ctx, cudaMemsetAsync(H.active, 0xff, S * sizeof(int32_t), st));   // all active (-1)
    FM_CUDA_TRY(ctx, cudaMemsetAsync(H.qprev, 0xff, S * sizeof(double), st));     // NaN
    FM_CUDA_TRY(ctx, cudaMemsetAsync(H.iter, 0, sizeof(int32_t), st));
    test(st);
    FM_CUDA_TRY(ctx, cudaStreamGetCaptureInfo(st, &cs, nullptr, &graph, &deps, nullptr, &nd));
    cudaGraphNodeParams np = {};
    np.type = cudaGraphNodeTypeConditional;
    np.conditional.handle = h;
    np.conditional.type = cudaGraphCondTypeWhile;
    np.conditional.size = 1;
    cudaGraphNode_t node;
    FM_CUDA_TRY(ctx, cudaGraphAddNode(&node, graph, deps, nullptr, nd, &np));
    FM_CUDA_TRY(ctx, cudaStreamUpdateCaptureDependencies(st, &node, nullptr, 1, cudaStreamSetCaptureDependencies));
    // the body is captured on a stream of the branch's own priority
    int prio = 0;
    FM_CUDA_TRY(ctx, cudaStreamGetPriority(st, &prio));
    prio = std::min(std::max(prio, ctx->prio_hi), ctx->prio_lo);
    cudaStream_t bs = ctx->body_stream[prio - ctx->prio_hi];
    FM_CUDA_TRY(ctx, cudaStreamBeginCaptureToGraph(bs, np.conditional.phGraph_out[0], nullptr, nullptr, 0,
                                                   cudaStreamCaptureModeRelaxed));
    // the body's strips enumerate the samples the last test listed
    H.dcount = H.order ? H.left : nullptr;
    vcycles(H, k, k, prm, H.active, bs, cycles_per_test(prm), mixed);
    H.dcount = nullptr;
    if (mixed)
        k_ir_update<T><<<ir_update_blocks(ctx, S * cells), kBlock, 0, bs>>>(g.n, S, g.p, g.p64, H.active,
                                                                              H.order, H.order ? H.left : nullptr);
    test(bs);
    cudaGraph_t body = nullptr;
    FM_CUDA_TRY(ctx, cudaStreamEndCapture(bs, &body));
    if (status) k_status<<<blocks_for(S), kBlock, 0, st>>>(S, H.active, status);
    return FM_OK;
}

// Cycles of one refined stage until every sample passes its residual test.
template <typename T>
static fm_status refine_stage(const Hierarchy<T>& H, int k, const fm_solve_params& prm, bool mixed,
                              int32_t* status, cudaStream_t st) {
    fm_ctx* ctx = H.ctx;
    cudaStreamCaptureStatus capturing = cudaStreamCaptureStatusNone;
    FM_CUDA_TRY(ctx, cudaStreamIsCapturing(st, &capturing));
    if (capturing == cudaStreamCaptureStatusActive) return refine_stage_graph(H, k, prm, mixed, status, st);
    const GridBufs<T>& g = H.g[k];
    const size_t S = H.S, cells = (size_t)g.n * g.n;
    FM_CUDA_TRY(ctx, cudaMemsetAsync(H.active, 0xff, S * sizeof(int32_t), st));   // all active (-1)
    FM_CUDA_TRY(ctx, cudaMemsetAsync(H.qprev, 0xff, S * sizeof(double), st));     // NaN
    int32_t left = 0;
    for (int it = 0;; ++it) {
        FM_CUDA_TRY(ctx, cudaMemsetAsync(H.left, 0, sizeof(int32_t), st));
        stage_test(H, k, prm, mixed, st);
        FM_CUDA_TRY(ctx, cudaMemcpyAsync(&left, H.left, sizeof(int32_t), cudaMemcpyDeviceToHost, st));
        FM_CUDA_TRY(ctx, cudaStreamSynchronize(st));
        H.busy = left > 0 ? (size_t)left : S;
        if (left == 0) break;
        if (it >= prm.max_cycles) {
            if (status) k_status<<<blocks_for(S), kBlock, 0, st>>>(S, H.active, status);
            break;
        }
        vcycles(H, k, k, prm, H.active, st, cycles_per_test(prm), mixed);
        if (mixed)
            k_ir_update<T><<<ir_update_blocks(ctx, (H.listed() ? H.busy : S) * cells), kBlock, 0, st>>>(
                g.n, H.listed() ? H.busy : S, g.p, g.p64, H.active, H.listed() ? H.order : nullptr, nullptr);
    }
    H.busy = 0;   // later stages run every sample
    return FM_OK;
}

template <typename T>
static fm_status fmg_batch(const Hierarchy<T>& H, const fm_solve_params& prm, double* qf, double* qc,
                           double* p_out, int32_t* status, cudaStream_t st) {
    fm_ctx* ctx = H.ctx;
    const size_t S = H.S;
    const bool mixed = prm.precision == FM_PREC_MIXED;
    const bool conv = prm.converged != 0;
    const double ts = sizeof(T);
    const Bnd bd = bnd_of(prm);
    if (status) FM_CUDA_TRY(ctx, cudaMemsetAsync(status, 0, sizeof(int32_t) * S, st));
    // coefficient hierarchy: inject, then faces and diagonals on every grid
    for (int k = H.m; k >= 1; --k) {
        const int nc = H.g[k - 1].n;
        const size_t cc = S * (size_t)nc * nc;
        FM_TIMED(ctx, kFamInject, st, 16.0 * cc, 0.0,
                 k_inject<<<blocks_for(cc), kBlock, 0, st>>>(nc, S, H.g[k].K, const_cast<double*>(H.g[k - 1].K)));
    }
    for (int k = 0; k <= H.m; ++k) {
        const GridBufs<T>& g = H.g[k];
        const size_t cells = S * (size_t)g.n * g.n;
        // FP64 arithmetic for FP64 grids and for the refined grids' FP64 copies
        if (sizeof(T) == 8 || g.Te64)
            FM_TIMED(ctx, kFamCoefficients, st, (8.0 + 3.0 * ts + (g.Te64 ? 24.0 : 0.0)) * cells, 16.0 * cells,
                     k_faces<T, double><<<blocks_for(cells), kBlock, 0, st>>>(g.n, S, bd.ns, g.K, g.Te, g.Tn,
                                                                              g.Te64, g.Tn64);
                     k_diagonal<T, double><<<blocks_for(cells), kBlock, 0, st>>>(g.n, S, bd.ns, g.K, g.Te, g.Tn,
                                                                                 g.Te64, g.Tn64, g.D, g.D64, g.rD));
        else
            FM_TIMED(ctx, kFamCoefficients, st, (8.0 + 3.0 * ts) * cells, 16.0 * cells,
                     k_faces<T, T><<<blocks_for(cells), kBlock, 0, st>>>(g.n, S, bd.ns, g.K, g.Te, g.Tn, nullptr,
                                                                         nullptr);
                     k_diagonal<T, T><<<blocks_for(cells), kBlock, 0, st>>>(g.n, S, bd.ns, g.K, g.Te, g.Tn, nullptr,
                                                                            nullptr, g.D, nullptr, g.rD));
    }
    for (int k = 0; k < H.m; ++k) {
        const GridBufs<T>& g = H.g[k];
        const size_t cells = S * (size_t)g.n * g.n;
        FM_TIMED(ctx, kFamCoefficients, st, (32.0 + 8.0 + 3.0 * ts) * cells, 40.0 * cells,
                 k_child_geomean<T><<<blocks_for(cells), kBlock, 0, st>>>(g.n, S, H.g[k + 1].K, g.Kc);
                 k_faces<T, T><<<blocks_for(cells), kBlock, 0, st>>>(g.n, S, bd.ns, g.Kc, g.TeC, g.TnC, nullptr,
                                                                     nullptr);
                 k_diagonal<T, T><<<blocks_for(cells), kBlock, 0, st>>>(g.n, S, bd.ns, g.Kc, g.TeC, g.TnC, nullptr,
                                                                        nullptr, g.DC, nullptr, g.rDC));
    }
    if (H.m >= 1) coarse_inverse<T>(ctx, H.n0, S, H.g[0].Kc, H.AinvC, bd.ns, st);
    coarse_inverse<T>(ctx, H.n0, S, H.g[0].K, H.Ainv, bd.ns, st);
    // the stage one grid coarser is refined only where its QoI is asked for:
    // otherwise it just gives the finest stage its starting guess
    const bool refine_c = conv && qc != nullptr;
    for (int k = 0; k <= H.m; ++k) {
        const GridBufs<T>& g = H.g[k];
        const size_t cells = S * (size_t)g.n * g.n;
        const bool refined = conv && (k == H.m || (k == H.m - 1 && refine_c));
        if (k > 0) {
            const GridBufs<T>& c = H.g[k - 1];
            if (mixed && refined && k == H.m && H.m >= 1 && refine_c) {
                FM_TIMED(ctx, kFamFmgInterp, st, 10.0 * cells, 8.0 * cells,
                         k_prolong<double><<<blocks_for(ring_threads(S, g.n)), kBlock, 0, st>>>(
                             c.n, S, c.p64, Ghost<double>{bd.g[0], bd.g[1], bd.g[2], bd.g[3], bd.ns}, 0, g.p64,
                             nullptr));
            } else {
                FM_TIMED(ctx, kFamFmgInterp, st, 1.25 * ts * cells, 8.0 * cells,
                         k_prolong<T><<<blocks_for(ring_threads(S, g.n)), kBlock, 0, st>>>(
                             c.n, S, c.p, Ghost<T>{(T)bd.g[0], (T)bd.g[1], (T)bd.g[2], (T)bd.g[3], bd.ns}, 0,
                             refined ? g.p : start_iterate(H, k, prm, prm.nu0), nullptr));
            }
        }
        // (a refined stage of the mixed form has its first residual written there instead;
        // the coarsest grid is solved first)
        if (!(mixed && refined && k > 0))
            FM_TIMED(ctx, kFamStageRhs, st, ts * cells, 2.0 * cells,
                     k_stage_rhs<T><<<blocks_for(ring_threads(S, g.n)), kBlock, 0, st>>>(g.n, S, g.K, bd, g.b));
        if (k == 0) vcycles(H, 0, 0, prm, nullptr, st, 1, false);
        if (!refined) {
            if (k > 0) vcycles(H, k, k, prm, nullptr, st, prm.nu0, false);
        } else {
            if (mixed && !(k == H.m && H.m >= 1 && refine_c))
                k_widen<T><<<blocks_for(cells), kBlock, 0, st>>>(cells, g.p, g.p64);
            FM_TRY(refine_stage(H, k, prm, mixed, status, st));
        }
        if (k == H.m - 1 && qc) {
            if (mixed && refined) outflux(ctx, g.n, S, g.K, g.p64, bd, qc, st);
            else outflux(ctx, g.n, S, g.K, g.p, bd, qc, st);
        }
    }
    const GridBufs<T>& f = H.g[H.m];
    const bool fine64 = mixed && conv;
    if (H.m == 0 && qc) k_fill<<<blocks_for(S), kBlock, 0, st>>>(S, std::nan(""), qc);
    if (fine64) outflux(ctx, f.n, S, f.K, f.p64, bd, qf, st);
    else outflux(ctx, f.n, S, f.K, f.p, bd, qf, st);
    if (p_out) {
        const size_t cells = S * (size_t)f.n * f.n;
        if (fine64)
            FM_CUDA_TRY(ctx, cudaMemcpyAsync(p_out, f.p64, sizeof(double) * cells, cudaMemcpyDeviceToDevice, st));
        else
            k_widen<T><<<blocks_for(cells), kBlock, 0, st>>>(cells, f.p, p_out);
    }
    return FM_OK;
}

template <typename T>
static fm_status levelwise(fm_ctx* ctx, Arena& ar, int n_fine, int n0, uint32_t S, const double* d_K,
                           const fm_solve_params& prm, double* d_qf, double* d_qc, double* d_p,
                           int32_t* d_status, cudaStream_t st) {
    const bool mixed = prm.precision == FM_PREC_MIXED;
    const int64_t lim = batch_limit(ctx, n_fine);
    for (uint64_t first = 0; first < S; first += (uint64_t)lim) {
        const size_t cnt = (size_t)std::min<uint64_t>((uint64_t)lim, S - first);
        const size_t off = first * (size_t)n_fine * n_fine;
        Hierarchy<T> H;
        FM_TRY(carve(ctx, ar, H, n_fine, n0, cnt, d_K + off, mixed, prm.converged != 0));
        FM_TRY(fmg_batch(H, prm, d_qf + first, d_qc ? d_qc + first : nullptr, d_p ? d_p + off : nullptr,
                         d_status ? d_status + first : nullptr, st));
        FM_CUDA_TRY(ctx, cudaGetLastError());
    }
    return FM_OK;
}

template <typename T>
static void append_shapes(const fm_ctx* ctx, int n_fine, size_t S, const fm_solve_params& prm,
                          std::vector<int64_t>* key) {
    for (int n = 2 * prm.n_coarsest; n <= n_fine; n *= 2) {
        int tile, threads;
        smooth_shape<T>(ctx, n, S, prm, &tile, &threads);
        key->push_back(tile);
        key->push_back(threads);
    }
}

void fmg_launch_key(const fm_ctx* ctx, int n_fine, uint32_t S, const fm_solve_params& prm,
                    std::vector<int64_t>* key) {
    const int64_t lim = batch_limit(ctx, n_fine), full = S / lim, rest = S % lim;
    key->push_back(full);
    for (int64_t cnt : {full ? lim : 0, rest}) {
        if (cnt == 0) key->push_back(-2);
        else if (prm.precision == FM_PREC_MIXED) append_shapes<float>(ctx, n_fine, (size_t)cnt, prm, key);
        else append_shapes<double>(ctx, n_fine, (size_t)cnt, prm, key);
    }
}

// Scratch bytes a level-wise solve of S samples of grid n_fine takes (one batch).
size_t fmg_levelwise_scratch(const fm_ctx* ctx, int n_fine, uint32_t S, const fm_solve_params& prm) {
    const bool mixed = prm.precision == FM_PREC_MIXED;
    const size_t cnt = (size_t)std::min<int64_t>(batch_limit(ctx, n_fine), S);
    return hierarchy_bytes(n_fine, prm.n_coarsest, cnt, mixed ? 4 : 8, mixed, prm.converged != 0);
}

fm_status fmg_solve_impl(fm_ctx* ctx, int n_fine, uint32_t S, const double* d_K,
                         const fm_solve_params& prm, double* d_qf, double* d_qc, double* d_p,
                         int32_t* d_status, cudaStream_t st) {
    return fmg_solve_with(ctx, ctx->arena, n_fine, S, d_K, prm, d_qf, d_qc, d_p, d_status, st);
}

fm_status fmg_solve_with(fm_ctx* ctx, Arena& ar, int n_fine, uint32_t S, const double* d_K,
                         const fm_solve_params& prm, double* d_qf, double* d_qc, double* d_p,
                         int32_t* d_status, cudaStream_t st) {
    const int n0 = prm.n_coarsest;
    FM_CHECK_ARG(ctx, n0 >= 2 && n0 <= 4, "fmg_solve_batch: n_coarsest must be 2..4");
    FM_CHECK_ARG(ctx, n_fine >= n0 && n_fine <= 8192, "fmg_solve_batch: bad n_fine");
    int m = 0;
    while ((n0 << m) < n_fine) ++m;
    FM_CHECK_ARG(ctx, (n0 << m) == n_fine, "fmg_solve_batch: n_fine must be n_coarsest * 2^m");
    FM_CHECK_ARG(ctx, prm.nu0 >= 1 && prm.nu1 >= 0 && prm.nu2 >= 0 && prm.nu1 + prm.nu2 >= 1,
                 "fmg_solve_batch: need nu0 >= 1 and nu1 + nu2 >= 1");
    FM_CHECK_ARG(ctx, prm.precision == FM_PREC_FP64 || prm.precision == FM_PREC_MIXED,
                 "fmg_solve_batch: unknown precision");
    FM_CHECK_ARG(ctx, prm.precision != FM_PREC_MIXED || prm.converged,
                 "fmg_solve_batch: the mixed form refines to a tolerance (converged = 1)");
    FM_CHECK_ARG(ctx, !prm.converged || (prm.tol > 0 && prm.max_cycles >= 1),
                 "fmg_solve_batch: converged mode needs tol > 0 and max_cycles >= 1");
    FM_CHECK_ARG(ctx, S == 0 || (d_K && d_qf), "fmg_solve_batch: null input or output");
    FM_CHECK_ARG(ctx, prm.kernel >= FM_KERNEL_AUTO && prm.kernel <= FM_KERNEL_RESIDENT,
                 "fmg_solve_batch: unknown kernel schedule");
    FM_CHECK_ARG(ctx, prm.ir_cycles >= 0 && prm.ir_cycles <= 64, "fmg_solve_batch: ir_cycles must be 0 .. 64");
    FM_CHECK_ARG(ctx, prm.bc_case == 0 || prm.bc_case == FM_CASE_I || prm.bc_case == FM_CASE_II,
                 "fmg_solve_batch: bc_case must be FM_CASE_I or FM_CASE_II");
    FM_CHECK_ARG(ctx, !prm.energy_step || (prm.converged && prm.kernel != FM_KERNEL_RESIDENT),
                 "fmg_solve_batch: the energy-optimal correction step runs in converged mode on the level-wise "
                 "schedule");
    if (S == 0) return FM_OK;
    bool resident = prm.kernel == FM_KERNEL_RESIDENT;
    if (prm.kernel == FM_KERNEL_AUTO) {
        resident = auto_resident(n_fine, S, ctx->sms, prm);
        // The resident kernel takes no scratch, so it runs what the level-wise schedule
        // would be faster at but finds no room for: none left, or a stream capture, in
        // which nothing can be allocated.  FP64 grids up to 16 x 16 take it in every
        // capture: their graphs keep no address of scratch that a later call may free.
        if (!resident && !prm.energy_step && fmg_resident_takes(n_fine, prm)) {
            const size_t need = fmg_levelwise_scratch(ctx, n_fine, S, prm);
            cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
            FM_CUDA_TRY(ctx, cudaStreamIsCapturing(st, &cs));
            if (cs != cudaStreamCaptureStatusNone) resident = n_fine <= 16 || ar.capacity < need;
            else resident = !arena_holds(ar, need);
        }
    }
    if (resident) {
        if (fmg_resident_launch(ctx, n_fine, n0, S, d_K, prm, d_qf, d_qc, d_p, d_status, st)) {
            FM_CUDA_TRY(ctx, cudaGetLastError());
            return FM_OK;
        }
        FM_CHECK_ARG(ctx, prm.kernel == FM_KERNEL_AUTO,
                     "fmg_solve_batch: the resident schedule needs the hierarchy in shared memory "
                     "(n_fine <= 64) and a power-of-two coarsest grid (2 or 4)");
    }
    // the context's own scratch serves calls on any stream, one after the other
    // (branches of an uneven batch have scratch of their own)
    const bool shared = &ar == &ctx->arena;
    if (shared) FM_CUDA_TRY(ctx, ctx->arena_order.begin(st));
    const fm_status rs = prm.precision == FM_PREC_MIXED
                             ? levelwise<float>(ctx, ar, n_fine, n0, S, d_K, prm, d_qf, d_qc, d_p, d_status, st)
                             : levelwise<double>(ctx, ar, n_fine, n0, S, d_K, prm, d_qf, d_qc, d_p, d_status, st);
    if (shared) FM_CUDA_TRY(ctx, ctx->arena_order.end(st));
    return rs;
}

// ------------------------------------------------------------------ allocation-free variant
// Scratch of fmg_solve_batch_static: one file-scope device array, present on
// every device that loads the library for as long as the process lives.
// What a batch may need, the reciprocal diagonals apart (at most a seventeenth
// of it), and the array with room for those.
constexpr size_t kStaticScratchBytes = (size_t)32 << 20;   // 32 MiB
static __device__ __align__(256) char g_static_scratch[kStaticScratchBytes + ((size_t)2 << 20)];

// Device address of the array on the current device.  Host code only sees a
// stand-in symbol, so the address is asked for once per device, with that
// device current, and kept.
static char* static_scratch_address(fm_ctx* ctx, fm_status* status) {
    static std::mutex mu;
    static char* addr[128] = {};
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 128) {
        set_error(ctx, "fmg_solve_batch_static: no current CUDA device");
        *status = FM_ECUDA;
        return nullptr;
    }
    std::lock_guard<std::mutex> lock(mu);
    if (!addr[dev]) {
        void* p = nullptr;
        const cudaError_t e = cudaGetSymbolAddress(&p, g_static_scratch);
        if (e != cudaSuccess || !p) {
            set_error(ctx, std::string("fmg_solve_batch_static: cudaGetSymbolAddress failed: ") +
                               cudaGetErrorString(e));
            *status = FM_ECUDA;
            return nullptr;
        }
        addr[dev] = static_cast<char*>(p);
    }
    *status = FM_OK;
    return addr[dev];
}

// The level-wise FP64 hierarchy of carve(), laid out in a caller-given buffer.
static void carve_into(fm_ctx* ctx, Hierarchy<double>& H, char* base, int n_fine, int n0, size_t S,
                       const double* d_K) {
    char* cur = base;
    auto take = [&](size_t bytes) {
        char* p = cur;
        cur += ((bytes + 255) / 256) * 256;
        return p;
    };
    H.ctx = ctx;
    H.n0 = n0;
    H.S = S;
    H.m = 0;
    while ((n0 << H.m) < n_fine) ++H.m;
    for (int k = 0; k <= H.m; ++k) {
        const int n = n0 << k;
        const size_t cnt = S * (size_t)n * n;
        GridBufs<double>& g = H.g[k];
        g.n = n;
        g.K = (k == H.m) ? d_K : (double*)take(cnt * 8);
        g.Te = (double*)take(cnt * 8);
        g.Tn = (double*)take(cnt * 8);
        g.D = (double*)take(cnt * 8);
        g.p = (double*)take(cnt * 8);
        g.b = (double*)take(cnt * 8);
        g.p2 = (double*)take(cnt * 8);
        g.Kc = nullptr;
        g.TeC = g.TnC = g.DC = nullptr;
        if (k < H.m) {
            g.Kc = (double*)take(cnt * 8);
            g.TeC = (double*)take(cnt * 8);
            g.TnC = (double*)take(cnt * 8);
            g.DC = (double*)take(cnt * 8);
        }
        g.rD = (double*)take(cnt * 8);
        g.rDC = k >= 1 ? g.Kc : nullptr;
        g.p64 = g.Te64 = g.Tn64 = g.D64 = nullptr;
    }
    H.Ainv = (double*)take(S * (size_t)n0 * n0 * n0 * n0 * 8);
    H.AinvC = (double*)take(S * (size_t)n0 * n0 * n0 * n0 * 8);
    H.active = nullptr;
    H.left = nullptr;
    H.iter = nullptr;
    H.qprev = nullptr;
    H.partial = nullptr;
    H.order = nullptr;
}

// ------------------------------------------------------------------ autotuning
// Synthetic smoothing problem for timing: faces in (0.5, 1.5), a diagonal
// that dominates them, rhs and iterate in (-1, 1) (a hash of the index).
template <typename T>
__global__ void k_tune_fill(size_t count, T* __restrict__ b, T* __restrict__ Te, T* __restrict__ Tn,
                            T* __restrict__ D, T* __restrict__ rD, T* __restrict__ p) {
    const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= count) return;
    uint64_t h = t * 0x9E3779B97F4A7C15ULL;
    h ^= h >> 31;
    h *= 0xBF58476D1CE4E5B9ULL;
    h ^= h >> 29;
    const double u0 = (double)(h & 0xFFFFF) / 1048576.0, u1 = (double)((h >> 20) & 0xFFFFF) / 1048576.0;
    const double u2 = (double)((h >> 40) & 0xFFFFF) / 1048576.0;
    Te[t] = (T)(0.5 + u0);
    Tn[t] = (T)(0.5 + u1);
    D[t] = (T)(4.5 + u2);
    rD[t] = recip_set(D[t]);
    b[t] = (T)(2.0 * u2 - 1.0);
    p[t] = (T)(2.0 * u0 - 1.0);
}

template <typename T>
static fm_status autotune_grid(fm_ctx* ctx, int n, int nsweeps, fm_tune_entry* e) {
    // about 64 Mi cells per call (well beyond L2), at least one sample
    const size_t S = std::max<size_t>(1, ((size_t)64 << 20) / ((size_t)n * n));
    const size_t cells = S * (size_t)n * n;
    T* buf = nullptr;
    FM_CUDA_TRY(ctx, cudaMalloc((void**)&buf, 7 * cells * sizeof(T)));
    T *b = buf, *Te = b + cells, *Tn = Te + cells, *D = Tn + cells, *p = D + cells, *p2 = p + cells, *rD = p2 + cells;
    k_tune_fill<T><<<blocks_for(cells), kBlock>>>(cells, b, Te, Tn, D, rD, p);
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    const bool prof = ctx->prof.active;
    ctx->prof.active = false;
    auto time_shape = [&](int tile, int threads) -> double {
        if (tile > 0 && tile_smem_bytes(tile, n, nsweeps, sizeof(T)) > kMaxSmem) return 1e30;
        auto smooth = [&](T* in, T* out) {
            if (tile != kShapeStrip) {
                smooth_with<T>(ctx, tile, threads, n, S, nsweeps, b, Te, Tn, D, sizeof(T) == 8 ? rD : nullptr, in, out,
                               nullptr, nullptr);
                return;
            }
            StripCall<T> c;
            c.n = n;
            c.S = S;
            c.hs = 2 * nsweeps;
            c.b = b;
            c.Te = Te;
            c.Tn = Tn;
            c.D = D;
            c.rD = rD;
            c.p_in = in;
            c.p_out = out;
            strip_launch(ctx, c, nullptr);
        };
        smooth(p, p2);   // warm-up
        cudaEventRecord(e0);
        for (int r = 0; r < 4; ++r) smooth(r & 1 ? p2 : p, r & 1 ? p : p2);   // p -> p2 -> p for tiles and strips
        cudaEventRecord(e1);
        cudaEventSynchronize(e1);
        float ms = 0.0f;
        cudaEventElapsedTime(&ms, e0, e1);
        return ms / 4.0;
    };
    fm_solve_params dp{};
    dp.nu1 = dp.nu2 = nsweeps;
    int def_tile = 0, def_threads = 0;
    const int pi = sizeof(T) == 4 ? 1 : 0, slot = tune_slot(n);
    ctx->tune.n[pi][slot] = 0;   // the untuned default
    smooth_shape<T>(ctx, n, S, dp, &def_tile, &def_threads);
    double best = 1e30;
    int bt = def_tile, bth = def_threads;
    e->ms_default = time_shape(def_tile, def_threads);
    const int tiles[] = {0, kShapeStrip, 8, 16, 32, 64};
    const int thr[] = {0, 128, 256};   // 0: register-blocked regions (fixed thread count)
    for (int tile : tiles) {
        if (tile > 0 && tile > n && tile != 8) continue;   // one whole-grid candidate is enough
        if (tile == kShapeStrip && !strip_fits(n, nsweeps, nsweeps)) continue;
        for (int th : thr) {
            if (tile <= 0 && th != 0) continue;               // colour launches and strips have a fixed shape
            const double ms = time_shape(tile, th);
            if (ms < best) {
                best = ms;
                bt = tile;
                bth = th;
            }
        }
    }
    if (e->ms_default <= best) {   // the default, timed first, stays unless beaten
        best = e->ms_default;
        bt = def_tile;
        bth = def_threads;
    }
    ctx->prof.active = prof;
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    cudaFree(buf);
    FM_CUDA_TRY(ctx, cudaGetLastError());
    ctx->tune.n[pi][slot] = n;
    ctx->tune.tile[pi][slot] = bt;
    ctx->tune.threads[pi][slot] = bth;
    ctx->tune.by_hand[pi][slot] = false;
    e->n = n;
    e->tile = bt;
    e->threads = bth;
    e->ms_best = best;
    e->samples = (int64_t)S;
    return FM_OK;
}

}  // namespace fm

using namespace fm;

extern "C" fm_status fm_autotune(fm_ctx* ctx, int32_t precision, int32_t nsweeps, int32_t n_min, int32_t n_max,
                                 fm_tune_entry* entries, int32_t max_entries, int32_t* n_entries) {
    FM_CHECK_ARG(ctx, ctx != nullptr, "fm_autotune: null context");
    FM_CHECK_ARG(ctx, precision == FM_PREC_FP64 || precision == FM_PREC_MIXED, "fm_autotune: unknown precision");
    FM_CHECK_ARG(ctx, nsweeps >= 1 && nsweeps <= 8, "fm_autotune: nsweeps must be 1..8");
    FM_CHECK_ARG(ctx, n_min >= 2 && n_max >= n_min && n_max <= 8192, "fm_autotune: bad grid range");
    int count = 0;
    for (int n = n_min; n <= n_max; n *= 2) {
        fm_tune_entry e{};
        if (precision == FM_PREC_MIXED) FM_TRY(autotune_grid<float>(ctx, n, nsweeps, &e));
        else FM_TRY(autotune_grid<double>(ctx, n, nsweeps, &e));
        if (entries && count < max_entries) entries[count] = e;
        ++count;
    }
    if (n_entries) *n_entries = std::min(count, max_entries);
    return FM_OK;
}

extern "C" fm_status fm_set_vcycle_tail(fm_ctx* ctx, int32_t n_max) {
    FM_CHECK_ARG(ctx, ctx != nullptr, "fm_set_vcycle_tail: null context");
    FM_CHECK_ARG(ctx, n_max == 0 || (n_max >= 2 && n_max <= kTailMaxN && (n_max & (n_max - 1)) == 0),
                 "fm_set_vcycle_tail: n_max must be 0 or a power of two up to 32");
    ctx->tail_max = n_max;
    return FM_OK;
}

extern "C" fm_status fm_set_smoother_shape(fm_ctx* ctx, int32_t precision, int32_t n, int32_t tile,
                                          int32_t threads) {
    FM_CHECK_ARG(ctx, ctx != nullptr, "fm_set_smoother_shape: null context");
    FM_CHECK_ARG(ctx, precision == FM_PREC_FP64 || precision == FM_PREC_MIXED,
                 "fm_set_smoother_shape: unknown precision");
    FM_CHECK_ARG(ctx, n >= 2 && n <= 8192 && (n & (n - 1)) == 0, "fm_set_smoother_shape: n must be a power of two");
    const bool tile_ok = tile == 8 || tile == 16 || tile == 32 || tile == 64;
    FM_CHECK_ARG(ctx, tile == -2 || tile == 0 || tile == kShapeStrip || tile_ok,
                 "fm_set_smoother_shape: tile must be -2, -1, 0, 8, 16, 32 or 64");
    FM_CHECK_ARG(ctx, (tile_ok && (threads == 0 || threads == 128 || threads == 256)) || (!tile_ok && threads == 0),
                 "fm_set_smoother_shape: threads must be 0 (or 128, 256 for tiles)");
    const int pi = precision == FM_PREC_MIXED ? 1 : 0, slot = tune_slot(n);
    if (tile == -2) {
        if (ctx->tune.n[pi][slot] == n) ctx->tune.n[pi][slot] = 0;
        return FM_OK;
    }
    ctx->tune.n[pi][slot] = n;
    ctx->tune.tile[pi][slot] = tile;
    ctx->tune.threads[pi][slot] = threads;
    ctx->tune.by_hand[pi][slot] = true;
    return FM_OK;
}

extern "C" fm_status fmg_solve_batch_static(fm_ctx* ctx, int32_t n_fine, uint32_t n, const double* d_K,
                                            const fm_solve_params* prm, double* d_qf, double* d_qc,
                                            void* stream) {
    FM_CHECK_ARG(ctx, ctx != nullptr, "fmg_solve_batch_static: null context");
    FM_CHECK_ARG(ctx, prm != nullptr, "fmg_solve_batch_static: null parameters");
    const int n0 = prm->n_coarsest;
    FM_CHECK_ARG(ctx, n0 >= 2 && n0 <= 4, "fmg_solve_batch_static: n_coarsest must be 2..4");
    FM_CHECK_ARG(ctx, n_fine >= n0 && n_fine <= 8192, "fmg_solve_batch_static: bad n_fine");
    int m = 0;
    while ((n0 << m) < n_fine) ++m;
    FM_CHECK_ARG(ctx, (n0 << m) == n_fine, "fmg_solve_batch_static: n_fine must be n_coarsest * 2^m");
    FM_CHECK_ARG(ctx, prm->nu0 >= 1 && prm->nu1 >= 0 && prm->nu2 >= 0 && prm->nu1 + prm->nu2 >= 1,
                 "fmg_solve_batch_static: need nu0 >= 1 and nu1 + nu2 >= 1");
    FM_CHECK_ARG(ctx, prm->precision == FM_PREC_FP64 && !prm->converged,
                 "fmg_solve_batch_static: only the FP64 fixed-cycle schedule (converged = 0)");
    // the energy step keeps per-sample dot products and step lengths that the
    // static hierarchy has no room for
    FM_CHECK_ARG(ctx, !prm->energy_step, "fmg_solve_batch_static: the energy-optimal step is not available here");
    FM_CHECK_ARG(ctx, prm->bc_case == 0 || prm->bc_case == FM_CASE_I || prm->bc_case == FM_CASE_II,
                 "fmg_solve_batch_static: bc_case must be FM_CASE_I or FM_CASE_II");
    FM_CHECK_ARG(ctx, n == 0 || (d_K && d_qf), "fmg_solve_batch_static: null input or output");
    if (n == 0) return FM_OK;
    const size_t need = hierarchy_bytes(n_fine, n0, n, 8, false, false) - n * rdiag_bytes(n_fine, n0);
    FM_CHECK_ARG(ctx, need <= kStaticScratchBytes,
                 "fmg_solve_batch_static: " + std::to_string(n) + " samples of " + std::to_string(n_fine) + "x" +
                     std::to_string(n_fine) + " need " + std::to_string(need) + " bytes of scratch; the static "
                     "scratch holds " + std::to_string(kStaticScratchBytes) + " bytes: split the batch");
    fm_status st = FM_OK;
    char* base = static_scratch_address(ctx, &st);
    if (!base) return st;
    Hierarchy<double> H;
    carve_into(ctx, H, base, n_fine, n0, n, d_K);
    // per-launch profiling creates events and counters: off for this call
    const bool prof = ctx->prof.active;
    ctx->prof.active = false;
    const fm_status rs = fmg_batch(H, *prm, d_qf, d_qc, nullptr, nullptr, as_stream(stream));
    ctx->prof.active = prof;
    FM_TRY(rs);
    FM_CUDA_TRY(ctx, cudaGetLastError());
    return FM_OK;
}

extern "C" fm_status fmg_solve_batch(fm_ctx* ctx, int32_t n_fine, uint32_t n, const double* d_K,
                                     const fm_solve_params* prm, double* d_qf, double* d_qc,
                                     double* d_p, int32_t* d_status, void* stream) {
    FM_CHECK_ARG(ctx, ctx != nullptr, "fmg_solve_batch: null context");
    FM_CHECK_ARG(ctx, prm != nullptr, "fmg_solve_batch: null parameters");
    return fmg_solve_impl(ctx, n_fine, n, d_K, *prm, d_qf, d_qc, d_p, d_status, as_stream(stream));
}
