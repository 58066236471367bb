// Multigrid-preconditioned conjugate gradients on the 7-point operators of
// the Gummel loop (included by gummel.cu only).
//
// Per grid level: face coefficients cx[p] (face to the +x neighbour,
// wrapping; zero across a no-flux wall), cy[p], cz[p] (face to +z; on the top
// plane the face to the upper Dirichlet plane) and czlo[p] (face to the lower
// Dirichlet plane, plane 0 only), an optional extra diagonal dg (screening),
// and the assembled diagonal dgn with its reciprocal idg:
//   (A u)_p = dgn_p u_p - sum_faces c u_nbr,  Dirichlet neighbours moved to b.
//
// What bounds these kernels.  GB300 has two FP64 lanes per SM and clock: any
// FP64 warp instruction holds its quarter of the SM for 64 clocks, dependent
// or not, however few lanes are active, and a division takes about 560; and
// the V-cycle is a chain of dependent phases, most of them too small to fill
// the chip.  So the diagonal is assembled once per operator and a sweep divides
// by it with three operations (quotient), every lane owns a point of the swept
// colour, index arithmetic is 32-bit multiply-shift, the first red sweep rides
// in the kernel that produces the right-hand side, dot products ride in the
// kernels that produce their operands and are finished by their consumers, and
// the small levels run inside one CTA (k_tail).
//
// The order of the floating-point operations is fixed: a sum of products here
// is one particular chain of fused multiply-adds, a dot product one particular
// tree.  The linear solves stop at a tolerance, and where a box has deep wells
// or hard walls a change of one rounding in one sweep moves the stopped iterate
// by up to 1e-6 relative (measured on the 48^3 served request), so a
// rearrangement of these sums is not a neutral change.
#pragma once

#include "pnp_internal.h"

namespace pnp {

// n / d for 0 <= n < 2^31: one 64-bit multiply and a shift
struct FastDiv {
    unsigned d = 1, m = 0x80000000u;
    int s = 31;
    __host__ __device__ FastDiv() {}
    explicit FastDiv(unsigned dd) : d(dd) {
        int l = 0;
        while ((1ull << l) < dd) ++l;
        s = 31 + l;
        m = (unsigned)(((1ull << s) + dd - 1) / dd);
    }
    __device__ __forceinline__ unsigned div(unsigned n) const {
        return (unsigned)(((unsigned long long)n * m) >> s);
    }
};

struct Level {
    int nx, ny, nz;
    size_t n;
    int fx, fy, fz;                // aggregation factors to the next level
    bool odd;                      // x or y wraps with odd extent: points of one colour can be neighbours
    double *cx, *cy, *cz, *czlo;   // operator being solved (Poisson or NP); czlo holds plane 0
    double *pcx, *pcy, *pcz, *pczlo;   // Poisson copy (built once)
    double *dg;                    // diagonal term of the screened Poisson operator
    double *dgn, *idg;             // assembled diagonal and reciprocal of the current operator
    double *x, *b;
    double *x2;                    // second iterate buffer of odd levels (x otherwise)
    bool punit;                    // every face of the Poisson operator is 1 (level 0, x and y periodic)
    bool unit;                     // and of the current operator
};

// what the level kernels read, by value
struct Op {
    int nx, ny, nz, hx;            // hx: points of one colour per row, at most
    unsigned plane, n, nt;         // nx ny, nx ny nz, hx ny nz
    FastDiv dnx, dny, dhx;
    const double *cx, *cy, *cz, *czlo;
    const double *dg;              // optional extra diagonal (Poisson-Boltzmann screening)
    const double *dgn, *idg;
    int odd;
    int unit;                      // every face is 1: kernels compiled for it do not read them
};

constexpr int kCoarseSweeps = 40;
constexpr double kCoarseScale = 1.8;
// blocks of 256 slots of the dot products, at most
constexpr int kDotBlocks = 512;
constexpr int kSweepThreads = 128;

// record of a linear solve in progress
struct LinCtl {
    double rz[2];                  // r . z of this and the previous iteration, by parity
    double tgt;                    // ||r||^2 to reach
    int it;                        // iterations done
};

static Op op_of(const Level &L, bool shift = false) {
    Op A{};
    A.nx = L.nx; A.ny = L.ny; A.nz = L.nz;
    A.hx = (L.nx + 1) / 2;
    A.plane = (unsigned)L.nx * L.ny;
    A.n = A.plane * (unsigned)L.nz;
    A.nt = (unsigned)A.hx * L.ny * L.nz;
    A.dnx = FastDiv(L.nx);
    A.dny = FastDiv(L.ny);
    A.dhx = FastDiv(A.hx);
    A.cx = L.cx; A.cy = L.cy; A.cz = L.cz; A.czlo = L.czlo;
    A.dg = shift ? L.dg : nullptr;
    A.dgn = L.dgn; A.idg = L.idg;
    A.odd = L.odd ? 1 : 0;
    A.unit = L.unit ? 1 : 0;
    return A;
}

struct Pt {
    int i, j, k;
    unsigned p;
};

// point of the flat index p
__device__ __forceinline__ Pt pt_flat(const Op &A, unsigned p) {
    const unsigned row = A.dnx.div(p), k = A.dny.div(row);
    return Pt{(int)(p - row * A.nx), (int)(row - k * A.ny), (int)k, p};
}

// point of colour c ((i + j + k) % 2 == c) with index t < nt; i may reach nx
// (no point) where nx is odd
__device__ __forceinline__ Pt pt_colour(const Op &A, unsigned t, int c) {
    const unsigned row = A.dhx.div(t), h = t - row * A.hx, k = A.dny.div(row), j = row - k * A.ny;
    const int i = (int)(2 * h + ((j + k + c) & 1));
    return Pt{i, (int)j, (int)k, row * A.nx + i};
}

__device__ __forceinline__ unsigned nbr_xp(const Op &A, const Pt &q) { return q.i + 1 == A.nx ? q.p + 1 - A.nx : q.p + 1; }
__device__ __forceinline__ unsigned nbr_xm(const Op &A, const Pt &q) { return q.i == 0 ? q.p + A.nx - 1 : q.p - 1; }
__device__ __forceinline__ unsigned nbr_yp(const Op &A, const Pt &q) {
    return q.j + 1 == A.ny ? q.p + A.nx - A.plane : q.p + A.nx;
}
__device__ __forceinline__ unsigned nbr_ym(const Op &A, const Pt &q) {
    return q.j == 0 ? q.p + A.plane - A.nx : q.p - A.nx;
}

// diagonal from the faces
__device__ __forceinline__ double op_diag(const Op &A, const Pt &q) {
    double d = A.cx[q.p] + A.cy[q.p] + A.cz[q.p];
    d += A.cx[nbr_xm(A, q)] + A.cy[nbr_ym(A, q)];
    d += q.k > 0 ? A.cz[q.p - A.plane] : A.czlo[q.p];
    if (A.dg) d += A.dg[q.p];
    return d;
}

// sum_faces c u_nbr; UNIT: every c is 1, where the same sums are plain additions
// (fma(1, a, 1 b) = a + b): six operations instead of eight and no faces to read.
// `wrap` serves the neighbours across an x or y wrap of
// odd extent (they have the point's own colour), u all others.
template <bool UNIT = false>
__device__ __forceinline__ double op_nbr(const Op &A, const double *u, const double *wrap, const Pt &q) {
    const unsigned xp = nbr_xp(A, q), xm = nbr_xm(A, q), yp = nbr_yp(A, q), ym = nbr_ym(A, q);
    const bool ox = A.odd && (A.nx & 1), oy = A.odd && (A.ny & 1);
    const double *uxp = ox && q.i + 1 == A.nx ? wrap : u, *uxm = ox && q.i == 0 ? wrap : u;
    const double *uyp = oy && q.j + 1 == A.ny ? wrap : u, *uym = oy && q.j == 0 ? wrap : u;
    if constexpr (UNIT) {
        double s = (uxp[xp] + uxm[xm]) + (uyp[yp] + uym[ym]);
        if (q.k + 1 < A.nz) s += u[q.p + A.plane];
        if (q.k > 0) s += u[q.p - A.plane];
        return s;
    }
    const double sx = fma(A.cx[q.p], uxp[xp], A.cx[xm] * uxm[xm]);
    const double sy = fma(A.cy[q.p], uyp[yp], A.cy[ym] * uym[ym]);
    double s = sx + sy;
    if (q.k + 1 < A.nz) s = fma(A.cz[q.p], u[q.p + A.plane], s);
    if (q.k > 0) s = fma(A.cz[q.p - A.plane], u[q.p - A.plane], s);
    return s;
}

// v / d from the stored reciprocal y = RN(1 / d): RN(v y) corrected once by its
// exact remainder (Markstein's division step), three operations against about
// nine for a division.  The result is the IEEE quotient unless v / d lies
// within 2^-105 of a rounding boundary.
__device__ __forceinline__ double quotient(double v, double d, double y) {
    const double q = v * y;
    return fma(fma(-d, q, v), y, q);
}

// b - (A u)_p
template <bool UNIT = false>
__device__ __forceinline__ double op_residual(const Op &A, const double *u, const Pt &q, double b) {
    return b - (__dmul_rn(A.dgn[q.p], u[q.p]) - op_nbr<UNIT>(A, u, u, q));
}

// ---------------------------------------------------------------------------
// fixed-shape reductions

// Dot products: element p belongs to slot p % (256 nb) of nb blocks of 256
// slots, a slot sums its elements in order, and a block's slots and then the
// blocks' sums (padded to 512) are summed as binary trees (slot t + slot
// t + w, w = 128 ... 1).  The tree below w = 32 is a warp's butterfly.

// sum of the 32 values a warp holds, as the tree's last five steps
__device__ __forceinline__ double warp_tree(double v) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

// tree over 128 values v of threads 0..127 (every thread of the block calls;
// valid in thread 0)
__device__ __forceinline__ double tree128(double v) {
    __shared__ double sh[128];
    if (threadIdx.x < 128) sh[threadIdx.x] = v;
    __syncthreads();
    if (threadIdx.x < 32) {
        const int t = threadIdx.x;
        v = warp_tree((sh[t] + sh[t + 64]) + (sh[t + 32] + sh[t + 96]));
    }
    __syncthreads();
    return v;
}

// sum over the 256 slots of a block of 256 threads; valid in thread 0
__device__ __forceinline__ double block_tree(double v) {
    __shared__ double up[128];
    if (threadIdx.x >= 128) up[threadIdx.x - 128] = v;
    __syncthreads();
    return tree128(threadIdx.x < 128 ? v + up[threadIdx.x] : 0.0);
}

// sum of nb <= 512 block sums; valid in thread 0 (blocks of at least 128 threads)
__device__ __forceinline__ double partials_tree(const double *__restrict__ part, int nb) {
    const int t = threadIdx.x;
    double v = 0.0;
    if (t < 128) {
        v = t < nb ? part[t] : 0.0;
        if (nb > 128) {
            double w = t + 128 < nb ? part[t + 128] : 0.0;
            if (nb > 256) {
                v += t + 256 < nb ? part[t + 256] : 0.0;
                w += t + 384 < nb ? part[t + 384] : 0.0;
            }
            v += w;
        }
    }
    return tree128(v);
}

// f(sum of the partials), evaluated by one thread and returned to the block
// (a division in every warp would take longer than the loop that follows)
template <typename F>
__device__ __forceinline__ double of_partials(const double *__restrict__ part, int nb, F f) {
    __shared__ double tot;
    const double v = partials_tree(part, nb);
    if (threadIdx.x == 0) tot = f(v);
    __syncthreads();
    return tot;
}

// ---------------------------------------------------------------------------
// operator set-up

// coarse face coefficients: sums of the fine faces leaving each aggregate;
// the extra diagonal is summed over the aggregate
__device__ __forceinline__ void coarsen_cell(const Op &F, int fx, int fy, int fz, const Op &C, unsigned q,
                                             double *__restrict__ cx, double *__restrict__ cy,
                                             double *__restrict__ cz, double *__restrict__ czlo) {
    const Pt Q = pt_flat(C, q);
    double sx = 0, sy = 0, sz = 0, sl = 0;
    for (int c = 0; c < fz; ++c)
        for (int b = 0; b < fy; ++b) {
            const int j = Q.j * fy + b, k = Q.k * fz + c;
            const unsigned row = ((unsigned)k * F.ny + j) * F.nx + Q.i * fx;
            sx += F.cx[row + fx - 1];
            if (b == fy - 1)
                for (int a = 0; a < fx; ++a) sy += F.cy[row + a];
            if (c == fz - 1)
                for (int a = 0; a < fx; ++a) sz += F.cz[row + a];
            if (c == 0 && Q.k == 0)
                for (int a = 0; a < fx; ++a) sl += F.czlo[row + a];
        }
    cx[q] = sx;
    cy[q] = sy;
    cz[q] = sz;
    if (Q.k == 0) czlo[q] = sl;
}

__global__ void k_coarsen(Op F, int fx, int fy, int fz, Op C, double *__restrict__ cx, double *__restrict__ cy,
                          double *__restrict__ cz, double *__restrict__ czlo) {
    const unsigned q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q < C.n) coarsen_cell(F, fx, fy, fz, C, q, cx, cy, cz, czlo);
}

// sum of a fine field over the aggregate of coarse cell Q
__device__ __forceinline__ double aggregate_sum(const Op &F, const double *__restrict__ f, int fx, int fy, int fz,
                                                const Pt &Q) {
    double s = 0;
    for (int c = 0; c < fz; ++c)
        for (int b = 0; b < fy; ++b) {
            const unsigned row = ((unsigned)(Q.k * fz + c) * F.ny + Q.j * fy + b) * F.nx + Q.i * fx;
            for (int a = 0; a < fx; ++a) s += f[row + a];
        }
    return s;
}

__global__ void k_restrict(Op F, const double *__restrict__ f, int fx, int fy, int fz, Op C, double *__restrict__ fc) {
    const unsigned q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q < C.n) fc[q] = aggregate_sum(F, f, fx, fy, fz, pt_flat(C, q));
}

__global__ void k_diag(Op A, double *__restrict__ dgn, double *__restrict__ idg) {
    const unsigned p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= A.n) return;
    const double d = op_diag(A, pt_flat(A, p));
    dgn[p] = d;
    idg[p] = 1.0 / d;
}

// ---------------------------------------------------------------------------
// one level of the V-cycle, chip-wide kernels (levels above the tail)

// one colour of a red-black sweep: x_p = (b_p + sum c x_nbr) / diag_p for the
// points of colour c, one point a thread.  xo holds the other colour, xs the
// own colour before the sweep (read across odd wraps only), xw takes the
// result; all three are one array on even levels.
//
// 11 FP64 operations a point instead of 24 on half-idle warps: a 96^3 colour is
// FP64-bound, and 128-thread CTAs put the 512 warps of a 32^3 colour on 128 SMs,
// one warp on each quarter of an SM.  A 96^3 colour takes 10.7 us with its
// operands in L2 (its operations alone: 9.2 at the measured FP64 rate) and 14.7 from
// HBM.  With the rest of this file a CG iteration went from 343 to 103 us at 32^3
// and from 700 to 290 us at 96^3.
//
// RES: the residual of the swept points is written too.  Their neighbours do not
// change before the restriction, so the sum just formed serves it: three more
// operations here against ten there.
template <bool UNIT, bool RES>
__global__ void __launch_bounds__(kSweepThreads) k_sweep(Op A, const double *xo, const double *xs, double *xw,
                                                         const double *__restrict__ b, int c,
                                                         double *__restrict__ res) {
    const unsigned t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= A.nt) return;
    const Pt q = pt_colour(A, t, c);
    if (q.i >= A.nx) return;
    const double s = op_nbr<UNIT>(A, xo, xs, q), bp = b[q.p], d = A.dgn[q.p];
    const double v = quotient(bp + s, d, A.idg[q.p]);
    xw[q.p] = v;
    if (RES) res[q.p] = bp - (__dmul_rn(d, v) - s);
}

// the last red sweep of the cycle on level 0 with the block sums of b . x, for
// even nx and at most 512 x 256 points: thread m owns the pair of slots
// (2m, 2m + 1), one red point and one black
template <bool UNIT>
__global__ void __launch_bounds__(128) k_sweep_dot(Op A, const double *xo, const double *xs, double *xw,
                                                   const double *__restrict__ b, double *__restrict__ part) {
    __shared__ double sh[256];
    const unsigned p0 = blockIdx.x * 256u + 2 * threadIdx.x;
    double d0 = 0.0, d1 = 0.0;
    if (p0 < A.n) {
        Pt q = pt_flat(A, p0);
        const int up = (q.j + q.k) & 1;               // the red point's place in the pair
        q.i += up;
        q.p += up;
        const double br = b[q.p];
        const double v = quotient(br + op_nbr<UNIT>(A, xo, xs, q), A.dgn[q.p], A.idg[q.p]);
        const double dr = br * v;
        const unsigned pb = p0 + 1 - up;
        const double db = b[pb] * xo[pb];
        xw[q.p] = v;
        d0 = up ? db : dr;
        d1 = up ? dr : db;
    }
    sh[2 * threadIdx.x] = d0;
    sh[2 * threadIdx.x + 1] = d1;
    __syncthreads();
    const double s = tree128(sh[threadIdx.x] + sh[threadIdx.x + 128]);
    if (threadIdx.x == 0) part[blockIdx.x] = s;
}

// coarse right-hand side = sum of the fine residuals b - A x over each
// aggregate, and the coarse level's start values: b / diag at red points (the
// first red sweep from zero), zero at black ones.  kRestrictCells aggregates a
// CTA: one thread per fine point, then one per aggregate sums them in order.
constexpr int kRestrictCells = 32;
__global__ void __launch_bounds__(256) k_residual_restrict(Op F, const double *__restrict__ x,
                                                           const double *__restrict__ b, int fx, int fy, int fz,
                                                           Op C, double *__restrict__ bc, double *__restrict__ xred,
                                                           double *__restrict__ xblack) {
    extern __shared__ double res[];                   // [child][cell], child = (c fy + b) fx + a
    const int nch = fx * fy * fz, per_row = kRestrictCells * fx;
    for (int e = threadIdx.x; e < nch * kRestrictCells; e += blockDim.x) {
        const int row = e / per_row, w = e - row * per_row, cell = w / fx, a = w - cell * fx;
        const unsigned q = blockIdx.x * kRestrictCells + cell;
        if (q >= C.n) continue;
        const Pt Q = pt_flat(C, q);
        Pt f{Q.i * fx + a, Q.j * fy + row % fy, Q.k * fz + row / fy, 0};
        f.p = ((unsigned)f.k * F.ny + f.j) * F.nx + f.i;
        res[(row * fx + a) * kRestrictCells + cell] = op_residual(F, x, f, b[f.p]);
    }
    __syncthreads();
    const unsigned q = blockIdx.x * kRestrictCells + threadIdx.x;
    if (threadIdx.x >= kRestrictCells || q >= C.n) return;
    double s = res[threadIdx.x];
    for (int k = 1; k < nch; ++k) s += res[k * kRestrictCells + threadIdx.x];
    const Pt Q = pt_flat(C, q);
    bc[q] = s;
    if ((Q.i + Q.j + Q.k) & 1) xblack[q] = 0.0;
    else xred[q] = quotient(s, C.dgn[q], C.idg[q]);
}

// The same on an even level with fx = 2 whose black residuals k_sweep left in
// `known`: of each pair of children along x the red one is computed, on full
// warps, and the black one read.
template <bool UNIT>
__global__ void __launch_bounds__(128) k_residual_restrict_red(Op F, const double *__restrict__ x,
                                                               const double *__restrict__ b,
                                                               const double *__restrict__ known, int fy, int fz, Op C,
                                                               double *__restrict__ bc, double *__restrict__ xred,
                                                               double *__restrict__ xblack) {
    extern __shared__ double res[];                   // [child][cell], child = 2 (c fy + b) + a
    const int rows = fy * fz;
    for (int e = threadIdx.x; e < rows * kRestrictCells; e += blockDim.x) {
        const int row = e / kRestrictCells, cell = e % kRestrictCells;
        const unsigned q = blockIdx.x * kRestrictCells + cell;
        if (q >= C.n) continue;
        const Pt Q = pt_flat(C, q);
        const int j = Q.j * fy + row % fy, k = Q.k * fz + row / fy, a = (j + k) & 1;
        Pt f{2 * Q.i + a, j, k, ((unsigned)k * F.ny + j) * F.nx + 2 * Q.i + a};
        res[(2 * row + a) * kRestrictCells + cell] = op_residual<UNIT>(F, x, f, b[f.p]);
        res[(2 * row + 1 - a) * kRestrictCells + cell] = known[f.p + 1 - 2 * a];
    }
    __syncthreads();
    const unsigned q = blockIdx.x * kRestrictCells + threadIdx.x;
    if (threadIdx.x >= kRestrictCells || q >= C.n) return;
    double s = res[threadIdx.x];
    for (int k = 1; k < 2 * rows; ++k) s += res[k * kRestrictCells + threadIdx.x];
    const Pt Q = pt_flat(C, q);
    bc[q] = s;
    if ((Q.i + Q.j + Q.k) & 1) xblack[q] = 0.0;
    else xred[q] = quotient(s, C.dgn[q], C.idg[q]);
}

// x += scale * x_coarse (piecewise constant) at the red points (the black
// sweep that follows overwrites the black ones), everywhere on odd levels;
// scale > 1 compensates the weak correction of piecewise-constant interpolation
__global__ void __launch_bounds__(kSweepThreads) k_prolong_add(Op A, double *__restrict__ x, FastDiv fx, FastDiv fy,
                                                               FastDiv fz, int cnx, int cny,
                                                               const double *__restrict__ xc, double scale) {
    const unsigned t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= A.nt) return;
    for (int c = 0; c <= A.odd; ++c) {
        const Pt q = pt_colour(A, t, c);
        if (q.i >= A.nx) continue;
        const unsigned P = (fz.div(q.k) * cny + fy.div(q.j)) * cnx + fx.div(q.i);
        x[q.p] = fma(scale, xc[P], x[q.p]);
    }
}

// ---------------------------------------------------------------------------
// coarsest level by sweeps (more than kCoarseWarp points: extents that do not
// coarsen): x = 0, then kCoarseSweeps symmetric (red, black, black, red)
// sweeps in one CTA; in shared memory up to kCoarseMax points
constexpr int kCoarseMax = 1024;
__global__ void k_coarse_solve(Op A, double *__restrict__ x, const double *__restrict__ b) {
    for (unsigned p = threadIdx.x; p < A.n; p += blockDim.x) x[p] = 0.0;
    __syncthreads();
    for (int s = 0; s < kCoarseSweeps; ++s) {
        const int order[4] = {0, 1, 1, 0};
        for (int c = 0; c < 4; ++c) {
            for (unsigned t = threadIdx.x; t < A.nt; t += blockDim.x) {
                const Pt q = pt_colour(A, t, order[c]);
                if (q.i < A.nx) x[q.p] = quotient(b[q.p] + op_nbr(A, x, x, q), A.dgn[q.p], A.idg[q.p]);
            }
            __syncthreads();
        }
    }
}

__global__ void k_coarse_smem(Op A, double *__restrict__ x_out, const double *__restrict__ b_in) {
    extern __shared__ double csm[];
    const unsigned n = A.n;
    double *x = csm, *b = csm + n, *id = csm + 2 * n, *cx = csm + 3 * n, *cy = csm + 4 * n, *cz = csm + 5 * n,
           *dn = csm + 6 * n;
    for (unsigned p = threadIdx.x; p < n; p += blockDim.x) {
        x[p] = 0.0;
        b[p] = b_in[p];
        id[p] = A.idg[p];
        dn[p] = A.dgn[p];
        cx[p] = A.cx[p];
        cy[p] = A.cy[p];
        cz[p] = A.cz[p];
    }
    __syncthreads();
    Op S = A;
    S.cx = cx;
    S.cy = cy;
    S.cz = cz;
    const int order[4] = {0, 1, 1, 0};
    for (int s = 0; s < kCoarseSweeps; ++s)
        for (int c = 0; c < 4; ++c) {
            for (unsigned t = threadIdx.x; t < A.nt; t += blockDim.x) {
                const Pt q = pt_colour(A, t, order[c]);
                if (q.i < A.nx) x[q.p] = quotient(b[q.p] + op_nbr(S, x, x, q), dn[q.p], id[q.p]);
            }
            __syncthreads();
        }
    for (unsigned p = threadIdx.x; p < n; p += blockDim.x) x_out[p] = x[p];
}

// block sums of a . b
__global__ void __launch_bounds__(256) k_dot(const double *__restrict__ a, const double *__restrict__ b, unsigned n,
                                             double *__restrict__ part) {
    double s = 0.0;
    for (unsigned k = blockIdx.x * 256 + threadIdx.x; k < n; k += gridDim.x * 256) s = fma(a[k], b[k], s);
    s = block_tree(s);
    if (threadIdx.x == 0) part[blockIdx.x] = s;
}

// ---------------------------------------------------------------------------
// conjugate gradients.  One loop iteration: z = M r (V-cycle, carrying the
// partials of r . z), p = z + beta p, Ap with the partials of p . Ap, then
// x += alpha p, r -= alpha Ap with the partials of r . r and the next cycle's
// start values, and the loop decision.

// r = b - A x, the cycle's start values, and the partials of b . b and r . r
template <bool UNIT>
__global__ void __launch_bounds__(256) k_pcg_start(Op A, const double *__restrict__ x, const double *__restrict__ b,
                                                   double *__restrict__ r, double *__restrict__ zred,
                                                   double *__restrict__ zblack, double *__restrict__ part_bb,
                                                   double *__restrict__ part_rr) {
    double bb = 0.0, rr = 0.0;
    for (unsigned p = blockIdx.x * 256 + threadIdx.x; p < A.n; p += gridDim.x * 256) {
        const Pt q = pt_flat(A, p);
        const double bp = b[p];
        const double v = op_residual<UNIT>(A, x, q, bp);
        r[p] = v;
        if ((q.i + q.j + q.k) & 1) zblack[p] = 0.0;
        else zred[p] = quotient(v, A.dgn[p], A.idg[p]);
        bb = fma(bp, bp, bb);
        rr = fma(v, v, rr);
    }
    bb = block_tree(bb);
    rr = block_tree(rr);
    if (threadIdx.x == 0) {
        part_bb[blockIdx.x] = bb;
        part_rr[blockIdx.x] = rr;
    }
}

// p = z + beta p (p = z in the first iteration)
__global__ void __launch_bounds__(256) k_pcg_direction(double *__restrict__ p, const double *__restrict__ z, LinCtl *ctl,
                                                       const double *__restrict__ part_rz, int nb, unsigned n) {
    const int it = ctl->it;
    const bool first = it == 0;
    const double beta = of_partials(part_rz, nb, [&](double rz) {
        if (blockIdx.x == 0) ctl->rz[it & 1] = rz;
        return first ? 0.0 : rz / ctl->rz[(it + 1) & 1];
    });
    for (unsigned k = blockIdx.x * 256 + threadIdx.x; k < n; k += gridDim.x * 256)
        p[k] = first ? z[k] : fma(beta, p[k], z[k]);
}

// Ap = A p and the partials of p . Ap
template <bool UNIT>
__global__ void __launch_bounds__(256) k_pcg_apply(Op A, const double *__restrict__ p, double *__restrict__ Ap,
                                                   double *__restrict__ part) {
    double acc = 0.0;
    for (unsigned k = blockIdx.x * 256 + threadIdx.x; k < A.n; k += gridDim.x * 256) {
        const double u = p[k];
        const double v = fma(A.dgn[k], u, -op_nbr<UNIT>(A, p, p, pt_flat(A, k)));
        Ap[k] = v;
        acc = fma(u, v, acc);
    }
    acc = block_tree(acc);
    if (threadIdx.x == 0) part[blockIdx.x] = acc;
}

// x += alpha p, r -= alpha Ap, partials of r . r, start values of the next cycle
__global__ void __launch_bounds__(256) k_pcg_update(Op A, double *__restrict__ x, double *__restrict__ r,
                                                    const double *__restrict__ p, const double *__restrict__ Ap,
                                                    double *__restrict__ zred, double *__restrict__ zblack,
                                                    const LinCtl *__restrict__ ctl,
                                                    const double *__restrict__ part_pap, int nb,
                                                    double *__restrict__ part_rr) {
    const double alpha = of_partials(part_pap, nb, [&](double pap) { return ctl->rz[ctl->it & 1] / pap; });
    double acc = 0.0;
    for (unsigned k = blockIdx.x * 256 + threadIdx.x; k < A.n; k += gridDim.x * 256) {
        x[k] = fma(alpha, p[k], x[k]);
        const double v = fma(-alpha, Ap[k], r[k]);
        r[k] = v;
        acc = fma(v, v, acc);
        const Pt q = pt_flat(A, k);
        if ((q.i + q.j + q.k) & 1) zblack[k] = 0.0;
        else zred[k] = quotient(v, A.dgn[k], A.idg[k]);
    }
    acc = block_tree(acc);
    if (threadIdx.x == 0) part_rr[blockIdx.x] = acc;
}

// start of a linear solve: target = tol^2 ||b||^2; enter the loop unless the
// warm start already meets it
__global__ void k_pcg_init(LinCtl *ctl, const double *__restrict__ part_bb, const double *__restrict__ part_rr,
                           int nb, double tol, const DevStats *st, int *flag, cudaGraphConditionalHandle h) {
    double bb = partials_tree(part_bb, nb);
    const double rr = partials_tree(part_rr, nb);
    if (threadIdx.x != 0) return;
    if (!(tol > 0)) tol = st->lin_tol;      // adaptive: set by the Gummel loop
    if (!(bb > 0)) bb = 1.0;
    const double tgt = tol * tol * bb;
    ctl->tgt = tgt;
    ctl->it = 0;
    const bool finite = isfinite(rr);
    if (!finite) atomicOr(flag, kFlagOverflow);
    cudaGraphSetConditional(h, (finite && rr > tgt) ? 1u : 0u);
}

// end of a CG iteration: continue while ||r||^2 > target and below maxit
__global__ void k_pcg_check(LinCtl *ctl, const double *__restrict__ part_rr, int nb, int maxit, DevStats *st, int *flag,
                            cudaGraphConditionalHandle h) {
    const double rr = partials_tree(part_rr, nb);
    if (threadIdx.x != 0) return;
    const int it = ++ctl->it;
    atomicAdd(&st->lin, 1ull);        // lanes run side by side
    const bool finite = isfinite(rr);
    if (!finite) atomicOr(flag, kFlagOverflow);
    cudaGraphSetConditional(h, (finite && rr > ctl->tgt && it < maxit) ? 1u : 0u);
}

// ---------------------------------------------------------------------------
// The tail of the V-cycle in one CTA.
//
// A level of at most kTailMaxPoints points is a chain of ten small dependent
// phases; as separate launches each costs about 2 us, most of it launch and
// first-touch latency.  One CTA of 512 threads runs all of them between
// __syncthreads: iterate, right-hand side, residual, coefficients and neighbour
// places of every level stay in shared memory, split by colour, so a warp reads
// and writes consecutive words.  512 points of one colour are 16 warps, four on
// each quarter of the SM: 4 x 11 FP64 instructions of 64 clocks, 1.4 of the 1.6 us
// that a phase takes;
// a 12^3 level (2.8 us) is faster as chip-wide launches, so the line is 1024
// points.  The coarsest level (at most kCoarseWarp points) runs its 40
// symmetric sweeps in one warp, in registers.
constexpr int kTailThreads = 512;
constexpr int kTailMaxLevels = 10;
constexpr int kTailMaxPoints = 1024;
constexpr int kTailOwn = 2;             // points of one colour per thread, at most
constexpr int kCoarseWarp = 32;         // points of the coarsest level, at most
constexpr size_t kTailSmemMax = 200 * 1024;

struct TailLevel {
    Op A;
    int fx, fy, fz;                // factors to the next level
    FastDiv dfx, dfy, dfz;
    unsigned off;                  // byte offset of the level's arrays in shared memory
    double *cx, *cy, *cz, *czlo, *dg, *dgn, *idg;   // set-up only
};

struct TailArgs {
    int nl;                        // levels; the last one is the coarsest, solved by one warp
    TailLevel lv[kTailMaxLevels];
    const double *b;               // top right-hand side and solution (global)
    double *x;
    unsigned off_coarse;           // x of the coarsest level
};

constexpr int kTailDoubles = 11;   // x, b, r, idg, dgn and six faces per point
static size_t tail_level_bytes(unsigned nt) { return (size_t)2 * nt * (kTailDoubles * 8 + 6 * 4); }

// one level's arrays; slot of a point = colour * nt + t
struct TailView {
    const TailLevel *L;
    double *x, *b, *r, *id, *dn, *c;   // c: six arrays
    unsigned *nb;                      // six arrays of neighbour slots
    int nt;
    __device__ __forceinline__ TailView(unsigned char *sm, const TailLevel &l) : L(&l), nt((int)l.A.nt) {
        const int m = 2 * nt;
        x = reinterpret_cast<double *>(sm + l.off);
        b = x + m;
        r = b + m;
        id = r + m;
        dn = id + m;
        c = dn + m;
        nb = reinterpret_cast<unsigned *>(c + 6 * m);
    }
    __device__ __forceinline__ unsigned slot(int i, int j, int k) const {
        return ((i + j + k) & 1) * nt + ((unsigned)k * L->A.ny + j) * L->A.hx + (i >> 1);
    }
};

// coefficients and neighbour slots
__device__ __forceinline__ void tail_load(const TailView &v) {
    const Op &A = v.L->A;
    const int m = 2 * v.nt;
    for (int s = threadIdx.x; s < m; s += kTailThreads) {
        const int c = s >= v.nt;
        const Pt q = pt_colour(A, s - c * v.nt, c);
        double f[6] = {0, 0, 0, 0, 0, 0}, id = 0, dn = 0;
        unsigned nb[6];
#pragma unroll
        for (int e = 0; e < 6; ++e) nb[e] = s;
        if (q.i < A.nx) {
            id = A.idg[q.p];
            dn = A.dgn[q.p];
            f[0] = A.cx[q.p];
            f[1] = A.cx[nbr_xm(A, q)];
            f[2] = A.cy[q.p];
            f[3] = A.cy[nbr_ym(A, q)];
            nb[0] = v.slot(q.i + 1 == A.nx ? 0 : q.i + 1, q.j, q.k);
            nb[1] = v.slot(q.i == 0 ? A.nx - 1 : q.i - 1, q.j, q.k);
            nb[2] = v.slot(q.i, q.j + 1 == A.ny ? 0 : q.j + 1, q.k);
            nb[3] = v.slot(q.i, q.j == 0 ? A.ny - 1 : q.j - 1, q.k);
            if (q.k + 1 < A.nz) {
                f[4] = A.cz[q.p];
                nb[4] = v.slot(q.i, q.j, q.k + 1);
            }
            if (q.k > 0) {
                f[5] = A.cz[q.p - A.plane];
                nb[5] = v.slot(q.i, q.j, q.k - 1);
            }
        }
        v.id[s] = id;
        v.dn[s] = dn;
#pragma unroll
        for (int e = 0; e < 6; ++e) {
            v.c[e * m + s] = f[e];
            v.nb[e * m + s] = nb[e];
        }
    }
}

__device__ __forceinline__ double tail_nbr(const TailView &v, int s) {
    const int m = 2 * v.nt;
    double u[6];
#pragma unroll
    for (int e = 0; e < 6; ++e) u[e] = v.x[v.nb[e * m + s]];
    const double *c = v.c + s;
    double w = fma(c[0], u[0], c[m] * u[1]) + fma(c[2 * m], u[2], c[3 * m] * u[3]);
    w = fma(c[4 * m], u[4], w);              // zero coefficient where there is no neighbour
    return fma(c[5 * m], u[5], w);
}

// One colour sweep.  On odd levels the own colour's old values are read across
// the wrap, so the results are held until every thread has read.
__device__ __forceinline__ void tail_sweep(const TailView &v, int c) {
    double w[kTailOwn];
#pragma unroll
    for (int e = 0; e < kTailOwn; ++e) {
        const int t = threadIdx.x + e * kTailThreads, s = c * v.nt + t;
        if (t < v.nt) w[e] = quotient(v.b[s] + tail_nbr(v, s), v.dn[s], v.id[s]);
    }
    if (v.L->A.odd) __syncthreads();
#pragma unroll
    for (int e = 0; e < kTailOwn; ++e) {
        const int t = threadIdx.x + e * kTailThreads;
        if (t < v.nt) v.x[c * v.nt + t] = w[e];
    }
    __syncthreads();
}

// sum of the fine residuals over the aggregate of coarse cell (I, J, K)
__device__ __forceinline__ double tail_gather(const TailView &f, int I, int J, int K) {
    const TailLevel &L = *f.L;
    double s = 0;
    for (int c = 0; c < L.fz; ++c)
        for (int b = 0; b < L.fy; ++b)
            for (int a = 0; a < L.fx; ++a) s += f.r[f.slot(I * L.fx + a, J * L.fy + b, K * L.fz + c)];
    return s;
}

// The coarsest level in one warp: x = 0, then kCoarseSweeps symmetric (red,
// black, black, red) sweeps.  This chain of FP64 instructions (64 clocks each,
// 160 half sweeps) is what bounds small solves, so it is made as short as the
// sums allow: up to 16 points two lanes share one, one forming the x and one
// the y pair of products; a second sweep of the same colour changes nothing
// unless the colour couples to itself (odd wraps), so it is left out, as is a
// colour without points; and the sweeps end once one leaves every value as it
// was.  2x2x2 points: 81 half sweeps of 8 + 3 instructions instead of 160 of 24.
// Lane < n gives b and gets x.
__device__ __forceinline__ double coarse_warp(const Op &A, double b) {
    const int lane = threadIdx.x & 31, n = (int)A.n;
    const bool split = n <= 16;
    const int me = split ? lane & 15 : lane, half = split ? lane >> 4 : 0;
    const bool in = me < n;
    const Pt q = pt_flat(A, in ? me : 0);
    b = __shfl_sync(0xffffffffu, b, me);
    const int xp = (int)nbr_xp(A, q), xm = (int)nbr_xm(A, q), yp = (int)nbr_yp(A, q), ym = (int)nbr_ym(A, q);
    const double cxp = A.cx[q.p], cxm = A.cx[xm], cyp = A.cy[q.p], cym = A.cy[ym];
    const bool up = q.k + 1 < A.nz, dn = q.k > 0;
    const int lu = up ? (int)(q.p + A.plane) : (int)q.p, ld = dn ? (int)(q.p - A.plane) : (int)q.p;
    const double cu = up ? A.cz[q.p] : 0.0, cd = dn ? A.cz[q.p - A.plane] : 0.0;
    const double d = A.dgn[q.p], y = A.idg[q.p];
    const int colour = (q.i + q.j + q.k) & 1;
    const bool black = __any_sync(0xffffffffu, in && colour == 1);
    const bool one_z = A.nz == 2;              // every point has one z neighbour
    const int l1 = half ? yp : xp, l2 = half ? ym : xm;
    const double c1 = half ? cyp : cxp, c2 = half ? cym : cxm;
    const int lz = up ? lu : ld;
    const double cz = up ? cu : cd;
    double x = 0.0;
    auto sweep = [&](int c) {
        const double t1 = __shfl_sync(0xffffffffu, x, l1), t2 = __shfl_sync(0xffffffffu, x, l2);
        double s;
        if (split) {
            s = fma(c1, t1, c2 * t2);
            s += __shfl_xor_sync(0xffffffffu, s, 16);
        } else {
            const double u1 = __shfl_sync(0xffffffffu, x, yp), u2 = __shfl_sync(0xffffffffu, x, ym);
            s = fma(cxp, t1, cxm * t2) + fma(cyp, u1, cym * u2);
        }
        if (one_z) {
            s = fma(cz, __shfl_sync(0xffffffffu, x, lz), s);
        } else if (A.nz > 1) {
            const double zu = __shfl_sync(0xffffffffu, x, lu), zd = __shfl_sync(0xffffffffu, x, ld);
            s = fma(cu, zu, s);
            s = fma(cd, zd, s);
        }
        const double v = quotient(b + s, d, y);
        if (in && colour == c) x = v;
    };
    for (int k = 0; k < kCoarseSweeps; ++k) {
        const double old = x;
        if (A.odd || k == 0) sweep(0);
        if (black) {
            sweep(1);
            if (A.odd) sweep(1);
        }
        if (A.odd || black) sweep(0);
        if (__all_sync(0xffffffffu, __double_as_longlong(x) == __double_as_longlong(old))) break;
    }
    return x;
}

__global__ void __launch_bounds__(kTailThreads) k_tail(const __grid_constant__ TailArgs a) {
    extern __shared__ __align__(16) unsigned char tail_sm[];
    const int last = a.nl - 1;
    const Op &D = a.lv[last].A;
    double *dx = reinterpret_cast<double *>(tail_sm + a.off_coarse);
    if (last == 0) {
        // the tail is the coarsest level alone
        if (threadIdx.x < 32) {
            const double x = coarse_warp(D, threadIdx.x < D.n ? a.b[threadIdx.x] : 0.0);
            if (threadIdx.x < D.n) a.x[threadIdx.x] = x;
        }
        return;
    }
    for (int l = 0; l < last; ++l) tail_load(TailView(tail_sm, a.lv[l]));
    const TailView top(tail_sm, a.lv[0]);
    for (int l = 0; l < last; ++l) {
        // right-hand side (the restricted residual) and start values, then
        // black, red, black and the residual
        const TailView v(tail_sm, a.lv[l]);
        const Op &A = v.L->A;
        for (int s = threadIdx.x; s < 2 * v.nt; s += kTailThreads) {
            const int c = s >= v.nt;
            const Pt q = pt_colour(A, s - c * v.nt, c);
            double r = 0.0;
            if (q.i < A.nx) r = l == 0 ? a.b[q.p] : tail_gather(TailView(tail_sm, a.lv[l - 1]), q.i, q.j, q.k);
            v.b[s] = r;
            v.x[s] = c == 0 ? quotient(r, v.dn[s], v.id[s]) : 0.0;
        }
        __syncthreads();
        tail_sweep(v, 1);
        tail_sweep(v, 0);
        tail_sweep(v, 1);
        for (int s = threadIdx.x; s < 2 * v.nt; s += kTailThreads)
            v.r[s] = v.b[s] - (__dmul_rn(v.dn[s], v.x[s]) - tail_nbr(v, s));
        __syncthreads();
    }
    if (threadIdx.x < 32) {
        const TailView f(tail_sm, a.lv[last - 1]);
        const bool in = threadIdx.x < D.n;
        const Pt Q = pt_flat(D, in ? threadIdx.x : 0);
        const double x = coarse_warp(D, in ? tail_gather(f, Q.i, Q.j, Q.k) : 0.0);
        if (in) dx[threadIdx.x] = x;
    }
    __syncthreads();
    for (int l = last - 1; l >= 0; --l) {
        // coarse correction (red points; all on odd levels), then black, red,
        // black, red
        const TailView v(tail_sm, a.lv[l]);
        const Op &A = v.L->A;
        for (int s = threadIdx.x; s < (1 + A.odd) * v.nt; s += kTailThreads) {
            const int c = s >= v.nt;
            const Pt q = pt_colour(A, s - c * v.nt, c);
            if (q.i >= A.nx) continue;
            const int I = v.L->dfx.div(q.i), J = v.L->dfy.div(q.j), K = v.L->dfz.div(q.k);
            const double xc = l + 1 == last ? dx[((unsigned)K * D.ny + J) * D.nx + I]
                                            : TailView(tail_sm, a.lv[l + 1]).x[TailView(tail_sm, a.lv[l + 1]).slot(I, J, K)];
            v.x[s] = fma(kCoarseScale, xc, v.x[s]);
        }
        __syncthreads();
        tail_sweep(v, 1);
        tail_sweep(v, 0);
        tail_sweep(v, 1);
        tail_sweep(v, 0);
    }
    for (int s = threadIdx.x; s < 2 * top.nt; s += kTailThreads) {
        const int c = s >= top.nt;
        const Pt q = pt_colour(top.L->A, s - c * top.nt, c);
        if (q.i < top.L->A.nx) a.x[q.p] = top.x[s];
    }
}

// The tail's levels of a new operator: coarse faces (coarsen != 0) and extra
// diagonal of every level below the first, and their diagonals.
__global__ void __launch_bounds__(kTailThreads) k_tail_setup(const __grid_constant__ TailArgs a, int coarsen) {
    for (int l = 0; l + 1 < a.nl; ++l) {
        const TailLevel &F = a.lv[l], &C = a.lv[l + 1];
        for (unsigned q = threadIdx.x; q < C.A.n; q += kTailThreads) {
            if (coarsen) coarsen_cell(F.A, F.fx, F.fy, F.fz, C.A, q, C.cx, C.cy, C.cz, C.czlo);
            if (F.A.dg) C.dg[q] = aggregate_sum(F.A, F.A.dg, F.fx, F.fy, F.fz, pt_flat(C.A, q));
        }
        __syncthreads();
        for (unsigned p = threadIdx.x; p < C.A.n; p += kTailThreads) {
            const double d = op_diag(C.A, pt_flat(C.A, p));
            C.dgn[p] = d;
            C.idg[p] = 1.0 / d;
        }
    }
}

}  // namespace pnp
