// Batched solve of many independent problems of uneven size, each with its
// own right-hand sides: the V-cycles (Algorithm 1) with multiplicative
// red-black cascade smoothing (eq. fwdm and its reverse), the FP64 residual
// and the update of every problem run in ONE persistent cooperative kernel
// per solve, launched from a CUDA graph.  Stages are separated by grid-wide
// barriers; the levels of all problems are aligned at the coarsest, so that
// level slot t of the batch holds level t - (D - nlev_p) of problem p
// (D = the largest level count) and every stage is one ragged sweep over the
// slot's levels.  Work is dealt out in tiles (a problem, a level, a contiguous
// range of its grid rows' nodes) of about equal work; the number of tiles per
// CTA and the CTA size are picked by a measuring autotuner.
//
// Data layout: vectors of problem p hold its m_p right-hand sides
// contiguously per node, v[i * m_p + r] (m_p <= 8); operators and Lambda are
// the problem's own level arrays (structure of arrays, FP32 or FP64).
#include <cooperative_groups.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "cs_internal.cuh"

namespace cg = cooperative_groups;

namespace csx {

constexpr int BMAXLEV = 16;
constexpr int BMAXRHS = 32;
constexpr int BMAXRESTART = 256;
constexpr int RED_DOUBLES = 4 * 512;  // the kernel's shared reduction buffer

template <typename T>
struct BLevel {
    int nx, ny, kind, inplace;
    int64_t N;
    int bs, nbx, nmax;  // blocks of bs x bs nodes (1: point blocks), nbx per row, nmax = bs^2
    int64_t nblocks;
    const T *A;    // [nst][N]
    const T *lam;  // [nu][N] (points) or [nu][nblocks][nmax][nmax] (blocks)
    T *b, *x, *t;  // [N][m]
};

template <typename T>
struct BProb {
    int nlev, m, slot0, cn;
    const double *A64;   // finest operator, FP64
    const double *cinv;  // coarsest dense inverse, FP64 row-major
    T *Z;                // GMRES work vector [N0][m] (the cycle precision)
    T *V;                // GMRES basis: restart + 1 vectors of [N0][m]
    T *ZB;               // right-preconditioned GMRES: restart vectors Z_j = M V_j of [N0][m]
    BLevel<T> lev[BMAXLEV];
};

struct BTile {
    int p, l, i0, ni;
};

// A tail item: right-hand sides r0 .. r0 + rc - 1 of problem p.
struct BTail {
    int p, r0, rc;
};

enum { OP_SWEEP = 0, OP_RESTRICT = 1, OP_COARSE = 2, OP_PROLONG = 3, OP_FRES = 4 };
// colour >= 0: a multiplicative colour step (in place on 5-point levels, else
// x -> t for parity 0 and t -> x for parity 1); colour < 0: an additive step
// from buffer src to dst (0: x, 1: t).  OP_FRES writes the residual of the
// iterate in src into dst, OP_RESTRICT gathers the coarse level's right-hand
// side from the fine level's buffer src; prolongation reads src and writes dst.  transpose: Lambda^T
// (the reversed smoother on block levels).
struct BStep {
    int op, slot, lv, colour, parity, src, dst, transpose;
};

struct BCtl {
    double tol;
    int maxit;
    int cnt[2];  // counts of the counting stages, alternating slots
};

enum { ST_ACTIVE = 0, ST_CONVERGED = 1, ST_DIVERGED = 2, ST_MAXIT = 3 };

struct BArgs {
    const void *probs;
    int nprob;
    const BTile *tiles;      // tiles of slot t: [slot_tile[t], slot_tile[t + 1])
    const int *slot_tile;
    const BTile *btiles;     // block tiles (i0, ni in blocks) of slot t, for block-level sweeps
    const int *slot_btile;
    int dmax;
    const BTile *ftiles;     // finest-level tiles; problem p: [ftile_of[p], ftile_of[p + 1])
    const int *ftile_of;
    int nftiles;
    const BStep *steps;
    int nsteps;
    // the cycle's tail: steps [tail_lo, tail_hi) touch the slots below the
    // tail slot only and run per (problem, right-hand sides) in one CTA each
    const BTail *tails;
    int ntails, tail_lo, tail_hi;
    const double *const *b64;  // per problem, [N0][m]
    double *const *x64;
    double *part;   // [nftiles][BMAXRHS]
    double *nb;     // [nprob][BMAXRHS]
    double *rel;    // [nprob][BMAXRHS]
    double *rel0;   // [nprob]
    int *state;     // [nprob]
    int *iters;     // [nprob]
    int *work;      // [nprob]: the problem takes part in the cycle stages
    BCtl *ctl;
    // GMRES (restarted, left or right preconditioned; per problem and right-hand side q = p * BMAXRHS + r)
    int method, restart, hstride;
    double *H;      // [q][(restart + 1) * restart]
    double *cs, *sn, *y;  // [q][restart]
    double *g;      // [q][restart + 1]
    double *inv;    // [q]: 1 / ||Z|| of the last normalisation
    double *nmb;    // [q]: ||M b|| (left) or ||b|| (right): the scale of the GMRES stopping test
    int *jcols;     // [q]: Krylov columns built in this cycle
    int *frozen;    // [q]: no longer extending in this cycle
    // classical Gram-Schmidt: per-tile projection partials, problem p's
    // block at p2off[p], [tile of p][slot i < restart + 2][r < m_p]
    double *part2;
    const int64_t *p2off;
    int qtot;            // right-hand sides of all problems
    const int *qlist;    // [qtot]: q = p * BMAXRHS + r
    double *hsum;        // [q][restart + 2]: this pass's <Z, V_i> (slot j + 1: <Z, Z>)
    double *znorm2;      // [q]: ||Z||^2 after the first projection
    int *reorth;         // [q]: the step projects a second time
    double *beta;        // [q]: ||M r|| at the start of the GMRES cycle
    double itol;         // inner stop |g_{j+1}| <= itol beta (FP32 Krylov vectors), 0: none
};

__device__ __forceinline__ int bcolour(int ix, int iy) { return ((ix + 1) + (iy + 1)) & 1; }

template <int KIND>
__device__ __forceinline__ void boff(int s, int &dx, int &dy) {
    if (KIND == STAR) {
        dx = s == 1 ? -1 : s == 2 ? 1 : 0;
        dy = s == 3 ? -1 : s == 4 ? 1 : 0;
    } else {
        dx = s % 3 - 1;
        dy = s / 3 - 1;
    }
}

// (A v)_{i,r} at node i = (ix, iy), computed in T; neighbours outside
// contribute nothing
template <int KIND, typename T, typename TA, typename TV = T>
__device__ __forceinline__ T row_apply(int nx, int ny, int64_t N, const TA *__restrict__ A, const TV *v, int m, int r,
                                       int ix, int iy, int i) {
    constexpr int NST = KIND == STAR ? 5 : 9;
    T ax = T(0);
#pragma unroll
    for (int s = 0; s < NST; ++s) {
        int dx, dy;
        boff<KIND>(s, dx, dy);
        const bool in = (unsigned)(ix + dx) < (unsigned)nx && (unsigned)(iy + dy) < (unsigned)ny;
        const T a = (T)A[(int64_t)s * N + i];
        const int j = i + dx + nx * dy;
        ax = fma(a, in ? (T)v[(int64_t)j * m + r] : T(0), ax);
    }
    return ax;
}

// Work items of a tile: item (node, right-hand side r).  Thread t < U, U the
// largest multiple of m not above the CTA size, takes r = t % m for the
// nodes i0 + t / m + k U / m, so no index is divided per item and the m
// threads of a node are adjacent (its coefficient loads are one broadcast).
struct TileMap {
    int r, n0, step;
    bool on;
};
__device__ __forceinline__ TileMap tile_map(int m, int r0 = 0) {
    TileMap t;
    const int U = ((int)blockDim.x / m) * m;
    t.on = (int)threadIdx.x < U;
    t.r = r0 + (int)threadIdx.x % m;
    t.n0 = (int)threadIdx.x / m;
    t.step = U / m;
    return t;
}

// Deterministic CTA sums per right-hand side: red[t] holds thread t's sum;
// threads t and t + k m (same r) are combined by a fixed pairwise tree over
// the groups g = t / m; out[r] = the sum of right-hand side r.
__device__ __forceinline__ void cta_sum_by_rhs(double v, int m, double *red, double *out) {
    const int t = threadIdx.x;
    const int G = (int)blockDim.x / m, U = G * m;
    red[t] = t < U ? v : 0.0;
    __syncthreads();
    int P = 1;
    while (2 * P <= G) P *= 2;
    if (t < (G - P) * m) red[t] += red[t + P * m];  // fold the groups beyond the largest power of two
    __syncthreads();
    for (int h = P / 2; h > 0; h /= 2) {
        if (t < h * m) red[t] += red[t + h * m];
        __syncthreads();
    }
    if (t < m) out[t] = red[t];
    __syncthreads();
}

// The same tree for nv <= 4 sums at once (red holds 4 x blockDim.x values):
// out[u * ostride + r] = the sum of value u over right-hand side r.
__device__ __forceinline__ void cta_sum4_by_rhs(const double *v, int nv, int m, double *red, double *out,
                                                int ostride) {
    const int t = threadIdx.x, T = (int)blockDim.x;
    const int G = T / m, U = G * m;
#pragma unroll
    for (int u = 0; u < 4; ++u) red[u * T + t] = t < U && u < nv ? v[u] : 0.0;
    __syncthreads();
    int P = 1;
    while (2 * P <= G) P *= 2;
    if (t < (G - P) * m)
#pragma unroll
        for (int u = 0; u < 4; ++u) red[u * T + t] += red[u * T + t + P * m];
    __syncthreads();
    for (int h = P / 2; h > 0; h /= 2) {
        if (t < h * m)
#pragma unroll
            for (int u = 0; u < 4; ++u) red[u * T + t] += red[u * T + t + h * m];
        __syncthreads();
    }
    if (t < m)
        for (int u = 0; u < nv; ++u) out[u * ostride + t] = red[u * T + t];
    __syncthreads();
}

// ------------------------------------------------------------- stages
// (the level descriptors are read once per tile into registers: the item
// loops touch only plain pointers and sizes)
// Items are taken SW at a time, all loads before any store: in place (a
// graph colouring) the loads of a colour step read only entries of the other
// colour, which its stores never touch, so the order is free, and the SW
// independent load groups keep SW times more requests in flight per thread.
constexpr int SW = 4;
// Krylov dot products and norms: products are summed in the vector precision
// over up to KCH items, and those partial sums in FP64 (on this part FP64
// adds issue at 1/64 of the FP32 rate, so FP32 vectors keep them rare)
constexpr int KCH = 8;

// Red-black colour c = (ix + iy) mod 2 of the nodes of an nx-wide grid,
// enumerated in index order: colour_before counts the colour-c nodes with
// index below i; colour_node gives the g-th one.  With nx odd the colour is
// i mod 2; with nx even every row holds nx / 2 nodes of each colour, at the
// x-parity (c + iy) mod 2.
__device__ __forceinline__ int colour_before(int nx, int c, int i) {
    if (nx & 1) return (i + 1 - c) >> 1;
    const int iy = i / nx, ix = i - iy * nx;
    return iy * (nx >> 1) + ((ix + 1 - ((c + iy) & 1)) >> 1);
}
__device__ __forceinline__ void colour_node(int nx, int c, int g, int &i, int &ix, int &iy) {
    if (nx & 1) {
        i = 2 * g + c;
        iy = i / nx;
        ix = i - iy * nx;
    } else {
        const int h = nx >> 1;
        iy = g / h;
        ix = 2 * (g - iy * h) + ((c + iy) & 1);
        i = ix + iy * nx;
    }
}

// x_i - lambda_i ((A x)_i - b_i) for cnt nodes: the nodes g0 .. g0 + cnt - 1
// (COL false) or the colour-`colour` nodes of those ranks (COL true)
template <typename T, int KIND, bool COL>
__device__ __forceinline__ void relax_nodes(int nx, int ny, int64_t N, const T *__restrict__ A,
                                            const T *__restrict__ lam, const T *__restrict__ b, int m, int r,
                                            int g0, int cnt, int n0, int step, int colour, const T *src, T *dst) {
    for (int nn = n0; nn < cnt; nn += SW * step) {
        T val[SW];
        int64_t ee[SW];
        bool wr[SW];
#pragma unroll
        for (int u = 0; u < SW; ++u) {
            const int n = nn + u * step;
            wr[u] = false;
            ee[u] = 0;
            val[u] = T(0);
            if (n < cnt) {
                int i, ix, iy;
                if (COL) {
                    colour_node(nx, colour, g0 + n, i, ix, iy);
                } else {
                    i = g0 + n;
                    iy = i / nx;
                    ix = i - iy * nx;
                }
                const int64_t e = (int64_t)i * m + r;
                ee[u] = e;
                const T ax = row_apply<KIND, T, T>(nx, ny, N, A, src, m, r, ix, iy, i);
                const T res = ax - b[e];
                val[u] = src[e] - lam[i] * res;
                wr[u] = true;
            }
        }
#pragma unroll
        for (int u = 0; u < SW; ++u)
            if (wr[u]) dst[ee[u]] = val[u];
    }
}

// One cascade step over the tile's nodes [i0, i0 + ni).  A colour step
// (colour >= 0) deals out only the nodes of its colour, so no lane idles on
// the other colour; out of place it then copies the other colour's nodes.
template <typename T, int KIND>
__device__ __forceinline__ void sweep_tile(int nx, int ny, int64_t N, const T *__restrict__ A,
                                           const T *__restrict__ lam, const T *__restrict__ b, int m, int r, int i0,
                                           int ni, int n0, int step, int colour, const T *src, T *dst) {
    if (colour < 0) {
        relax_nodes<T, KIND, false>(nx, ny, N, A, lam, b, m, r, i0, ni, n0, step, -1, src, dst);
        return;
    }
    const int g0 = colour_before(nx, colour, i0);
    relax_nodes<T, KIND, true>(nx, ny, N, A, lam, b, m, r, g0, colour_before(nx, colour, i0 + ni) - g0, n0, step,
                               colour, src, dst);
    if (src != dst) {
        const int oc = colour ^ 1, h0 = colour_before(nx, oc, i0), hc = colour_before(nx, oc, i0 + ni) - h0;
#pragma unroll 4
        for (int nn = n0; nn < hc; nn += step) {
            int i, ix, iy;
            colour_node(nx, oc, h0 + nn, i, ix, iy);
            const int64_t e = (int64_t)i * m + r;
            dst[e] = src[e];
        }
    }
}

// Block step over a range of blocks (one thread per block and right-hand
// side): the residual rows of the block's present nodes, then
// x_b -= Lambda_b^(T) r_b (eq. fwda / fwdm with block Lambda).  Blocks of the
// other colour are copied when the step is not in place.
template <typename T, int KIND, int BS>
__device__ __forceinline__ void block_sweep_tile(int nx, int ny, int64_t N, int nbx, const T *__restrict__ A,
                                                 const T *__restrict__ lam, const T *__restrict__ b, int m, int r,
                                                 int b0, int nb, int n0, int step, int colour, int transpose,
                                                 const T *src, T *dst) {
    constexpr int NM = BS * BS;
    const bool copy = src != dst;
    for (int nn = n0; nn < nb; nn += step) {
        const int blk = b0 + nn;
        const int by = blk / nbx, bx = blk - by * nbx;
        int node[NM];
        bool pres[NM];
#pragma unroll
        for (int lp = 0; lp < NM; ++lp) {
            const int ix = BS * bx + lp % BS, iy = BS * by + lp / BS;
            pres[lp] = ix < nx && iy < ny;
            node[lp] = ix + nx * iy;
        }
        if (colour >= 0 && (((bx + 1) + (by + 1)) & 1) != colour) {
            if (copy)
#pragma unroll
                for (int lp = 0; lp < NM; ++lp)
                    if (pres[lp]) dst[(int64_t)node[lp] * m + r] = src[(int64_t)node[lp] * m + r];
            continue;
        }
        T res[NM], xv[NM];
#pragma unroll 1
        for (int lp = 0; lp < NM; ++lp) {
            res[lp] = T(0);
            xv[lp] = T(0);
            if (pres[lp]) {
                const int i = node[lp], iy = i / nx, ix = i - iy * nx;
                const int64_t e = (int64_t)i * m + r;
                res[lp] = row_apply<KIND, T, T>(nx, ny, N, A, src, m, r, ix, iy, i) - b[e];
                xv[lp] = src[e];
            }
        }
        const T *lb = lam + (int64_t)blk * (NM * NM);
#pragma unroll 1
        for (int lp = 0; lp < NM; ++lp) {
            if (!pres[lp]) continue;
            T acc = xv[lp];
#pragma unroll
            for (int q = 0; q < NM; ++q)
                acc = fma(-(transpose ? lb[q * NM + lp] : lb[lp * NM + q]), res[q], acc);
            dst[(int64_t)node[lp] * m + r] = acc;
        }
    }
}

// r = A x - b on a level: the restriction's fine residuals, once each.  One
// stage that formed the nine residuals of every coarse node itself took 37 us
// on the finest slot of 16 problems; these two take 14 and 10.
template <typename T, int KIND>
__device__ __forceinline__ void residual_tile(int nx, int ny, int64_t N, const T *__restrict__ A, const T *x,
                                              const T *__restrict__ b, T *rr, int m, int r, int i0, int ni, int n0,
                                              int step) {
#pragma unroll 2
    for (int nn = n0; nn < ni; nn += step) {
        const int i = i0 + nn, iy = i / nx, ix = i - iy * nx;
        const int64_t e = (int64_t)i * m + r;
        rr[e] = row_apply<KIND, T, T>(nx, ny, N, A, x, m, r, ix, iy, i) - b[e];
    }
}

// coarse node I of level l+1: b_c = 2^-2 sum_f P_{f,I} r_f, x_c = 0
template <typename T>
__device__ __forceinline__ void restrict_tile(int fnx, int fny, const T *rf, int cnx, T *__restrict__ bc,
                                              T *__restrict__ xc, int m, int r, int i0, int ni, int n0, int step) {
    for (int nn = n0; nn < ni; nn += step) {
        const int I = i0 + nn;
        const int cy = I / cnx, cx = I - cy * cnx;
        T v[9];
#pragma unroll
        for (int t = 0; t < 9; ++t) {
            const int fy = 2 * cy + t / 3, fx = 2 * cx + t % 3;
            v[t] = fy < fny && fx < fnx ? rf[(int64_t)(fx + fnx * fy) * m + r] : T(0);
        }
        T acc = T(0);
#pragma unroll
        for (int t = 0; t < 9; ++t)
            if (2 * cy + t / 3 < fny && 2 * cx + t % 3 < fnx)
                acc = fma(T((t % 3 != 1 ? 0.5 : 1.0) * (t / 3 != 1 ? 0.5 : 1.0)), v[t], acc);
        bc[(int64_t)I * m + r] = acc * T(0.25);
        xc[(int64_t)I * m + r] = T(0);
    }
}

// 1D interpolation weights of fine node f from the coarse nodes (as in the
// single-problem prolongation): odd f sits on coarse (f-1)/2, even f takes
// half of coarse f/2-1 and f/2 where present.
__device__ __forceinline__ int bp1d(int f, int nc, int *c, float *w) {
    if (f & 1) {
        c[0] = (f - 1) >> 1;
        w[0] = 1.f;
        return 1;
    }
    int k = 0;
    const int lo = (f >> 1) - 1, hi = f >> 1;
    if (lo >= 0) { c[k] = lo; w[k] = 0.5f; ++k; }
    if (hi < nc) { c[k] = hi; w[k] = 0.5f; ++k; }
    return k;
}

template <typename T>
__device__ __forceinline__ void prolong_tile(int fnx, const T *xs, T *xf, int cnx, int cny,
                                             const T *__restrict__ xc, int m, int r, int i0, int ni, int n0,
                                             int step) {
    for (int nn = n0; nn < ni; nn += step) {
        const int f = i0 + nn;
        const int fy = f / fnx, fx = f - fy * fnx;
        int cxs[2], cys[2];
        float wx[2], wy[2];
        const int kx = bp1d(fx, cnx, cxs, wx), ky = bp1d(fy, cny, cys, wy);
        T acc = T(0);
        for (int bb = 0; bb < ky; ++bb)
            for (int a = 0; a < kx; ++a) {
                const T w = T(wx[a] * wy[bb] * 1.f);
                const int c = cxs[a] + cnx * cys[bb];
                acc = fma(w, xc[(int64_t)c * m + r], acc);
            }
        const int64_t e = (int64_t)f * m + r;
        xf[e] = xs[e] - acc;
    }
}

// One cycle step over the items [i0, i0 + ni) (blocks for sweeps of block
// levels, else nodes) of the problem's level l (described by *Lp).
template <typename T>
__device__ __forceinline__ void op_tile(const BProb<T> &pr, const BLevel<T> *Lp, const BStep &st, int l, int i0, int ni, int m, bool blocks,
                                        const TileMap &tm) {
    const int r = tm.r;
    if (st.op == OP_SWEEP) {
        const BLevel<T> L = *Lp;
        const T *src;
        T *dst;
        if (st.colour >= 0) {
            src = L.inplace || st.parity == 0 ? L.x : L.t;
            dst = L.inplace || st.parity == 1 ? L.x : L.t;
        } else {
            src = st.src ? L.t : L.x;
            dst = st.dst ? L.t : L.x;
        }
        if (blocks) {
            const T *lamb = L.lam + (int64_t)st.lv * L.nblocks * L.nmax * L.nmax;
            if (L.kind == STAR)  // 2x2-node blocks (the batch plan admits no others)
                block_sweep_tile<T, STAR, 2>(L.nx, L.ny, L.N, L.nbx, L.A, lamb, L.b, m, r, i0, ni,
                                             tm.n0, tm.step, st.colour, st.transpose, src, dst);
            else
                block_sweep_tile<T, BOX, 2>(L.nx, L.ny, L.N, L.nbx, L.A, lamb, L.b, m, r, i0, ni, tm.n0,
                                            tm.step, st.colour, st.transpose, src, dst);
            return;
        }
        const T *lam = L.lam + (int64_t)st.lv * L.N;
        if (L.kind == STAR)
            sweep_tile<T, STAR>(L.nx, L.ny, L.N, L.A, lam, L.b, m, r, i0, ni, tm.n0, tm.step, st.colour,
                                src, dst);
        else
            sweep_tile<T, BOX>(L.nx, L.ny, L.N, L.A, lam, L.b, m, r, i0, ni, tm.n0, tm.step, st.colour,
                               src, dst);
    } else if (st.op == OP_FRES) {
        const BLevel<T> L = *Lp;
        const T *x = st.src ? L.t : L.x;
        T *rr = st.dst ? L.t : L.x;
        if (L.kind == STAR)
            residual_tile<T, STAR>(L.nx, L.ny, L.N, L.A, x, L.b, rr, m, r, i0, ni, tm.n0, tm.step);
        else
            residual_tile<T, BOX>(L.nx, L.ny, L.N, L.A, x, L.b, rr, m, r, i0, ni, tm.n0, tm.step);
    } else if (st.op == OP_RESTRICT) {
        const BLevel<T> F = pr.lev[l - 1], C = *Lp;
        restrict_tile<T>(F.nx, F.ny, st.src ? F.t : F.x, C.nx, C.b, C.x, m, r, i0, ni, tm.n0, tm.step);
    } else if (st.op == OP_COARSE) {
        const BLevel<T> L = *Lp;
        const int n = pr.cn;
        const double *__restrict__ cinv = pr.cinv;
        const T *__restrict__ lb = L.b;
        T *__restrict__ lx = L.x;
        for (int nn = tm.n0; nn < ni; nn += tm.step) {
            const int i = i0 + nn;
            double sacc = 0.0;
            for (int j = 0; j < n; ++j) sacc = fma(cinv[(int64_t)i * n + j], (double)lb[(int64_t)j * m + r], sacc);
            lx[(int64_t)i * m + r] = (T)sacc;
        }
    } else {  // OP_PROLONG
        const BLevel<T> F = *Lp, C = pr.lev[l + 1];
        prolong_tile<T>(F.nx, st.src ? F.t : F.x, st.dst ? F.t : F.x, C.nx, C.ny, C.x, m, r, i0, ni,
                        tm.n0, tm.step);
    }
}

// A CTA's tiles of every slot with their level's description, kept in shared
// memory: a stage otherwise starts with three dependent loads (tile, the
// problem's work flag, the level), each from L2, since a grid barrier drops
// L1.  The flags change only in the per-problem stages: they are read once per
// cycle.  CTAs with more tiles than fit read them from the tables.
template <typename T>
struct CTile {
    BLevel<T> L;
    BTile t;
    int m, on;
};
constexpr int CT_MAX = 32;
template <typename T>
struct Cache {
    CTile<T> tile[CT_MAX];
    int first[BMAXLEV + 1];  // tiles of slot t: [first[t], first[t + 1])
    int n;                   // 0: not cached
};

template <typename T>
__device__ void cache_tiles(const BArgs &a, const BProb<T> *P, Cache<T> &c) {
    if (threadIdx.x == 0) {
        int n = 0;
        for (int t = 0; t < a.dmax; ++t) {
            c.first[t] = n;
            for (int k = a.slot_tile[t] + blockIdx.x; k < a.slot_tile[t + 1]; k += gridDim.x) {
                if (n < CT_MAX) {
                    c.tile[n].t = a.tiles[k];
                    c.tile[n].m = P[c.tile[n].t.p].m;
                    c.tile[n].L = P[c.tile[n].t.p].lev[c.tile[n].t.l];
                }
                ++n;
            }
        }
        c.first[a.dmax] = n;
        c.n = n <= CT_MAX ? n : 0;
    }
    __syncthreads();
}
template <typename T>
__device__ __forceinline__ void cache_flags(const BArgs &a, Cache<T> &c) {
    for (int e = threadIdx.x; e < c.n; e += blockDim.x) c.tile[e].on = __ldcg(a.work + c.tile[e].t.p);
    __syncthreads();
}

// Step s of the cycle over its slot's tiles; or, at the tail's first step,
// the whole cycle below the tail slot, one CTA per (problem, right-hand
// sides) with CTA barriers between the steps: those levels are too small for
// a grid barrier and a tile's start-up latency per step.
template <typename T>
__device__ void stage_step(const BArgs &a, const BProb<T> *P, int s, Cache<T> &cache) {
    const bool tail = s == a.tail_lo && a.tail_hi > a.tail_lo;
    const BStep s0 = a.steps[s];
    const int tslot = s0.op == OP_RESTRICT ? s0.slot + 1 : s0.slot;
    const bool bl0 = s0.op == OP_SWEEP && a.btiles != nullptr;
    const bool cached = !tail && !bl0 && cache.n > 0;
    const BTile *tiles = bl0 ? a.btiles : a.tiles;
    const int *slot_tile = bl0 ? a.slot_btile : a.slot_tile;
    const int t0 = cached ? cache.first[tslot] : (tail ? 0 : slot_tile[tslot]) + (int)blockIdx.x;
    const int t1 = cached ? cache.first[tslot + 1] : tail ? a.ntails : slot_tile[tslot + 1];
    for (int k = t0; k < t1; k += cached ? 1 : (int)gridDim.x) {
        BTile tile;
        BTail tt = {0, 0, 0};
        if (cached) {
            tile = cache.tile[k].t;
            if (!cache.tile[k].on) continue;  // the same for the whole CTA, here and below
        } else {
            if (tail) {
                tt = a.tails[k];
                tile.p = tt.p;
            } else {
                tile = tiles[k];
            }
            if (__ldcg(a.work + tile.p) == 0) continue;
        }
        const BProb<T> &pr = P[tile.p];
        const int m = cached ? cache.tile[k].m : pr.m;
        const TileMap tm = tail ? tile_map(tt.rc, tt.r0) : tile_map(m);
        const int s1 = tail ? a.tail_hi : s + 1;
        for (int q = s; q < s1; ++q) {
            const BStep st = a.steps[q];
            const bool blocks = st.op == OP_SWEEP && a.btiles != nullptr;
            if (tail) {
                // a problem's levels begin at its slot0
                tile.l = (st.op == OP_RESTRICT ? st.slot + 1 : st.slot) - pr.slot0;
                if (tile.l < 0) continue;
                tile.i0 = 0;
                tile.ni = (int)(blocks ? pr.lev[tile.l].nblocks : pr.lev[tile.l].N);
            }
            if (st.op == OP_RESTRICT && tile.l == 0) continue;  // this problem's finest level starts at the coarse slot
            if (tm.on) op_tile<T>(pr, cached ? &cache.tile[k].L : &pr.lev[tile.l], st, tile.l, tile.i0, tile.ni, m, blocks, tm);
            if (tail) __syncthreads();
        }
    }
}

// finest-level FP64 stages over the finest tiles.  Stages marked (A) run
// for every problem still iterating (state active); (W) ones only for
// problems with a right-hand side still extending its Krylov space in the
// current GMRES cycle (for the refinement method W = A).
enum {
    F_BNORM = 0,   // (A) partial sums of b^2
    F_ZEROX,       // (A) x = 0 for right-hand sides with b = 0
    F_RESID,       // (A) r = b - A x in FP64 -> cycle input (T), cycle output = 0; partial sums of r^2
    F_UPDATE,      // (A) x += cycle output (refinement)
    F_MB,          // (A) cycle input = b, output = 0 (for ||M b||)
    F_CONVZ,       // (W) Z = cycle output in FP64; partial sums of Z^2
    F_MATVEC,      // (W) cycle input = A V_j, output = 0
    F_PROJ,        // (W) partial sums of <Z, V_i>, i <= j (pass 0 also <Z, Z>) -> part2
    F_PAXPY,       // (W) Z -= sum_i hsum_i V_i, i <= j; partial sums of Z^2
    F_SCALEV,      // (W) V_j = Z / ||Z||
    F_XUPD,        // (A) x += sum_k y_k V_k (left) or sum_k y_k Z_k (right)
    F_VTOB,        // (W) right: cycle input = V_j, output = 0
    F_AZ           // (W) right: Z_j = cycle output (kept), Z = A Z_j in FP64
};

__device__ __forceinline__ bool fine_gate_all(int what) {
    return what == F_BNORM || what == F_ZEROX || what == F_RESID || what == F_UPDATE || what == F_MB ||
           what == F_XUPD;
}
__device__ __forceinline__ bool fine_reduces(int what) {
    return what == F_BNORM || what == F_RESID || what == F_CONVZ;
}

template <typename T>
__device__ void stage_fine(const BArgs &a, const BProb<T> *P, int what, int iarg, int jarg, double *red) {
    const bool gate_all = fine_gate_all(what), reduces = fine_reduces(what);
    for (int k = blockIdx.x; k < a.nftiles; k += gridDim.x) {
        const BTile tile = a.ftiles[k];
        const int p = tile.p;
        // uniform over the CTA: the flags change only in the per-problem stages
        if (gate_all ? __ldcg(a.state + p) != ST_ACTIVE : __ldcg(a.work + p) == 0) continue;
        const BProb<T> &pr = P[p];
        const BLevel<T> L = pr.lev[0];
        const int m = pr.m, nx = L.nx, ny = L.ny;
        const int64_t N = L.N, nm = N * m;
        const TileMap tm = tile_map(m);
        const int r = tm.r, q = p * BMAXRHS + r;
        const int i0 = tile.i0, ni = tile.ni, n0 = tm.n0, step = tm.step;
        const double *__restrict__ b = a.b64[p];
        double *__restrict__ x = a.x64[p];
        T *__restrict__ Z = pr.Z;
        const T *__restrict__ V = pr.V;
        T *__restrict__ lb = L.b;
        T *__restrict__ lx = L.x;
        if (what == F_PROJ) {
            // projections of Z on V_0..V_j (pass 0 adds <Z, Z> as slot j + 1),
            // four slots per sweep over the tile's items; products summed in
            // T over up to KCH items, those partial sums in FP64
            const int nsl = iarg == 0 ? jarg + 2 : jarg + 1;
            const bool on = tm.on && (iarg == 0 ? !a.frozen[q] : a.reorth[q] != 0);
            double *dst = a.part2 + a.p2off[p] + (int64_t)(k - a.ftile_of[p]) * (a.restart + 2) * m;
            for (int s0 = 0; s0 < nsl; s0 += 4) {
                double pacc[4] = {0.0, 0.0, 0.0, 0.0};
                const T *__restrict__ vs[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int i = s0 + u;
                    vs[u] = i <= jarg ? V + (int64_t)i * nm : Z;
                }
                const int nv = min(4, nsl - s0);
                if (on)
                    for (int nn = n0; nn < ni;) {
                        T c[4] = {T(0), T(0), T(0), T(0)};
                        int t = 0;
                        for (; t + 2 <= KCH && nn + step < ni; t += 2, nn += 2 * step) {  // 10 loads in flight
                            T z[2], v[2][4];
#pragma unroll
                            for (int w = 0; w < 2; ++w) {
                                const int64_t e = (int64_t)(i0 + nn + w * step) * m + r;
                                z[w] = Z[e];
#pragma unroll
                                for (int u = 0; u < 4; ++u) v[w][u] = u < nv ? vs[u][e] : T(0);
                            }
#pragma unroll
                            for (int w = 0; w < 2; ++w)
#pragma unroll
                                for (int u = 0; u < 4; ++u) c[u] = fma(z[w], v[w][u], c[u]);
                        }
                        for (; t < KCH && nn < ni; ++t, nn += step) {
                            const int64_t e = (int64_t)(i0 + nn) * m + r;
                            const T z = Z[e];
#pragma unroll
                            for (int u = 0; u < 4; ++u)
                                if (u < nv) c[u] = fma(z, vs[u][e], c[u]);
                        }
#pragma unroll
                        for (int u = 0; u < 4; ++u) pacc[u] += (double)c[u];
                    }
                cta_sum4_by_rhs(pacc, nv, m, red, dst + (int64_t)s0 * m, m);
            }
            continue;
        }
        if (what == F_PAXPY) {
            // Z -= sum_i h_i V_i in T (the coefficients staged in shared
            // memory as T, in chunks of slots that fit the reduction buffer:
            // one chunk up to restart 64 with 32 RHS), ||Z||^2 as in F_PROJ;
            // pass iarg: 0 -> every extending right-hand side, 1 -> those
            // reprojected
            T *hs = reinterpret_cast<T *>(red);
            const int cap = (int)((sizeof(double) * RED_DOUBLES) / sizeof(T)) / m;  // slots per chunk
            const bool act = tm.on && (iarg == 0 ? !a.frozen[q] : a.reorth[q] != 0);
            double acc = 0.0;
            for (int s0 = 0; s0 <= jarg; s0 += cap) {
                const int s1 = min(jarg + 1, s0 + cap);
                const bool last = s1 == jarg + 1;
                for (int t = threadIdx.x; t < (s1 - s0) * m; t += blockDim.x) {
                    const int i = t / m, rr = t - i * m;
                    hs[t] = (T)a.hsum[(int64_t)(p * BMAXRHS + rr) * (a.restart + 2) + s0 + i];
                }
                __syncthreads();
                if (act) {
                    for (int nn = n0; nn < ni;) {
                        T c = T(0);
                        for (int t = 0; t < KCH && nn < ni; ++t, nn += step) {
                            const int64_t e = (int64_t)(i0 + nn) * m + r;
                            T z = Z[e];
#pragma unroll 4
                            for (int i = s0; i < s1; ++i) z = fma(-hs[(i - s0) * m + r], V[(int64_t)i * nm + e], z);
                            Z[e] = z;
                            if (last) c = fma(z, z, c);
                        }
                        acc += (double)c;
                    }
                }
                __syncthreads();  // hs aliases the reduction buffer
            }
            cta_sum_by_rhs(acc, m, red, a.part + (int64_t)k * BMAXRHS);
            continue;
        }
        double acc = 0.0;
        if (tm.on) {
            if (what == F_BNORM) {
                for (int nn = n0; nn < ni; nn += step) {
                    const double v = b[(int64_t)(i0 + nn) * m + r];
                    acc = fma(v, v, acc);
                }
            } else if (what == F_ZEROX) {
                if (a.nb[q] == 0.0)
                    for (int nn = n0; nn < ni; nn += step) x[(int64_t)(i0 + nn) * m + r] = 0.0;
            } else if (what == F_RESID) {
                // the true residual: FP64 operator and arithmetic
                const double *__restrict__ A64 = pr.A64;
                const bool star = L.kind == STAR;
                for (int nn = n0; nn < ni; nn += step) {
                    const int i = i0 + nn;
                    const int iy = i / nx, ix = i - iy * nx;
                    const double ax = star ? row_apply<STAR, double, double>(nx, ny, N, A64, x, m, r, ix, iy, i)
                                           : row_apply<BOX, double, double>(nx, ny, N, A64, x, m, r, ix, iy, i);
                    const int64_t e = (int64_t)i * m + r;
                    const double v = b[e] - ax;
                    acc = fma(v, v, acc);
                    lb[e] = (T)v;
                    lx[e] = T(0);
                    if (a.method == CS_GMRES_RIGHT) Z[e] = (T)v;  // V_0 = r / ||r|| next
                }
            } else if (what == F_AZ) {
                // right preconditioning: keep Z_j = M V_j (the cycle output,
                // exact in T) and form the Krylov product A Z_j with the FP64
                // operator, as F_MATVEC does for the left form
                T *__restrict__ zj = pr.ZB + (int64_t)jarg * nm;
                const double *__restrict__ A64 = pr.A64;
                const bool star = L.kind == STAR;
                for (int nn = n0; nn < ni; nn += step) {
                    const int i = i0 + nn;
                    const int iy = i / nx, ix = i - iy * nx;
                    const double ax = star ? row_apply<STAR, double, double, T>(nx, ny, N, A64, lx, m, r, ix, iy, i)
                                           : row_apply<BOX, double, double, T>(nx, ny, N, A64, lx, m, r, ix, iy, i);
                    const int64_t e = (int64_t)i * m + r;
                    zj[e] = lx[e];
                    Z[e] = (T)ax;
                }
            } else if (what == F_VTOB) {
                const T *__restrict__ vj = V + (int64_t)jarg * nm;
                for (int nn = n0; nn < ni; nn += step) {
                    const int64_t e = (int64_t)(i0 + nn) * m + r;
                    lb[e] = vj[e];
                    lx[e] = T(0);
                }
            } else if (what == F_MATVEC) {
                // the Krylov product A V_j: the FP64 operator applied in FP64
                // to the basis vector's (exact) values.  The cycles' rounded
                // operator would perturb it by about u |A| |V_j|, which the
                // preconditioner amplifies by the operator's (Skeel)
                // condition number: too much for high-contrast coefficients.
                const T *__restrict__ vj = V + (int64_t)jarg * nm;
                const double *__restrict__ A64 = pr.A64;
                const bool star = L.kind == STAR;
                for (int nn = n0; nn < ni; nn += step) {
                    const int i = i0 + nn;
                    const int iy = i / nx, ix = i - iy * nx;
                    const double ax = star ? row_apply<STAR, double, double, T>(nx, ny, N, A64, vj, m, r, ix, iy, i)
                                           : row_apply<BOX, double, double, T>(nx, ny, N, A64, vj, m, r, ix, iy, i);
                    const int64_t e = (int64_t)i * m + r;
                    lb[e] = (T)ax;
                    lx[e] = T(0);
                }
            } else if (what == F_UPDATE) {
                for (int nn = n0; nn < ni; nn += step) {
                    const int64_t e = (int64_t)(i0 + nn) * m + r;
                    x[e] += (double)lx[e];
                }
            } else if (what == F_MB) {
                for (int nn = n0; nn < ni; nn += step) {
                    const int64_t e = (int64_t)(i0 + nn) * m + r;
                    lb[e] = (T)b[e];
                    lx[e] = T(0);
                }
            } else if (what == F_CONVZ) {
                for (int nn = n0; nn < ni;) {
                    T c = T(0);
                    for (int t = 0; t < KCH && nn < ni; ++t, nn += step) {
                        const int64_t e = (int64_t)(i0 + nn) * m + r;
                        const T z = lx[e];
                        Z[e] = z;
                        c = fma(z, z, c);
                    }
                    acc += (double)c;
                }
            } else if (what == F_SCALEV) {
                if (!a.frozen[q] || jarg == 0) {
                    T *__restrict__ Vj = pr.V + (int64_t)jarg * nm;
                    const T inv = (T)a.inv[q];
                    for (int nn = n0; nn < ni; nn += step) {
                        const int64_t e = (int64_t)(i0 + nn) * m + r;
                        Vj[e] = Z[e] * inv;
                    }
                }
            } else {  // F_XUPD: x += V y (left) or Z y (right) in FP64 (y can combine with heavy cancellation)
                const int nc = a.jcols[q];
                const double *__restrict__ y = a.y + (int64_t)q * a.restart;
                const T *__restrict__ basis = a.method == CS_GMRES_RIGHT ? pr.ZB : V;
                for (int nn = n0; nn < ni; nn += step) {
                    const int64_t e = (int64_t)(i0 + nn) * m + r;
                    double sx = x[e];
                    for (int kk = 0; kk < nc; ++kk) sx = fma(y[kk], (double)basis[(int64_t)kk * nm + e], sx);
                    x[e] = sx;
                }
            }
        }
        if (reduces) cta_sum_by_rhs(acc, m, red, a.part + (int64_t)k * BMAXRHS);
    }
}

// Per-problem stages (one warp per problem, a right-hand side per lane): they
// sum the problem's tile partials and advance the small per-right-hand-side
// state.  One lane taking the right-hand sides in turn, through global memory,
// made the rotations of a step 76 us with 8 right-hand sides, 23 here.  Stages that count write ctl->cnt[ph] and clear
// ctl->cnt[ph ^ 1] (read before the barriers that precede this stage).
enum {
    P_NORMB = 0,  // ||b||
    P_NORM,       // true relative residuals: convergence, divergence, limit; counts active problems
    P_NMB,        // ||M b|| (GMRES stopping estimate scale)
    P_BETA,       // beta = ||M r|| (left) or ||r|| (right), g = beta e_1, V_0 scale; counts extending ones
    P_REORTH,     // ||Z||^2 after the first projection; reproject where it fell below half <Z, Z>; counts them
    P_GIVENS,     // H(j+1, j) = ||Z||, rotations, g, freeze; counts extending right-hand sides
    P_SOLVEY      // y = H^{-1} g (back substitution over the columns built)
};

template <typename T>
__device__ void stage_prob(const BArgs &a, const BProb<T> *P, int what, int iarg, int jarg, int ph, bool first,
                           double *wsum) {
    const int gid = blockIdx.x * blockDim.x + threadIdx.x;
    if ((what == P_NORM || what == P_BETA || what == P_GIVENS || what == P_REORTH) && gid == 0)
        a.ctl->cnt[ph ^ 1] = 0;
    const int R = a.restart;
    const int lane = threadIdx.x & 31;
    double *ws = wsum + (threadIdx.x >> 5) * BMAXRHS;
    const bool sums = what != P_SOLVEY;
    // the lanes sum the problem's tile partials (lane l takes tiles k0 + l,
    // k0 + l + 32, ...; fixed shuffle tree)
    for (int p = gid >> 5; p < a.nprob; p += (gridDim.x * blockDim.x) >> 5) {
        if (a.state[p] != ST_ACTIVE) continue;  // warp-uniform
        if ((what == P_REORTH || what == P_GIVENS) && !a.work[p]) continue;
        const int m = P[p].m;
        const int q0 = p * BMAXRHS;
        if (sums) {
            const int k0 = a.ftile_of[p], k1 = a.ftile_of[p + 1];
#pragma unroll 4
            for (int r = 0; r < m; ++r) {
                double v = 0.0;
                for (int k = k0 + lane; k < k1; k += 32) v += __ldcg(a.part + (int64_t)k * BMAXRHS + r);
                for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
                if (lane == 0) ws[r] = v;
            }
        }
        __syncwarp();
        // a right-hand side per lane; the problem's own state after a vote
        const int r = lane, q = q0 + r;
        const bool mine = lane < m;
        const double ss = sums && mine ? ws[r] : 0.0;
        if (what == P_NORMB || what == P_NMB) {
            double *dst = what == P_NORMB ? a.nb : a.nmb;
            if (mine) {
                dst[q] = sqrt(ss);
                if (what == P_NORMB && a.method == CS_GMRES_RIGHT) a.nmb[q] = sqrt(ss);  // right: the test is on ||r|| / ||b||
            }
        } else if (what == P_NORM) {
            double rel = 0.0;
            if (mine) {
                const double nb = a.nb[q];
                rel = nb > 0.0 ? sqrt(ss) / nb : 0.0;
                a.rel[q] = rel;
            }
            const bool conv = __all_sync(0xffffffffu, rel <= a.ctl->tol);
            const bool bad = __any_sync(0xffffffffu, !isfinite(rel));
            double worst = fmax(rel, 0.0);  // a NaN counts in `bad`, as fmax drops it
            for (int o = 16; o > 0; o >>= 1) worst = fmax(worst, __shfl_xor_sync(0xffffffffu, worst, o));
            if (lane == 0) {
                if (first) a.rel0[p] = worst;
                if (!first && a.method == CS_REFINE) a.iters[p] += 1;
                int st = ST_ACTIVE;
                if (conv) st = ST_CONVERGED;
                else if (bad || (a.method == CS_REFINE && worst > 1e3 * fmax(a.rel0[p], 1.0))) st = ST_DIVERGED;
                else if (a.iters[p] >= a.ctl->maxit) st = ST_MAXIT;
                a.state[p] = st;
                a.work[p] = st == ST_ACTIVE;
                if (st == ST_ACTIVE) atomicAdd(&a.ctl->cnt[ph], 1);
            }
        } else if (what == P_BETA) {
            bool ext = false;
            if (mine) {
                const double beta = sqrt(ss);
                a.g[(int64_t)q * (R + 1)] = beta;
                a.beta[q] = beta;
                a.inv[q] = beta > 0.0 ? 1.0 / sqrt(ss) : 0.0;
                a.jcols[q] = 0;
                ext = beta > 0.0 && a.iters[p] < a.ctl->maxit;
                a.frozen[q] = !ext;
            }
            const int n = __popc(__ballot_sync(0xffffffffu, ext));
            if (lane == 0) {
                a.work[p] = n > 0;
                if (n) atomicAdd(&a.ctl->cnt[ph], n);
            }
        } else if (what == P_REORTH) {
            // DGKS criterion: a second projection when ||Z - V h|| < ||Z|| / sqrt(2)
            bool re = false;
            if (mine) {
                if (!a.frozen[q]) {
                    a.znorm2[q] = ss;
                    re = ss < 0.5 * a.hsum[(int64_t)q * (R + 2) + jarg + 1];
                }
                a.reorth[q] = re;
            }
            const int n = __popc(__ballot_sync(0xffffffffu, re));
            if (lane == 0 && n) atomicAdd(&a.ctl->cnt[ph], n);
        } else if (what == P_GIVENS) {
            const int j = jarg;
            const int it = a.iters[p] + 1;
            const bool limit = it >= a.ctl->maxit;
            bool ext = false;
            if (mine && !a.frozen[q]) {
                double *H = a.H + (int64_t)q * a.hstride;
                double *cs = a.cs + (int64_t)q * R, *sn = a.sn + (int64_t)q * R, *g = a.g + (int64_t)q * (R + 1);
                const double zz = a.reorth[q] ? ss : a.znorm2[q];  // ||Z||^2 after the last projection
                const double hn = sqrt(zz);
                a.inv[q] = hn > 0.0 ? 1.0 / sqrt(zz) : 0.0;
                // the column through the earlier rotations: one value is carried, the loads run ahead
                double x0 = H[j];
#pragma unroll 8
                for (int i = 0; i < j; ++i) {
                    const double x1 = H[(i + 1) * R + j], c = cs[i], sv = sn[i];
                    H[i * R + j] = c * x0 + sv * x1;
                    x0 = -sv * x0 + c * x1;
                }
                const double d = sqrt(x0 * x0 + hn * hn);
                const double cj = d > 0 ? x0 / d : 1.0, sj = d > 0 ? hn / d : 0.0, gj = g[j];
                cs[j] = cj;
                sn[j] = sj;
                H[j * R + j] = d;
                H[(j + 1) * R + j] = 0.0;
                g[j + 1] = -sj * gj;
                g[j] = cj * gj;
                a.jcols[q] = j + 1;
                const double est = fabs(-sj * gj);
                if (est <= a.ctl->tol * a.nmb[q] || est <= a.itol * a.beta[q] || hn == 0.0 || limit || j + 1 >= R)
                    a.frozen[q] = 1;
                else ext = true;
            }
            const int n = __popc(__ballot_sync(0xffffffffu, ext));
            __syncwarp();
            if (lane == 0) {
                a.iters[p] = it;
                a.work[p] = n > 0;
                if (n) atomicAdd(&a.ctl->cnt[ph], n);
            }
        } else if (mine) {  // P_SOLVEY
            const double *H = a.H + (int64_t)q * a.hstride, *g = a.g + (int64_t)q * (R + 1);
            double *y = a.y + (int64_t)q * R;
            const int nc = a.jcols[q];
            for (int i = nc - 1; i >= 0; --i) {
                double sum = g[i];
#pragma unroll 4
                for (int k = i + 1; k < nc; ++k) sum -= H[i * R + k] * y[k];
                y[i] = sum / H[i * R + i];
            }
        }
        __syncwarp();  // ws is reused for the warp's next problem
    }
}

// Sums of the projection partials over each problem's tiles, one warp per
// (slot i, right-hand side): hsum_i = <Z, V_i> (pass 0 also slot j + 1 =
// <Z, Z>); H(i, j) takes the first pass's value and adds the second's.
template <typename T>
__device__ void stage_hsum(const BArgs &a, const BProb<T> *P, int j, int pass) {
    const int R = a.restart, nsl = pass == 0 ? j + 2 : j + 1;
    const int lane = threadIdx.x & 31;
    const int64_t nitems = (int64_t)nsl * a.qtot;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; w < nitems; w += nwarps) {
        const int qi = (int)(w % a.qtot), i = (int)(w / a.qtot);
        const int q = a.qlist[qi], p = q / BMAXRHS, r = q - p * BMAXRHS;
        // warp-uniform gates (flags written before the preceding barrier)
        if (__ldcg(a.state + p) != ST_ACTIVE || __ldcg(a.work + p) == 0) continue;
        if (pass == 0 ? __ldcg(a.frozen + q) != 0 : __ldcg(a.reorth + q) == 0) continue;
        const int m = P[p].m;
        const int k0 = a.ftile_of[p], k1 = a.ftile_of[p + 1];
        const int64_t ts = (int64_t)(R + 2) * m;
        const double *src = a.part2 + a.p2off[p] + (int64_t)i * m + r;
        double v = 0.0;
        for (int k = k0 + lane; k < k1; k += 32) v += __ldcg(src + (int64_t)(k - k0) * ts);
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) {
            a.hsum[(int64_t)q * (R + 2) + i] = v;
            if (i <= j) {
                double *h = a.H + (int64_t)q * a.hstride + i * R + j;
                *h = pass == 0 ? v : *h + v;
            }
        }
    }
}

// A grid-wide barrier between stages; the code names the stage it closes
// (1000 + 100 op + slot: cycle stages, 2000 + F_*: fine stages, 3000 + P_*:
// per-problem stages, 4000 + pass: projection sums, 5000: loop tests).
#define BSYNC(code) grid.sync()

template <typename T>
__device__ __forceinline__ void vcycle_stages(const BArgs &a, const BProb<T> *P, cg::grid_group &grid,
                                              Cache<T> &cache) {
    cache_flags<T>(a, cache);
    for (int s = 0; s < a.nsteps; ++s) {
        stage_step<T>(a, P, s, cache);
        if (s == a.tail_lo && a.tail_hi > a.tail_lo) s = a.tail_hi - 1;
        BSYNC(1000 + 100 * a.steps[s].op + a.steps[s].slot);
    }
}

// The whole solve: every CTA runs every stage and passes every grid barrier
// (no early exit anywhere).  Each loop ends for all CTAs at once: the count
// it tests was written before the barrier that precedes the test, and the
// counting stage that clears it again runs only after at least one more
// barrier (or only when the count is zero); every loop is bounded by the
// iteration limit in any case.
template <typename T>
__global__ void __launch_bounds__(512, sizeof(T) == 4 ? 2 : 1) k_batch_solve(BArgs a) {
    cg::grid_group grid = cg::this_grid();
    __shared__ double red[RED_DOUBLES];
    __shared__ double wsum[16 * BMAXRHS];
    __shared__ Cache<T> cache;
    const BProb<T> *P = static_cast<const BProb<T> *>(a.probs);
    cache_tiles<T>(a, P, cache);
    const int maxit = a.ctl->maxit;
    // counting stages write ctl->cnt[ph] after flipping ph and clear the other
    // slot; the loop tests read the slot written last
    int ph = 0;
    stage_fine<T>(a, P, F_BNORM, 0, 0, red);
    BSYNC(2000 + F_BNORM);
    stage_prob<T>(a, P, P_NORMB, 0, 0, ph, true, wsum);
    BSYNC(3000 + P_NORMB);
    stage_fine<T>(a, P, F_ZEROX, 0, 0, red);
    BSYNC(2000 + F_ZEROX);
    const bool gmres = a.method == CS_GMRES || a.method == CS_GMRES_RIGHT;
    const bool right = a.method == CS_GMRES_RIGHT;
    if (a.method == CS_GMRES) {  // ||M b|| per right-hand side
        stage_fine<T>(a, P, F_MB, 0, 0, red);
        BSYNC(2000 + F_MB);
        vcycle_stages<T>(a, P, grid, cache);
        stage_fine<T>(a, P, F_CONVZ, 0, 0, red);
        BSYNC(2000 + F_CONVZ);
        stage_prob<T>(a, P, P_NMB, 0, 0, ph, true, wsum);
        BSYNC(3000 + P_NMB);
    }
    stage_fine<T>(a, P, F_RESID, 0, 0, red);
    BSYNC(2000 + F_RESID);
    ph ^= 1;
    stage_prob<T>(a, P, P_NORM, 0, 0, ph, true, wsum);
    BSYNC(3000 + P_NORM);
    if (!gmres) {
        for (int it = 0; it < maxit; ++it) {
            if (__ldcg(&a.ctl->cnt[ph]) == 0) break;  // active problems
            vcycle_stages<T>(a, P, grid, cache);
            stage_fine<T>(a, P, F_UPDATE, 0, 0, red);
            BSYNC(2000 + F_UPDATE);
            stage_fine<T>(a, P, F_RESID, 0, 0, red);
            BSYNC(2000 + F_RESID);
            ph ^= 1;
            stage_prob<T>(a, P, P_NORM, 0, 0, ph, false, wsum);
            BSYNC(3000 + P_NORM);
        }
        return;
    }
    const int R = a.restart;
    for (int cyc = 0; cyc <= maxit; ++cyc) {
        if (__ldcg(&a.ctl->cnt[ph]) == 0) break;  // active problems
        if (!right) {
            vcycle_stages<T>(a, P, grid, cache);  // M r (the cycle input is r from F_RESID)
            stage_fine<T>(a, P, F_CONVZ, 0, 0, red);
            BSYNC(2000 + F_CONVZ);
        } else {
            // right: Z = r and the partial sums of r^2 come from F_RESID.  P_BETA
            // clears the count slot every CTA has just tested; the barrier keeps
            // a fast CTA from clearing it before a slow one has read it
            BSYNC(5000);
        }
        ph ^= 1;
        stage_prob<T>(a, P, P_BETA, 0, 0, ph, false, wsum);
        BSYNC(3000 + P_BETA);
        stage_fine<T>(a, P, F_SCALEV, 0, 0, red);
        BSYNC(2000 + F_SCALEV);
        for (int j = 0; j < R; ++j) {
            if (__ldcg(&a.ctl->cnt[ph]) == 0) break;  // right-hand sides still extending
            if (right) {  // Z = A M V_j, M V_j kept
                stage_fine<T>(a, P, F_VTOB, 0, j, red);
                BSYNC(2000 + F_VTOB);
                vcycle_stages<T>(a, P, grid, cache);
                stage_fine<T>(a, P, F_AZ, 0, j, red);
                BSYNC(2000 + F_AZ);
            } else {  // Z = M A V_j
                stage_fine<T>(a, P, F_MATVEC, 0, j, red);
                BSYNC(2000 + F_MATVEC);
                vcycle_stages<T>(a, P, grid, cache);
                stage_fine<T>(a, P, F_CONVZ, 0, 0, red);
                BSYNC(2000 + F_CONVZ);
            }
            // classical Gram-Schmidt with a second projection where the
            // first cancelled more than half of ||Z|| (DGKS)
            stage_fine<T>(a, P, F_PROJ, 0, j, red);
            BSYNC(2000 + F_PROJ);
            stage_hsum<T>(a, P, j, 0);
            BSYNC(4000);
            stage_fine<T>(a, P, F_PAXPY, 0, j, red);
            BSYNC(2000 + F_PAXPY);
            ph ^= 1;
            stage_prob<T>(a, P, P_REORTH, 0, j, ph, false, wsum);
            BSYNC(3000 + P_REORTH);
            if (__ldcg(&a.ctl->cnt[ph]) != 0) {  // right-hand sides projected again
                stage_fine<T>(a, P, F_PROJ, 1, j, red);
                BSYNC(2000 + F_PROJ);
                stage_hsum<T>(a, P, j, 1);
                BSYNC(4001);
                stage_fine<T>(a, P, F_PAXPY, 1, j, red);
                BSYNC(2000 + F_PAXPY);
            }
            ph ^= 1;
            stage_prob<T>(a, P, P_GIVENS, 0, j, ph, false, wsum);
            BSYNC(3000 + P_GIVENS);
            stage_fine<T>(a, P, F_SCALEV, 0, j + 1, red);
            BSYNC(2000 + F_SCALEV);
        }
        // every problem still active solves its small systems and updates x
        // (work flags may have cleared: these stages are gated on the state)
        stage_prob<T>(a, P, P_SOLVEY, 0, 0, ph, false, wsum);
        BSYNC(3000 + P_SOLVEY);
        stage_fine<T>(a, P, F_XUPD, 0, 0, red);
        BSYNC(2000 + F_XUPD);
        stage_fine<T>(a, P, F_RESID, 0, 0, red);
        BSYNC(2000 + F_RESID);
        ph ^= 1;
        stage_prob<T>(a, P, P_NORM, 0, 0, ph, false, wsum);
        BSYNC(3000 + P_NORM);
    }
}

}  // namespace csx

using namespace csx;


struct cs_batch {
    int nprob = 0, dmax = 0, precision = CS_FP32, order = CS_RF, mu_pre = 1, mu_post = 1, nu = 1;
    int kind = CS_MULTIPLICATIVE, bs = 1;
    int dev = 0;
    std::vector<int> m, nlev, slot0;
    std::vector<int64_t> nfine;
    std::vector<std::vector<int>> nx, ny;  // per problem per level
    void *probs = nullptr;
    size_t probs_bytes = 0;
    std::vector<unsigned char> hprobs;
    void *vec = nullptr;  // all multi-RHS level vectors
    BTile *tiles = nullptr, *ftiles = nullptr, *btiles = nullptr;
    int *slot_btile = nullptr;
    int *slot_tile = nullptr, *ftile_of = nullptr;
    int ntiles = 0, nftiles = 0;
    BStep *steps = nullptr;
    int nsteps = 0;
    std::vector<BStep> hsteps;
    BTail *tails = nullptr;
    int ntails = 0, tail_lo = 0, tail_hi = 0;
    double *part = nullptr, *nb = nullptr, *rel = nullptr, *rel0 = nullptr;
    int *state = nullptr, *iters = nullptr, *work = nullptr;
    BCtl *ctl = nullptr;
    int method = CS_REFINE, restart = 0;
    void *gm = nullptr;   // GMRES basis and work vectors of all problems
    void *gsm = nullptr;  // GMRES per-right-hand-side small state
    double *H = nullptr, *gcs = nullptr, *gsn = nullptr, *gy = nullptr, *gg = nullptr, *ginv = nullptr,
           *gnmb = nullptr;
    int *jcols = nullptr, *frozen = nullptr;
    double *part2 = nullptr, *hsum = nullptr, *znorm2 = nullptr, *gbeta = nullptr;
    int64_t *p2off = nullptr;
    int *qlist = nullptr, *reorth = nullptr;
    int qtot = 0;
    const double **bptr = nullptr;
    double **xptr = nullptr;
    // pinned host staging
    void *hstage = nullptr;
    size_t hstage_bytes = 0;
    int threads = 256, tiles_per_cta = 2, ctas = 0;
    std::vector<cs_batch_tune> tuned;
    cudaGraphExec_t graph = nullptr;
    bool graph_ok = true;
    double *tune_b = nullptr, *tune_x = nullptr;
    int64_t bytes = 0;
};

namespace {

template <typename T>
void *kernel_ptr() {
    return reinterpret_cast<void *>(&k_batch_solve<T>);
}

void *kernel_of(const cs_batch *B) {
    return B->precision == CS_FP32 ? kernel_ptr<float>() : kernel_ptr<double>();
}

// Work tiles of about equal work (grid nodes x right-hand sides): every
// slot's items, the finest levels' items and (block cascades) every slot's
// block items are cut into about tiles_per_cta x CTAs tiles, but no tile
// holds fewer items than a CTA has threads.  A problem's tiles are ranges of
// its own nodes (or blocks), so a tile's node count is its item share over
// the problem's right-hand side count.  Few large tiles per CTA keep each
// stage's serial chain of tile start-up latencies short; equal work per tile
// keeps the CTAs arriving at the stage barrier together.
cs_status build_tiles(cs_batch *B, int tiles_per_cta, cudaStream_t s) {
    const int64_t want = std::max<int64_t>(1, (int64_t)B->ctas * tiles_per_cta);
    auto tile_items = [&](int64_t items) { return std::max<int64_t>(B->threads, (items + want - 1) / want); };
    auto cut = [](std::vector<BTile> &out, int p, int l, int64_t n, int64_t per) {
        for (int64_t i0 = 0; i0 < n; i0 += per) out.push_back({p, l, (int)i0, (int)std::min<int64_t>(per, n - i0)});
    };
    std::vector<BTile> tl;
    std::vector<int> st(B->dmax + 1, 0);
    for (int t = 0; t < B->dmax; ++t) {
        st[t] = (int)tl.size();
        int64_t items = 0;
        for (int p = 0; p < B->nprob; ++p) {
            const int l = t - B->slot0[p];
            if (l >= 0) items += (int64_t)B->nx[p][l] * B->ny[p][l] * B->m[p];
        }
        const int64_t ti = tile_items(items);
        for (int p = 0; p < B->nprob; ++p) {
            const int l = t - B->slot0[p];
            if (l < 0) continue;
            cut(tl, p, l, (int64_t)B->nx[p][l] * B->ny[p][l], (ti + B->m[p] - 1) / B->m[p]);
        }
    }
    st[B->dmax] = (int)tl.size();
    std::vector<BTile> ft;
    std::vector<int> fo(B->nprob + 1, 0);
    {
        int64_t items = 0;
        for (int p = 0; p < B->nprob; ++p) items += B->nfine[p] * B->m[p];
        const int64_t ti = tile_items(items);
        for (int p = 0; p < B->nprob; ++p) {
            fo[p] = (int)ft.size();
            cut(ft, p, 0, B->nfine[p], (ti + B->m[p] - 1) / B->m[p]);
        }
    }
    fo[B->nprob] = (int)ft.size();
    // block tiles (block-level sweeps: one item per block and right-hand side)
    std::vector<BTile> bt;
    std::vector<int> sb(B->dmax + 1, 0);
    if (B->bs > 1) {
        auto nblk = [&](int p, int l) {
            return (int64_t)((B->nx[p][l] + B->bs - 1) / B->bs) * ((B->ny[p][l] + B->bs - 1) / B->bs);
        };
        for (int t = 0; t < B->dmax; ++t) {
            sb[t] = (int)bt.size();
            int64_t items = 0;
            for (int p = 0; p < B->nprob; ++p) {
                const int l = t - B->slot0[p];
                if (l >= 0) items += nblk(p, l) * B->m[p];
            }
            const int64_t ti = tile_items(items);
            for (int p = 0; p < B->nprob; ++p) {
                const int l = t - B->slot0[p];
                if (l < 0) continue;
                cut(bt, p, l, nblk(p, l), (ti + B->m[p] - 1) / B->m[p]);
            }
        }
        sb[B->dmax] = (int)bt.size();
    }
    // The tail slot: the first slot from which on an item of the tail, one CTA,
    // holds at most tail_n values of a level.  A stage over all CTAs costs its
    // barrier and a tile's start, the tail the steps of its values one after the
    // other: nine per thread of 256 are worth it with a CTA for every right-hand
    // side, half as many per thread in smaller CTAs, of which an SM holds more.
    // With more right-hand sides than CTAs an item takes all of a problem's, all
    // CTAs are busy, and the line is at twice that.  FP64, at 1/64 of the FP32
    // rate: half.  FP32 cycles on 48^2 with 256 threads went from 201 to 153 us
    // (1 right-hand side) and from 301 to 283 (16 problems with 8); with tails up
    // to 65^2, whatever the threads, 16 problems of 65^2 went from 320 to 432 us
    // (now 269), and from 378 to 1183 with 128 threads (now 339).
    std::vector<BTail> tails;
    {
        int64_t q = 0;
        for (int p = 0; p < B->nprob; ++p) q += B->m[p];
        const bool each = q <= B->ctas;
        const int64_t tail_n =
            9 * (B->threads < 256 ? B->threads / 2 : 256) * (each ? 1 : 2) / (B->precision == CS_FP32 ? 1 : 2);
        int ts = B->dmax;
        for (int t = B->dmax - 1; t >= 0; --t) {
            int64_t mx = 0;
            for (int p = 0; p < B->nprob; ++p) {
                const int l = t - B->slot0[p];
                if (l >= 0) mx = std::max(mx, (int64_t)B->nx[p][l] * B->ny[p][l] * (each ? 1 : B->m[p]));
            }
            if (mx > tail_n) break;
            ts = t;
        }
        int lo = 0;
        while (lo < B->nsteps && B->hsteps[lo].slot < ts) ++lo;
        int hi = lo;
        while (hi < B->nsteps && B->hsteps[hi].slot >= ts) ++hi;
        B->tail_lo = lo;
        B->tail_hi = hi;
        for (int p = 0; p < B->nprob; ++p)
            for (int r = 0; r < B->m[p]; r += each ? 1 : B->m[p]) tails.push_back({p, r, each ? 1 : B->m[p]});
        // the items with the most work first: they start in the first round
        std::stable_sort(tails.begin(), tails.end(), [&](const BTail &u, const BTail &v) {
            return B->nfine[u.p] * u.rc > B->nfine[v.p] * v.rc;
        });
        B->ntails = (int)tails.size();
    }
    // a captured graph holds the old table pointers
    if (B->graph) {
        cudaGraphExecDestroy(B->graph);
        B->graph = nullptr;
    }
    dfree(B->tiles, s); dfree(B->ftiles, s); dfree(B->slot_tile, s); dfree(B->ftile_of, s); dfree(B->part, s);
    dfree(B->btiles, s); dfree(B->slot_btile, s); dfree(B->part2, s); dfree(B->p2off, s); dfree(B->tails, s);
    B->tails = nullptr;
    B->tiles = nullptr; B->ftiles = nullptr; B->slot_tile = nullptr; B->ftile_of = nullptr; B->part = nullptr;
    B->btiles = nullptr; B->slot_btile = nullptr; B->part2 = nullptr; B->p2off = nullptr;
    if (B->method != CS_REFINE) {  // projection partials: (restart + 2) slots x m_p per finest tile
        std::vector<int64_t> po(B->nprob + 1, 0);
        for (int p = 0; p < B->nprob; ++p)
            po[p + 1] = po[p] + (int64_t)(fo[p + 1] - fo[p]) * (B->restart + 2) * B->m[p];
        CSX_TRY(dalloc_t(&B->p2off, po.size(), nullptr, s));
        CSX_TRY(dalloc_t(&B->part2, (size_t)std::max<int64_t>(1, po[B->nprob]), nullptr, s));
        CSX_CUDA(cudaMemcpyAsync(B->p2off, po.data(), po.size() * sizeof(int64_t), cudaMemcpyHostToDevice, s));
        CSX_CUDA(cudaStreamSynchronize(s));
    }
    if (B->bs > 1) {
        CSX_TRY(dalloc_t(&B->btiles, bt.size(), nullptr, s));
        CSX_TRY(dalloc_t(&B->slot_btile, sb.size(), nullptr, s));
        CSX_CUDA(cudaMemcpyAsync(B->btiles, bt.data(), bt.size() * sizeof(BTile), cudaMemcpyHostToDevice, s));
        CSX_CUDA(cudaMemcpyAsync(B->slot_btile, sb.data(), sb.size() * sizeof(int), cudaMemcpyHostToDevice, s));
    }
    CSX_TRY(dalloc_t(&B->tails, tails.size(), nullptr, s));
    CSX_CUDA(cudaMemcpyAsync(B->tails, tails.data(), tails.size() * sizeof(BTail), cudaMemcpyHostToDevice, s));
    CSX_TRY(dalloc_t(&B->tiles, tl.size(), nullptr, s));
    CSX_TRY(dalloc_t(&B->ftiles, ft.size(), nullptr, s));
    CSX_TRY(dalloc_t(&B->slot_tile, st.size(), nullptr, s));
    CSX_TRY(dalloc_t(&B->ftile_of, fo.size(), nullptr, s));
    CSX_TRY(dalloc_t(&B->part, ft.size() * BMAXRHS, nullptr, s));
    CSX_CUDA(cudaMemcpyAsync(B->tiles, tl.data(), tl.size() * sizeof(BTile), cudaMemcpyHostToDevice, s));
    CSX_CUDA(cudaMemcpyAsync(B->ftiles, ft.data(), ft.size() * sizeof(BTile), cudaMemcpyHostToDevice, s));
    CSX_CUDA(cudaMemcpyAsync(B->slot_tile, st.data(), st.size() * sizeof(int), cudaMemcpyHostToDevice, s));
    CSX_CUDA(cudaMemcpyAsync(B->ftile_of, fo.data(), fo.size() * sizeof(int), cudaMemcpyHostToDevice, s));
    CSX_CUDA(cudaStreamSynchronize(s));  // the host vectors go out of scope
    B->ntiles = (int)tl.size();
    B->nftiles = (int)ft.size();
    B->tiles_per_cta = tiles_per_cta;
    return CS_OK;
}

BArgs args_of(const cs_batch *B) {
    BArgs a;
    a.probs = B->probs;
    a.nprob = B->nprob;
    a.tiles = B->tiles;
    a.slot_tile = B->slot_tile;
    a.btiles = B->btiles;
    a.slot_btile = B->slot_btile;
    a.dmax = B->dmax;
    a.ftiles = B->ftiles;
    a.ftile_of = B->ftile_of;
    a.nftiles = B->nftiles;
    a.steps = B->steps;
    a.nsteps = B->nsteps;
    a.tails = B->tails;
    a.ntails = B->ntails;
    a.tail_lo = B->tail_lo;
    a.tail_hi = B->tail_hi;
    a.b64 = B->bptr;
    a.x64 = B->xptr;
    a.part = B->part;
    a.nb = B->nb;
    a.rel = B->rel;
    a.rel0 = B->rel0;
    a.state = B->state;
    a.iters = B->iters;
    a.work = B->work;
    a.ctl = B->ctl;
    a.method = B->method;
    a.restart = B->restart;
    a.hstride = (B->restart + 1) * B->restart;
    a.H = B->H;
    a.cs = B->gcs;
    a.sn = B->gsn;
    a.y = B->gy;
    a.g = B->gg;
    a.inv = B->ginv;
    a.nmb = B->gnmb;
    a.jcols = B->jcols;
    a.frozen = B->frozen;
    a.part2 = B->part2;
    a.p2off = B->p2off;
    a.qtot = B->qtot;
    a.qlist = B->qlist;
    a.hsum = B->hsum;
    a.znorm2 = B->znorm2;
    a.reorth = B->reorth;
    a.beta = B->gbeta;
    // FP32 Krylov vectors resolve about 1e-6 of ||M r||: a GMRES cycle stops
    // at 1e-5 and the restart's FP64 residual refines (GMRES-IR)
    a.itol = B->precision == CS_FP32 ? 1e-5 : 0.0;
    return a;
}

// CTAs that can be co-resident (a cooperative launch needs all of them)
cs_status coresident(const cs_batch *B, int threads, int *ctas) {
    int nsm = 0, per = 0;
    CSX_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, B->dev));
    CSX_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel_of(B), threads, 0));
    if (per < 1) {
        set_error("batched solve kernel cannot run %d threads per CTA", threads);
        return CS_ERR_UNSUPPORTED;
    }
    *ctas = per * nsm;
    return CS_OK;
}

cs_status launch(cs_batch *B, cudaStream_t s) {
    BArgs a = args_of(B);
    void *params[] = {&a};
    CSX_CUDA(cudaLaunchCooperativeKernel(kernel_of(B), dim3((unsigned)B->ctas), dim3((unsigned)B->threads), params, 0,
                                         s));
    count_launch();
    return CS_OK;
}

// per-solve control: tolerance, iteration limit, zeroed counters and states
cs_status reset_control(cs_batch *B, double tol, int maxit, cudaStream_t s) {
    BCtl c;
    c.tol = tol;
    c.maxit = maxit;
    c.cnt[0] = c.cnt[1] = 0;
    std::memcpy(B->hstage, &c, sizeof(c));
    CSX_CUDA(cudaMemcpyAsync(B->ctl, B->hstage, sizeof(c), cudaMemcpyHostToDevice, s));
    CSX_CUDA(cudaMemsetAsync(B->state, 0, sizeof(int) * B->nprob, s));
    CSX_CUDA(cudaMemsetAsync(B->iters, 0, sizeof(int) * B->nprob, s));
    CSX_CUDA(cudaMemsetAsync(B->work, 1, sizeof(int) * B->nprob, s));  // nonzero: every problem takes part
    return CS_OK;
}

cs_status set_pointers(cs_batch *B, const double *const *b, double *const *x, cudaStream_t s) {
    char *h = static_cast<char *>(B->hstage) + 64;
    std::memcpy(h, b, sizeof(double *) * B->nprob);
    std::memcpy(h + sizeof(double *) * B->nprob, x, sizeof(double *) * B->nprob);
    CSX_CUDA(cudaMemcpyAsync(B->bptr, h, sizeof(double *) * B->nprob, cudaMemcpyHostToDevice, s));
    CSX_CUDA(cudaMemcpyAsync(B->xptr, h + sizeof(double *) * B->nprob, sizeof(double *) * B->nprob,
                             cudaMemcpyHostToDevice, s));
    return CS_OK;
}

// the kernel, captured once per configuration into a graph; if capturing a
// cooperative launch is refused, it is launched directly
cs_status run(cs_batch *B, cudaStream_t s) {
    if (!B->graph && B->graph_ok) {
        cudaStream_t cs = nullptr;
        CSX_CUDA(cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking));
        cudaGraph_t g = nullptr;
        cudaError_t e = cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal);
        if (e == cudaSuccess) {
            BArgs a = args_of(B);
            void *params[] = {&a};
            cudaError_t le = cudaLaunchCooperativeKernel(kernel_of(B), dim3((unsigned)B->ctas),
                                                         dim3((unsigned)B->threads), params, 0, cs);
            e = cudaStreamEndCapture(cs, &g);
            if (le != cudaSuccess) e = le;
        }
        if (e == cudaSuccess) e = cudaGraphInstantiate(&B->graph, g, 0);
        if (g) cudaGraphDestroy(g);
        cudaStreamDestroy(cs);
        if (e != cudaSuccess) {
            (void)cudaGetLastError();
            B->graph = nullptr;
            B->graph_ok = false;
        }
    }
    if (B->graph) {
        CSX_CUDA(cudaGraphLaunch(B->graph, s));
        count_launch();
        return CS_OK;
    }
    return launch(B, s);
}

void build_steps(const cs_batch *B, std::vector<BStep> &out) {
    // The buffer holding a level's iterate is the same for every problem at a
    // slot: multiplicative steps come in colour pairs that end in x; additive
    // steps flip between x and t, and the prolongation writes the buffer from
    // which the post-smoothing steps end in x (the single-problem rule).
    const bool rf = B->order == CS_RF, mult = B->kind == CS_MULTIPLICATIVE;
    std::vector<int> pre_cur(B->dmax, 0);
    for (int t = 0; t + 1 < B->dmax; ++t) {
        int cur = 0;
        for (int mu = 0; mu < B->mu_pre; ++mu)
            for (int step = 0; step < B->nu; ++step) {
                const int lv = rf ? B->nu - 1 - step : step;
                if (mult) {
                    for (int kk = 0; kk < 2; ++kk) out.push_back({OP_SWEEP, t, lv, rf ? 1 - kk : kk, kk, 0, 0, rf});
                } else {
                    out.push_back({OP_SWEEP, t, lv, -1, 0, cur, 1 - cur, rf});
                    cur ^= 1;
                }
            }
        // the buffer without the iterate is free until the prolongation
        out.push_back({OP_FRES, t, 0, 0, 0, cur, 1 - cur, 0});
        out.push_back({OP_RESTRICT, t, 0, 0, 0, 1 - cur, 0, 0});
        pre_cur[t] = cur;
    }
    out.push_back({OP_COARSE, B->dmax - 1, 0, 0, 0, 0, 0, 0});
    const int post_flips = mult ? 0 : B->mu_post * B->nu;
    for (int t = B->dmax - 2; t >= 0; --t) {
        int cur = post_flips % 2 == 0 ? 0 : 1;
        out.push_back({OP_PROLONG, t, 0, 0, 0, pre_cur[t], cur, 0});
        for (int mu = 0; mu < B->mu_post; ++mu)
            for (int step = 0; step < B->nu; ++step) {
                if (mult) {
                    for (int kk = 0; kk < 2; ++kk) out.push_back({OP_SWEEP, t, step, kk, kk, 0, 0, 0});
                } else {
                    out.push_back({OP_SWEEP, t, step, -1, 0, cur, 1 - cur, 0});
                    cur ^= 1;
                }
            }
    }
}

template <typename T>
cs_status fill_probs(cs_batch *B, cs_hierarchy *const *h, cs_cascade *const *c, T *vec, T *gm) {
    B->probs_bytes = sizeof(BProb<T>) * B->nprob;
    B->hprobs.assign(B->probs_bytes, 0);
    BProb<T> *hp = reinterpret_cast<BProb<T> *>(B->hprobs.data());
    T *v = vec;
    for (int p = 0; p < B->nprob; ++p) {
        BProb<T> &q = hp[p];
        q.nlev = h[p]->nlev;
        q.m = B->m[p];
        q.slot0 = B->slot0[p];
        q.cn = h[p]->cn;
        q.A64 = h[p]->lev[0].A;
        q.cinv = h[p]->cinv;
        q.Z = nullptr;
        q.V = nullptr;
        q.ZB = nullptr;
        if (gm) {
            const int64_t n0 = h[p]->lev[0].g.N * B->m[p];
            q.Z = gm;
            q.V = gm + n0;
            gm += (int64_t)(B->restart + 2) * n0;
            if (B->method == CS_GMRES_RIGHT) {
                q.ZB = gm;
                gm += (int64_t)B->restart * n0;
            }
        }
        for (int l = 0; l < q.nlev; ++l) {
            const Level &L = h[p]->lev[l];
            BLevel<T> &d = q.lev[l];
            d.nx = L.g.nx;
            d.ny = L.g.ny;
            d.kind = L.kind;
            // red-black (of nodes or of blocks) is a graph colouring of the 5-point stencil only
            d.inplace = B->kind == CS_MULTIPLICATIVE && L.kind == STAR ? 1 : 0;
            d.N = L.g.N;
            d.bs = L.bs;
            d.nbx = L.nbx;
            d.nmax = L.nmax;
            d.nblocks = L.nblocks;
            if (sizeof(T) == sizeof(float)) {
                d.A = reinterpret_cast<const T *>(c[p]->lo[l].A);
                d.lam = l < c[p]->nlev ? reinterpret_cast<const T *>(c[p]->lo[l].lam) : nullptr;
            } else {
                d.A = reinterpret_cast<const T *>(L.A);
                d.lam = l < c[p]->nlev ? reinterpret_cast<const T *>(c[p]->lam[l]) : nullptr;
            }
            const int64_t n = L.g.N * q.m;
            d.b = v; v += n;
            d.x = v; v += n;
            d.t = v; v += n;
        }
    }
    return CS_OK;
}

}  // namespace

extern "C" {

cs_status cs_batch_create(int nprob, cs_hierarchy *const *h, cs_cascade *const *c, const int *nrhs,
                          const cs_batch_opts *o, cs_stream stream, cs_batch **out) {
    if (!out || !h || !c || !nrhs || !o || nprob < 1) { set_error("null argument or empty batch"); return CS_ERR_ARG; }
    *out = nullptr;
    if (o->precision != CS_FP32 && o->precision != CS_FP64) { set_error("bad precision"); return CS_ERR_ARG; }
    if (o->order != CS_RF && o->order != CS_FF) { set_error("bad order"); return CS_ERR_ARG; }
    if (o->method != CS_REFINE && o->method != CS_GMRES && o->method != CS_GMRES_RIGHT) {
        set_error("batched method must be CS_REFINE, CS_GMRES or CS_GMRES_RIGHT");
        return CS_ERR_ARG;
    }
    if (o->method != CS_REFINE && (o->restart < 0 || o->restart > BMAXRESTART)) {
        set_error("GMRES restart must be in 1..%d", BMAXRESTART);
        return CS_ERR_ARG;
    }
    if (o->mu_pre < 0 || o->mu_post < 0 || o->mu_pre + o->mu_post < 1 || o->mu_pre > 16 || o->mu_post > 16) {
        set_error("bad smoothing counts");
        return CS_ERR_ARG;
    }
    int nu = -1;
    for (int p = 0; p < nprob; ++p) {
        const cs_hierarchy *hp = h[p];
        const cs_cascade *cp = c[p];
        if (!hp || !cp || cp->h != hp) { set_error("problem %d: missing or mismatched handles", p); return CS_ERR_ARG; }
        if (nrhs[p] < 1 || nrhs[p] > BMAXRHS) { set_error("problem %d: nrhs must be in 1..%d", p, BMAXRHS); return CS_ERR_ARG; }
        if (hp->dim != 2 || hp->periodic) { set_error("problem %d: the batched solver takes 2D Dirichlet grids", p); return CS_ERR_UNSUPPORTED; }
        if (cp->kind != c[0]->kind) { set_error("all problems of a batch need the same cascade kind"); return CS_ERR_ARG; }
        if (hp->nlev < 2 || hp->nlev > BMAXLEV || !hp->cinv) { set_error("problem %d: need 2..%d levels and a coarsest factorisation", p, BMAXLEV); return CS_ERR_UNSUPPORTED; }
        for (int l = 0; l < hp->nlev; ++l)
            if (hp->lev[l].bs != h[0]->lev[0].bs) { set_error("all problems of a batch need the same block size"); return CS_ERR_ARG; }
        if (hp->lev[0].bs > 2) { set_error("problem %d: the batched solver takes point blocks or 2x2-node blocks", p); return CS_ERR_UNSUPPORTED; }
        if (o->precision == CS_FP32 && !cp->lowp) { set_error("problem %d: FP32 cycles need a cascade built with lowp", p); return CS_ERR_ARG; }
        if (nu < 0) nu = cp->nu;
        if (cp->nu != nu) { set_error("all problems of a batch need the same cascade depth"); return CS_ERR_ARG; }
    }
    cudaStream_t s = (cudaStream_t)stream;
    cs_batch *B = new cs_batch();
    cs_status rc = CS_OK;
    B->nprob = nprob;
    B->precision = o->precision;
    B->order = o->order;
    B->mu_pre = o->mu_pre;
    B->mu_post = o->mu_post;
    B->nu = nu;
    B->kind = c[0]->kind;
    B->bs = h[0]->lev[0].bs;
    B->method = o->method;
    B->restart = o->restart > 0 ? o->restart : 30;
    cudaGetDevice(&B->dev);
    B->m.assign(nrhs, nrhs + nprob);
    B->nlev.resize(nprob);
    B->slot0.resize(nprob);
    B->nfine.resize(nprob);
    B->nx.resize(nprob);
    B->ny.resize(nprob);
    int64_t nvec = 0;
    for (int p = 0; p < nprob; ++p) {
        B->nlev[p] = h[p]->nlev;
        B->dmax = std::max(B->dmax, h[p]->nlev);
        B->nfine[p] = h[p]->lev[0].g.N;
        for (int l = 0; l < h[p]->nlev; ++l) {
            B->nx[p].push_back(h[p]->lev[l].g.nx);
            B->ny[p].push_back(h[p]->lev[l].g.ny);
            nvec += 3 * h[p]->lev[l].g.N * nrhs[p];
        }
    }
    for (int p = 0; p < nprob; ++p) B->slot0[p] = B->dmax - B->nlev[p];
    const size_t esz = o->precision == CS_FP32 ? sizeof(float) : sizeof(double);
    std::vector<BStep> steps;
    build_steps(B, steps);
    B->nsteps = (int)steps.size();
    B->hsteps = steps;
    int64_t nfine_rhs = 0;
    for (int p = 0; p < nprob; ++p) nfine_rhs += B->nfine[p] * B->m[p];
    if ((rc = dalloc(&B->vec, (size_t)nvec * esz, &B->bytes, s)) != CS_OK) goto fail;
    if (B->method != CS_REFINE) {
        // basis (restart + 1 vectors) and Z per problem, in the cycle precision, [N0][m] each;
        // right preconditioning keeps restart more (Z_j = M V_j)
        const size_t nv = (size_t)(B->restart + 2) + (B->method == CS_GMRES_RIGHT ? (size_t)B->restart : 0);
        if ((rc = dalloc(&B->gm, nv * nfine_rhs * esz, &B->bytes, s)) != CS_OK)
            goto fail;
        const size_t nq = (size_t)nprob * BMAXRHS, R = (size_t)B->restart;
        const size_t nd = nq * ((R + 1) * R + 3 * R + (R + 1) + 2 + (R + 2) + 2);
        if ((rc = dalloc(&B->gsm, nd * sizeof(double) + 3 * nq * sizeof(int), &B->bytes, s)) != CS_OK) goto fail;
        double *d = static_cast<double *>(B->gsm);
        B->H = d; d += nq * (R + 1) * R;
        B->gcs = d; d += nq * R;
        B->gsn = d; d += nq * R;
        B->gy = d; d += nq * R;
        B->gg = d; d += nq * (R + 1);
        B->ginv = d; d += nq;
        B->gnmb = d; d += nq;
        B->hsum = d; d += nq * (R + 2);
        B->znorm2 = d; d += nq;
        B->gbeta = d; d += nq;
        B->jcols = reinterpret_cast<int *>(d);
        B->frozen = B->jcols + nq;
        B->reorth = B->frozen + nq;
        // every right-hand side of every problem, for the projection sums
        std::vector<int> ql;
        for (int p = 0; p < nprob; ++p)
            for (int r = 0; r < B->m[p]; ++r) ql.push_back(p * BMAXRHS + r);
        B->qtot = (int)ql.size();
        if ((rc = dalloc_t(&B->qlist, ql.size(), &B->bytes, s)) != CS_OK) goto fail;
        if (cudaMemcpyAsync(B->qlist, ql.data(), ql.size() * sizeof(int), cudaMemcpyHostToDevice, s) != cudaSuccess ||
            cudaStreamSynchronize(s) != cudaSuccess) {
            rc = cuda_fail(cudaGetLastError(), "batch create", __FILE__, __LINE__);
            goto fail;
        }
    }
    if (o->precision == CS_FP32)
        rc = fill_probs<float>(B, h, c, static_cast<float *>(B->vec), static_cast<float *>(B->gm));
    else rc = fill_probs<double>(B, h, c, static_cast<double *>(B->vec), static_cast<double *>(B->gm));
    if (rc != CS_OK) goto fail;
    if ((rc = dalloc(&B->probs, B->probs_bytes, &B->bytes, s)) != CS_OK) goto fail;
    if ((rc = dalloc_t(&B->steps, steps.size(), &B->bytes, s)) != CS_OK) goto fail;
    if ((rc = dalloc_t(&B->nb, (size_t)nprob * BMAXRHS, &B->bytes, s)) != CS_OK) goto fail;
    if ((rc = dalloc_t(&B->rel, (size_t)nprob * BMAXRHS, &B->bytes, s)) != CS_OK) goto fail;
    if ((rc = dalloc_t(&B->rel0, (size_t)nprob, &B->bytes, s)) != CS_OK) goto fail;
    if ((rc = dalloc_t(&B->state, (size_t)nprob, &B->bytes, s)) != CS_OK) goto fail;
    if ((rc = dalloc_t(&B->iters, (size_t)nprob, &B->bytes, s)) != CS_OK) goto fail;
    if ((rc = dalloc_t(&B->work, (size_t)nprob, &B->bytes, s)) != CS_OK) goto fail;
    if ((rc = dalloc_t(&B->ctl, 1, &B->bytes, s)) != CS_OK) goto fail;
    if ((rc = dalloc_t(&B->bptr, (size_t)nprob, &B->bytes, s)) != CS_OK) goto fail;
    if ((rc = dalloc_t(&B->xptr, (size_t)nprob, &B->bytes, s)) != CS_OK) goto fail;
    B->hstage_bytes = 64 + 2 * sizeof(double *) * nprob + sizeof(double) * nprob * (BMAXRHS + 1) + sizeof(int) * 2 * nprob;
    {
        cudaError_t e = cudaMallocHost(&B->hstage, B->hstage_bytes);
        if (e == cudaSuccess)
            e = cudaMemcpyAsync(B->probs, B->hprobs.data(), B->probs_bytes, cudaMemcpyHostToDevice, s);
        if (e == cudaSuccess)
            e = cudaMemcpyAsync(B->steps, steps.data(), steps.size() * sizeof(BStep), cudaMemcpyHostToDevice, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) { rc = cuda_fail(e, "batch create", __FILE__, __LINE__); goto fail; }
    }
    {
        int threads = o->threads > 0 ? o->threads : 256;
        int tile = o->tiles_per_cta > 0 ? o->tiles_per_cta : 2;
        if (o->autotune) {
            // time each candidate on the batch itself: two cycles from x = 0
            // with b = 1 (tol 0: exactly two iterations), best of three
            if ((rc = dalloc_t(&B->tune_b, (size_t)nfine_rhs, nullptr, s)) != CS_OK) goto fail;
            if ((rc = dalloc_t(&B->tune_x, (size_t)nfine_rhs, nullptr, s)) != CS_OK) goto fail;
            std::vector<double> ones((size_t)std::min<int64_t>(nfine_rhs, 1 << 20), 1.0);
            for (int64_t o0 = 0; o0 < nfine_rhs; o0 += (int64_t)ones.size()) {
                const int64_t n = std::min<int64_t>((int64_t)ones.size(), nfine_rhs - o0);
                if (cudaMemcpyAsync(B->tune_b + o0, ones.data(), n * sizeof(double), cudaMemcpyHostToDevice, s) !=
                    cudaSuccess) {
                    rc = cuda_fail(cudaGetLastError(), "autotune input", __FILE__, __LINE__);
                    goto fail;
                }
            }
            std::vector<const double *> bp(nprob);
            std::vector<double *> xp(nprob);
            int64_t off = 0;
            for (int p = 0; p < nprob; ++p) {
                bp[p] = B->tune_b + off;
                xp[p] = B->tune_x + off;
                off += B->nfine[p] * B->m[p];
            }
            const int cand_threads[] = {128, 256, 512};
            const int cand_tile[] = {1, 2, 4};
            float best = 1e30f;
            cudaEvent_t e0, e1;
            cudaEventCreate(&e0);
            cudaEventCreate(&e1);
            for (int ct : cand_threads)
                for (int tt : cand_tile) {
                    int ctas = 0;
                    if (coresident(B, ct, &ctas) != CS_OK) continue;
                    B->threads = ct;
                    B->ctas = ctas;
                    if ((rc = build_tiles(B, tt, s)) != CS_OK) break;
                    float ms_best = 1e30f;
                    for (int rep = 0; rep < 3 && rc == CS_OK; ++rep) {
                        if (cudaMemsetAsync(B->tune_x, 0, sizeof(double) * nfine_rhs, s) != cudaSuccess) {
                            rc = cuda_fail(cudaGetLastError(), "autotune", __FILE__, __LINE__);
                            break;
                        }
                        if ((rc = set_pointers(B, bp.data(), xp.data(), s)) != CS_OK) break;
                        if ((rc = reset_control(B, 0.0, 2, s)) != CS_OK) break;
                        cudaEventRecord(e0, s);
                        if ((rc = launch(B, s)) != CS_OK) break;
                        cudaEventRecord(e1, s);
                        if (cudaEventSynchronize(e1) != cudaSuccess) {
                            rc = cuda_fail(cudaGetLastError(), "autotune", __FILE__, __LINE__);
                            break;
                        }
                        float ms = 0.f;
                        cudaEventElapsedTime(&ms, e0, e1);
                        ms_best = std::min(ms_best, ms);
                    }
                    if (rc != CS_OK) break;
                    B->tuned.push_back({ct, tt, ms_best});
                    if (ms_best < best) {
                        best = ms_best;
                        threads = ct;
                        tile = tt;
                    }
                }
            cudaEventDestroy(e0);
            cudaEventDestroy(e1);
            dfree(B->tune_b, s);
            dfree(B->tune_x, s);
            B->tune_b = B->tune_x = nullptr;
            if (rc != CS_OK) goto fail;
        }
        if ((rc = coresident(B, threads, &B->ctas)) != CS_OK) goto fail;
        B->threads = threads;
        if ((rc = build_tiles(B, tile, s)) != CS_OK) goto fail;
    }
    *out = B;
    return CS_OK;
fail:
    cs_batch_destroy(B);
    return rc;
}

cs_status cs_batch_solve(cs_batch *B, const double *const *b, double *const *x, double tol, int maxit,
                         cs_solve_info *info, cs_stream stream) {
    if (!B || !b || !x) { set_error("null argument"); return CS_ERR_ARG; }
    for (int p = 0; p < B->nprob; ++p)
        if (!b[p] || !x[p]) { set_error("problem %d: null vector", p); return CS_ERR_ARG; }
    if (tol <= 0) tol = 1e-10;
    if (maxit <= 0) maxit = 100;
    cudaStream_t s = (cudaStream_t)stream;
    CSX_TRY(set_pointers(B, b, x, s));
    CSX_TRY(reset_control(B, tol, maxit, s));
    CSX_TRY(run(B, s));
    const int np = B->nprob;
    char *h = static_cast<char *>(B->hstage) + 64 + 2 * sizeof(double *) * np;
    double *hrel = reinterpret_cast<double *>(h);
    int *hst = reinterpret_cast<int *>(hrel + (size_t)np * BMAXRHS);
    int *hit = hst + np;
    CSX_CUDA(cudaMemcpyAsync(hrel, B->rel, sizeof(double) * np * BMAXRHS, cudaMemcpyDeviceToHost, s));
    CSX_CUDA(cudaMemcpyAsync(hst, B->state, sizeof(int) * np, cudaMemcpyDeviceToHost, s));
    CSX_CUDA(cudaMemcpyAsync(hit, B->iters, sizeof(int) * np, cudaMemcpyDeviceToHost, s));
    CSX_CUDA(cudaStreamSynchronize(s));
    cs_status rc = CS_OK;
    int ndiv = 0, nnc = 0;
    for (int p = 0; p < np; ++p) {
        double worst = 0.0;
        for (int r = 0; r < B->m[p]; ++r) worst = std::max(worst, hrel[(size_t)p * BMAXRHS + r]);
        if (info) info[p] = {hit[p], hst[p] == ST_CONVERGED ? 1 : 0, worst, 0};
        if (hst[p] == ST_DIVERGED) ++ndiv;
        else if (hst[p] != ST_CONVERGED) ++nnc;
    }
    if (ndiv) {
        set_error("%d of %d problems diverged", ndiv, np);
        rc = CS_ERR_DIVERGED;
    } else if (nnc) {
        set_error("%d of %d problems not converged after %d iterations", nnc, np, maxit);
        rc = CS_ERR_NOTCONV;
    }
    return rc;
}

cs_status cs_batch_config(const cs_batch *B, int *threads, int *tiles_per_cta, int *ctas, cs_batch_tune *tuned,
                          int cap, int *ntuned) {
    if (!B) { set_error("null argument"); return CS_ERR_ARG; }
    if (threads) *threads = B->threads;
    if (tiles_per_cta) *tiles_per_cta = B->tiles_per_cta;
    if (ctas) *ctas = B->ctas;
    if (ntuned) *ntuned = (int)B->tuned.size();
    if (tuned)
        for (int k = 0; k < cap && k < (int)B->tuned.size(); ++k) tuned[k] = B->tuned[k];
    return CS_OK;
}

cs_status cs_batch_set_config(cs_batch *B, int threads, int tiles_per_cta, cs_stream stream) {
    if (!B || threads < 32 || threads > 512 || (threads & 31) || tiles_per_cta < 1 || tiles_per_cta > 1024) {
        set_error("bad batch configuration");
        return CS_ERR_ARG;
    }
    cudaStream_t s = (cudaStream_t)stream;
    int ctas = 0;
    CSX_TRY(coresident(B, threads, &ctas));
    B->threads = threads;
    B->ctas = ctas;
    CSX_TRY(build_tiles(B, tiles_per_cta, s));
    return CS_OK;
}

int64_t cs_batch_bytes(const cs_batch *B) { return B ? B->bytes : 0; }

void cs_batch_destroy(cs_batch *B) {
    if (!B) return;
    if (B->graph) cudaGraphExecDestroy(B->graph);
    dfree(B->vec); dfree(B->probs); dfree(B->tiles); dfree(B->ftiles); dfree(B->slot_tile); dfree(B->ftile_of);
    dfree(B->btiles); dfree(B->slot_btile);
    dfree(B->tails); dfree(B->steps); dfree(B->part); dfree(B->nb); dfree(B->rel); dfree(B->rel0); dfree(B->state); dfree(B->iters);
    dfree(B->ctl); dfree(B->bptr); dfree(B->xptr); dfree(B->tune_b); dfree(B->tune_x); dfree(B->work);
    dfree(B->gm); dfree(B->gsm); dfree(B->part2); dfree(B->p2off); dfree(B->qlist);
    if (B->hstage) cudaFreeHost(B->hstage);
    delete B;
}

cs_status cs_solve_batched(int nprob, cs_hierarchy *const *h, cs_cascade *const *c, const cs_solve_opts *o,
                           const double *const *b, double *const *x, const int *nrhs, cs_solve_info *info,
                           cs_stream stream) {
    if (!o) { set_error("null argument"); return CS_ERR_ARG; }
    cs_batch_opts bo{};
    bo.precision = o->cycle.precision;
    bo.order = o->cycle.order;
    bo.mu_pre = o->cycle.mu_pre;
    bo.mu_post = o->cycle.mu_post;
    bo.autotune = 0;
    bo.method = (o->method == CS_GMRES || o->method == CS_GMRES_RIGHT) ? o->method : CS_REFINE;
    bo.restart = o->restart;
    cs_batch *B = nullptr;
    CSX_TRY(cs_batch_create(nprob, h, c, nrhs, &bo, stream, &B));
    cs_status rc = cs_batch_solve(B, b, x, o->tol, o->maxit, info, stream);
    cs_batch_destroy(B);
    return rc;
}

}  // extern "C"
