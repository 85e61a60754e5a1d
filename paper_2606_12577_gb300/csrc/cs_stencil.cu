// Stencil kernels of the V-cycle: cascade sweeps (eq. fwda / fwdm and their
// reverse forms), the restricted residual and the interpolated correction of
// Algorithm 1, the bottom-level solve, and FP64 reductions.
//
// One thread per node; x fastest across a warp so that every coefficient
// array A[s][.] is streamed with coalesced loads, and the neighbour reads of
// x hit L1/L2.  These kernels are HBM-bound in FP32 (bytes per node per
// additive step: nst*sizeof(T) + 4*sizeof(T) for A, Lambda, b, x read, x
// written).
#include <algorithm>
#include <atomic>
#include <type_traits>
#include <cstdint>
#include <cstdio>

#include <cooperative_groups.h>
#include <cuda_bf16.h>

#include "cs_internal.cuh"

namespace csx {

// canonical stencil offsets -------------------------------------------------
template <int DIM, int KIND>
struct Sten {
    static constexpr int NST = KIND == STAR ? 2 * DIM + 1 : (DIM == 3 ? 27 : 9);
    static __host__ __device__ __forceinline__ void off(int s, int &dx, int &dy, int &dz) {
        if (KIND == STAR) {
            dx = dy = dz = 0;
            if (s == 1) dx = -1;
            else if (s == 2) dx = 1;
            else if (s == 3) dy = -1;
            else if (s == 4) dy = 1;
            else if (s == 5) dz = -1;
            else if (s == 6) dz = 1;
        } else {
            dx = s % 3 - 1;
            dy = (s / 3) % 3 - 1;
            dz = DIM == 3 ? s / 9 - 1 : 0;
        }
    }
};

// Arithmetic type of a storage type: FP64 and FP32 compute in their own
// type, BF16 storage computes in FP32 (FP32 accumulation).
template <typename T> struct AccT { using type = T; };
template <> struct AccT<__nv_bfloat16> { using type = float; };
template <typename T>
__device__ __forceinline__ typename AccT<T>::type ld(T v) { return v; }
template <>
__device__ __forceinline__ float ld<__nv_bfloat16>(__nv_bfloat16 v) { return __bfloat162float(v); }
template <typename T>
__device__ __forceinline__ T st(typename AccT<T>::type v) { return v; }
template <>
__device__ __forceinline__ __nv_bfloat16 st<__nv_bfloat16>(float v) { return __float2bfloat16_rn(v); }
template <typename T>
__device__ __forceinline__ T zero() { return st<T>(typename AccT<T>::type(0)); }

__device__ __forceinline__ int node_colour(int dim, int ix, int iy, int iz) {
    return ((ix + 1) + (iy + 1) + (dim == 3 ? iz + 1 : 0)) & 1;
}

// the coefficients of row i
template <int DIM, int KIND, typename T>
__device__ __forceinline__ void load_row(const Grid &g, const T *__restrict__ A, int64_t i, T *a) {
#pragma unroll
    for (int s = 0; s < Sten<DIM, KIND>::NST; ++s) a[s] = A[(int64_t)s * g.N + i];
}

// (A x)_i at node (ix,iy,iz) from the row's coefficients; neighbours outside
// the grid contribute nothing
template <int DIM, int KIND, typename T>
__device__ __forceinline__ typename AccT<T>::type apply_coeff(const Grid &g, const T *a, const T *x, int ix, int iy,
                                                              int iz, int64_t i) {
    using S = Sten<DIM, KIND>;
    using C = typename AccT<T>::type;
    C ax = C(0);
#pragma unroll
    for (int s = 0; s < S::NST; ++s) {
        int dx, dy, dz;
        S::off(s, dx, dy, dz);
        bool in = (unsigned)(ix + dx) < (unsigned)g.nx && (unsigned)(iy + dy) < (unsigned)g.ny &&
                  (DIM == 2 || (unsigned)(iz + dz) < (unsigned)g.nz);
        C xv = in ? ld<T>(x[i + dx + (int64_t)g.nx * (dy + (int64_t)g.ny * dz)]) : C(0);
        ax = fma(ld<T>(a[s]), xv, ax);
    }
    return ax;
}
template <int DIM, int KIND, typename T>
__device__ __forceinline__ typename AccT<T>::type apply_row(const Grid &g, const T *__restrict__ A, const T *x, int ix,
                                                            int iy, int iz, int64_t i) {
    T a[Sten<DIM, KIND>::NST];
    load_row<DIM, KIND, T>(g, A, i, a);
    return apply_coeff<DIM, KIND, T>(g, a, x, ix, iy, iz, i);
}

// ---- 3D 27-point levels with symmetric FP32 storage (Level::sym32):
// Af[k][i] holds entry 13 + k of row i (centre and forward couplings); the
// backward entry s < 13 of row i is the forward entry 26 - s of the
// neighbour j = i + off(s).  Same summation order as apply_row, so only the
// (mirrored) coefficient values can differ from the full copy's.
__device__ __forceinline__ void load_row_box_sym(const Grid &g, const float *__restrict__ Af, int ix, int iy, int iz,
                                                 int64_t i, float *a) {
#pragma unroll
    for (int s = 0; s < 27; ++s) {
        const int dx = s % 3 - 1, dy = (s / 3) % 3 - 1, dz = s / 9 - 1;
        const bool in = (unsigned)(ix + dx) < (unsigned)g.nx && (unsigned)(iy + dy) < (unsigned)g.ny &&
                        (unsigned)(iz + dz) < (unsigned)g.nz;
        a[s] = 0.f;
        if (s >= 13) a[s] = Af[(int64_t)(s - 13) * g.N + i];
        else if (in) a[s] = Af[(int64_t)(13 - s) * g.N + i + dx + (int64_t)g.nx * (dy + (int64_t)g.ny * dz)];
    }
}
// 7 points, symmetric (Level::symstar): the full layout, of which only the
// centre and the forward couplings (entries 0, 2, 4, 6) are read
__device__ __forceinline__ void load_row_star_sym(const Grid &g, const float *__restrict__ A, int ix, int iy, int iz,
                                                  int64_t i, float *a) {
    const int64_t N = g.N, sy = g.nx, sz = (int64_t)g.nx * g.ny;
    a[0] = A[i];
    a[2] = A[2 * N + i];
    a[4] = A[4 * N + i];
    a[6] = A[6 * N + i];
    a[1] = ix > 0 ? A[2 * N + i - 1] : 0.f;
    a[3] = iy > 0 ? A[4 * N + i - sy] : 0.f;
    a[5] = iz > 0 ? A[6 * N + i - sz] : 0.f;
}
template <int DIM, int KIND, typename T, bool SYM>
__device__ __forceinline__ void load_coeff(const Grid &g, const T *__restrict__ A, int ix, int iy, int iz, int64_t i,
                                           T *a) {
    if constexpr (SYM && KIND == STAR) load_row_star_sym(g, A, ix, iy, iz, i, a);
    else if constexpr (SYM) load_row_box_sym(g, A, ix, iy, iz, i, a);
    else load_row<DIM, KIND, T>(g, A, i, a);
}

// ---- repeated rows.  On an operator with constant coefficients almost every
// row is the grid-centre row, and deep rows hold the Lambda of their colour's
// representative (see the cascade setup); such rows take both from the
// kernel's parameters instead of reading nst + 1 values each.  Rows next to
// a face repeat the centre row too where they differ only in couplings to
// nodes outside the grid, whose value is zero.
template <typename T, int NST>
struct Rep {
    T a[NST];
    int lo[3], hi[3];    // box of the rows with coefficients a (empty: lo > hi)
    int dist, rep[2];    // rows at boundary distance >= dist hold lam[rep[colour]]
};
template <typename T, int NST>
__device__ __forceinline__ bool rep_row(const Rep<T, NST> &r, int ix, int iy, int iz) {
    return ix >= r.lo[0] && ix <= r.hi[0] && iy >= r.lo[1] && iy <= r.hi[1] && iz >= r.lo[2] && iz <= r.hi[2];
}
template <int DIM, typename T, int NST>
__device__ __forceinline__ bool rep_lam(const Grid &g, const Rep<T, NST> &r, int ix, int iy, int iz) {
    int d = min(min(ix, g.nx - 1 - ix), min(iy, g.ny - 1 - iy));
    if (DIM == 3) d = min(d, min(iz, g.nz - 1 - iz));
    return d >= r.dist;
}
template <typename T> static T from_double(double v) { return (T)v; }
template <> __nv_bfloat16 from_double<__nv_bfloat16>(double v) { return __double2bfloat16(v); }
template <typename T, int NST>
static Rep<T, NST> make_rep(const Level &L, const LamDeep *deep) {
    Rep<T, NST> r;
    const bool mirror = std::is_same<T, float>::value && L.sym32;  // as the symmetric copy stores them
    for (int s = 0; s < NST; ++s) r.a[s] = from_double<T>(L.cbox ? L.crow[mirror && s < 13 ? 26 - s : s] : 0.0);
    for (int d = 0; d < 3; ++d) {
        r.lo[d] = L.cbox ? L.clo[d] : 1;
        r.hi[d] = L.cbox ? L.chi[d] : 0;
    }
    r.dist = deep ? deep->dist : Level::NO_MARGIN;
    r.rep[0] = deep ? deep->rep[0] : 0;
    r.rep[1] = deep ? deep->rep[1] : 0;
    return r;
}

// Cascade step: out_i = x_i - lam_i ((A x)_i - b_i).
// COLOURED: only nodes of colour `colour`; the others keep x (copied when
// out != x, i.e. snapshot semantics for non-graph colourings).  A thread
// takes two x-adjacent nodes, of which one has the colour, so no lane idles.
// Otherwise every node (additive step, out != x).
// settled: A and lam may be read before the kernels ahead have finished.
template <int DIM, int KIND, typename T, bool COLOURED, bool SYM = false>
__global__ void __launch_bounds__(TBX *TBY) k_sweep(Grid g, const T *__restrict__ A, const T *__restrict__ lam,
                                                     const T *b, const T *x, T *out, int colour,
                                                     int xzero, int settled,
                                                     const __grid_constant__ Rep<T, Sten<DIM, KIND>::NST> rep) {
    constexpr int NST = Sten<DIM, KIND>::NST;
    using C = typename AccT<T>::type;
    pdl_trigger();
    if (!settled) pdl_wait();
    int ix = blockIdx.x * TBX + threadIdx.x;
    const int iy = blockIdx.y * TBY + threadIdx.y, iz = blockIdx.z;
    int ox = g.nx;  // the thread's node of the other colour
    if (COLOURED) {
        const int px = 2 * ix, par = node_colour(DIM, px, iy, iz) == colour ? 0 : 1;
        ix = px + par;
        ox = px + 1 - par;
    }
    const int64_t row = (int64_t)g.nx * (iy + (int64_t)g.ny * iz), i = ix + row;
    const bool in = ix < g.nx && iy < g.ny;
    T a[NST];
    C li = C(0);
    if (in) {
        if (!xzero) {
            if (rep_row(rep, ix, iy, iz)) {
#pragma unroll
                for (int s = 0; s < NST; ++s) a[s] = rep.a[s];
            } else {
                load_coeff<DIM, KIND, T, SYM>(g, A, ix, iy, iz, i, a);
            }
        }
        li = ld<T>(lam[rep_lam<DIM>(g, rep, ix, iy, iz) ? rep.rep[COLOURED ? colour : 0] : i]);
    }
    if (settled) pdl_wait();
    if (COLOURED && ox < g.nx && iy < g.ny) {
        if (xzero) out[ox + row] = zero<T>();
        else if (out != x) out[ox + row] = x[ox + row];
    }
    if (!in) return;
    C r;
    C xi;
    if (xzero) {
        r = -ld<T>(b[i]);
        xi = C(0);
    } else {
        r = apply_coeff<DIM, KIND, T>(g, a, x, ix, iy, iz, i) - ld<T>(b[i]);
        xi = ld<T>(x[i]);
    }
    out[i] = st<T>(xi - li * r);
}

// The neighbourhood of an (ix, iy) column of a 3D grid, plane by plane: v
// holds the stencil's values of x at the current node, in stencil order, and
// advancing one plane reads only the new plane's (9 values for 27 points, 5
// for 7).
template <int KIND, typename T>
struct Column {
    T v[Sten<3, KIND>::NST];
    T up[KIND == STAR ? 1 : 9];  // the plane above
    __device__ __forceinline__ void plane(const Grid &g, const T *x, int ix, int iy, int iz, int64_t i) {
#pragma unroll
        for (int s = 0; s < (KIND == STAR ? 1 : 9); ++s) {
            const int dx = KIND == STAR ? 0 : s % 3 - 1, dy = KIND == STAR ? 0 : s / 3 - 1;
            const bool in = (unsigned)(ix + dx) < (unsigned)g.nx && (unsigned)(iy + dy) < (unsigned)g.ny &&
                            (unsigned)iz < (unsigned)g.nz;
            up[s] = in ? x[i + dx + (int64_t)g.nx * dy] : T(0);
        }
    }
    // i: the node's index at plane iz
    __device__ __forceinline__ void start(const Grid &g, const T *x, int ix, int iy, int iz, int64_t i) {
        const int64_t pl = (int64_t)g.nx * g.ny;
        plane(g, x, ix, iy, iz - 1, i - pl);
        if (KIND == STAR) v[5] = up[0];
        else
#pragma unroll
            for (int s = 0; s < 9; ++s) v[s] = up[s];
        plane(g, x, ix, iy, iz, i);
        if (KIND == STAR) v[0] = up[0];
        else
#pragma unroll
            for (int s = 0; s < 9; ++s) v[9 + s] = up[s];
        plane(g, x, ix, iy, iz + 1, i + pl);
        top(g, x, ix, iy, iz, i);
    }
    __device__ __forceinline__ void top(const Grid &g, const T *x, int ix, int iy, int iz, int64_t i) {
        if (KIND == STAR) {
            v[1] = ix > 0 ? x[i - 1] : T(0);
            v[2] = ix + 1 < g.nx ? x[i + 1] : T(0);
            v[3] = iy > 0 ? x[i - g.nx] : T(0);
            v[4] = iy + 1 < g.ny ? x[i + g.nx] : T(0);
            v[6] = up[0];
        } else {
#pragma unroll
            for (int s = 0; s < 9; ++s) v[18 + s] = up[s];
        }
    }
    // to plane iz (index i), reading plane iz + 1
    __device__ __forceinline__ void advance(const Grid &g, const T *x, int ix, int iy, int iz, int64_t i) {
        if (KIND == STAR) {
            v[5] = v[0];
            v[0] = v[6];
        } else {
#pragma unroll
            for (int s = 0; s < 18; ++s) v[s] = v[s + 9];
        }
        plane(g, x, ix, iy, iz + 1, i + (int64_t)g.nx * g.ny);
        top(g, x, ix, iy, iz, i);
    }
    __device__ __forceinline__ T centre() const { return v[KIND == STAR ? 0 : 13]; }
    // sum over the stencil in its order
    __device__ __forceinline__ T apply(const T *a) const {
        T ax = T(0);
#pragma unroll
        for (int s = 0; s < Sten<3, KIND>::NST; ++s) ax = fma(a[s], v[s], ax);
        return ax;
    }
};

// Additive step (RES false) or residual out = A x - b (RES true) of a 3D
// level with a box of repeated rows, RZ planes per thread: in the box a node
// reads x, b and writes out only, 12 B in FP32 where the general kernel moves
// 44 (7 points) or 72 (27 points, symmetric copy), and the column of x values
// moves up in registers.  Rows outside the box read their coefficients.
// FP32 finest step on 256^3: 104.7 us reading every row, 66 us here and 46.6
// with quads (k_sweep_rep4; 201 MB, floor 30 us); 128^3 27-point step 42, 38
// and 25.6 us; FP64 127^3 red-black steps (k_sweep) 36.6 -> 20 us.
constexpr int RZ = 4;
constexpr int64_t RZ_MIN_N = 1 << 18;  // below, the planes' parallelism is worth more than the rereads
template <int KIND, bool RES, bool SYM>
__global__ void __launch_bounds__(TBX *TBY, KIND == STAR ? 6 : 3)
    k_sweep_rep(Grid g, const float *__restrict__ A, const float *__restrict__ lam, const float *b, const float *x,
                float *__restrict__ out, int settled, const __grid_constant__ Rep<float, Sten<3, KIND>::NST> rep) {
    constexpr int NST = Sten<3, KIND>::NST;
    pdl_trigger();
    if (!settled) pdl_wait();
    const int ix = blockIdx.x * TBX + threadIdx.x, iy = blockIdx.y * TBY + threadIdx.y, z0 = blockIdx.z * RZ;
    const float lrep = RES ? 0.f : lam[rep.dist == Level::NO_MARGIN ? 0 : rep.rep[0]];
    if (settled) pdl_wait();
    if (ix >= g.nx || iy >= g.ny) return;
    const int64_t pl = (int64_t)g.nx * g.ny;
    int64_t i = ix + (int64_t)g.nx * iy + pl * z0;
    Column<KIND, float> col;
    col.start(g, x, ix, iy, z0, i);
#pragma unroll
    for (int r = 0; r < RZ; ++r, i += pl) {
        const int iz = z0 + r;
        if (iz < g.nz) {
            if (r > 0) col.advance(g, x, ix, iy, iz, i);
            float ax;
            if (rep_row(rep, ix, iy, iz)) {
                ax = col.apply(rep.a);
            } else {
                float a[NST];
                load_coeff<3, KIND, float, SYM>(g, A, ix, iy, iz, i, a);
                ax = col.apply(a);
            }
            const float res = ax - b[i];
            if (RES) {
                out[i] = res;
            } else {
                const float li = rep_lam<3>(g, rep, ix, iy, iz) ? lrep : lam[i];
                out[i] = col.centre() - li * res;
            }
        }
    }
}

// The same in FP32 with four x-adjacent nodes per thread (nx a multiple of 4,
// 16-byte aligned vectors): rows of x, b and out move as float4 and a row's
// end values come from the neighbouring lanes, so a 27-point node costs 2.3
// load instructions instead of 11 and is bound by L2 / HBM rather than by
// issue and latency.  Threads take the quads of a plane in order, whatever
// its width.  Rows outside the box go to CTAs of their own behind the others
// (one node per thread, coefficients read), so no warp of the box waits for
// their loads.
template <int KIND, bool RES, bool SYM>
__global__ void __launch_bounds__(256) k_sweep_rep4(Grid g, const float *__restrict__ A, const float *__restrict__ lam,
                                                    const float *b, const float *x,
                                                    float *__restrict__ out, int settled, int nbox, RowSet shell,
                                                    const __grid_constant__ Rep<float, Sten<3, KIND>::NST> rep) {
    constexpr int NST = Sten<3, KIND>::NST;
    constexpr int NR = KIND == STAR ? 1 : 3;  // x rows per plane that the column keeps
    pdl_trigger();
    if (!settled) pdl_wait();
    if ((int)blockIdx.x >= nbox) {  // rows outside the box
        int ix, iy, iz;
        const int64_t t = (int64_t)((int)blockIdx.x - nbox) * 256 + threadIdx.x;
        const bool in = t < shell.nshell && rowset_coord(shell, g, t, ix, iy, iz);
        float a[NST], li = 0.f;
        int64_t i = 0;
        if (in) {
            i = ix + (int64_t)g.nx * (iy + (int64_t)g.ny * iz);
            load_coeff<3, KIND, float, SYM>(g, A, ix, iy, iz, i, a);
            if (!RES) li = lam[rep_lam<3>(g, rep, ix, iy, iz) ? rep.rep[0] : i];
        }
        if (settled) pdl_wait();
        if (!in) return;
        const float res = apply_coeff<3, KIND, float>(g, a, x, ix, iy, iz, i) - b[i];
        out[i] = RES ? res : x[i] - li * res;
        return;
    }
    const int nq = g.nx >> 2, per = nq * g.ny, lane = threadIdx.x & 31;
    const int ncta = (per + 255) >> 8;  // CTAs per slab of RZ planes
    const int slab = (int)blockIdx.x / ncta, t = ((int)blockIdx.x - slab * ncta) * 256 + threadIdx.x;
    const bool in = t < per;
    const int iy = in ? t / nq : 0, q = in ? t - iy * nq : 0, ix = 4 * q, z0 = slab * RZ;
    const float lrep = RES ? 0.f : lam[rep.dist == Level::NO_MARGIN ? 0 : rep.rep[0]];
    if (settled) pdl_wait();
    const int64_t pl = (int64_t)g.nx * g.ny;
    int64_t i = ix + (int64_t)g.nx * iy + pl * z0;
    auto row4 = [&](const float *p, bool ok) {
        return ok ? *reinterpret_cast<const float4 *>(p) : make_float4(0.f, 0.f, 0.f, 0.f);
    };
    // a row of six values around the quad: its left and right ends are the neighbouring lanes' values
    auto row6 = [&](const float *p, bool ok, float *w) {
        const float4 c = row4(p, ok);
        float l = __shfl_up_sync(0xffffffffu, c.w, 1), r = __shfl_down_sync(0xffffffffu, c.x, 1);
        if (lane == 0) l = ok && q > 0 ? p[-1] : 0.f;
        if (lane == 31) r = ok && q + 1 < nq ? p[4] : 0.f;
        w[0] = q > 0 ? l : 0.f;
        w[1] = c.x; w[2] = c.y; w[3] = c.z; w[4] = c.w;
        w[5] = q + 1 < nq ? r : 0.f;
    };
    float w[3][NR][6];  // planes below, at and above the current one
    auto plane = [&](int iz, int64_t j, float (*u)[6]) {
        const bool oz = in && (unsigned)iz < (unsigned)g.nz;
        if (KIND == STAR) {
            const float4 c = row4(x + j, oz);
            u[0][1] = c.x; u[0][2] = c.y; u[0][3] = c.z; u[0][4] = c.w;
        } else {
#pragma unroll
            for (int k = 0; k < 3; ++k) row6(x + j + (k - 1) * (int64_t)g.nx, oz && (unsigned)(iy + k - 1) < (unsigned)g.ny, u[k % NR]);
        }
    };
    plane(z0 - 1, i - pl, w[0]);
    plane(z0, i, w[1]);
#pragma unroll
    for (int r = 0; r < RZ; ++r, i += pl) {
        const int iz = z0 + r;
        if (iz >= g.nz) break;  // uniform over the CTA
        plane(iz + 1, i + pl, w[2]);
        const float4 bv = row4(b + i, in);
        float ax[4] = {0.f, 0.f, 0.f, 0.f}, xc[4];
        if (KIND == STAR) {
            const float4 ym = row4(x + i - g.nx, in && iy > 0), yp = row4(x + i + g.nx, in && iy + 1 < g.ny);
            float l = __shfl_up_sync(0xffffffffu, w[1][0][4], 1), rr = __shfl_down_sync(0xffffffffu, w[1][0][1], 1);
            if (lane == 0) l = in && q > 0 ? x[i - 1] : 0.f;
            if (lane == 31) rr = in && q + 1 < nq ? x[i + 4] : 0.f;
            w[1][0][0] = q > 0 ? l : 0.f;
            w[1][0][5] = q + 1 < nq ? rr : 0.f;
            const float yl[4] = {ym.x, ym.y, ym.z, ym.w}, yh[4] = {yp.x, yp.y, yp.z, yp.w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                xc[e] = w[1][0][e + 1];
                float v = fmaf(rep.a[0], xc[e], 0.f);
                v = fmaf(rep.a[1], w[1][0][e], v);
                v = fmaf(rep.a[2], w[1][0][e + 2], v);
                v = fmaf(rep.a[3], yl[e], v);
                v = fmaf(rep.a[4], yh[e], v);
                v = fmaf(rep.a[5 % NST], w[0][0][e + 1], v);
                ax[e] = fmaf(rep.a[6 % NST], w[2][0][e + 1], v);
            }
        } else {
#pragma unroll
            for (int s = 0; s < NST; ++s)
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    ax[e] = fmaf(rep.a[s], w[s / 9][((s / 3) % 3) % NR][e + s % 3], ax[e]);
#pragma unroll
            for (int e = 0; e < 4; ++e) xc[e] = w[1][1 % NR][e + 1];
        }
        float o[4];
        const float be[4] = {bv.x, bv.y, bv.z, bv.w};
        if (RES) {
#pragma unroll
            for (int e = 0; e < 4; ++e) o[e] = ax[e] - be[e];
        } else {
            float4 l4 = make_float4(lrep, lrep, lrep, lrep);
            // a row's ends are its nodes nearest to a face
            if (!rep_lam<3>(g, rep, ix, iy, iz) || !rep_lam<3>(g, rep, ix + 3, iy, iz)) l4 = row4(lam + i, in);
            const float le[4] = {l4.x, l4.y, l4.z, l4.w};
#pragma unroll
            for (int e = 0; e < 4; ++e) o[e] = xc[e] - le[e] * (ax[e] - be[e]);
        }
        if (in) {
            if (rep_row(rep, ix, iy, iz) && rep_row(rep, ix + 3, iy, iz)) {
                *reinterpret_cast<float4 *>(out + i) = make_float4(o[0], o[1], o[2], o[3]);
            } else {
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    if (rep_row(rep, ix + e, iy, iz)) out[i + e] = o[e];
            }
        }
#pragma unroll
        for (int k = 0; k < NR; ++k)
#pragma unroll
            for (int e = 0; e < 6; ++e) {
                w[0][k][e] = w[1][k][e];
                w[1][k][e] = w[2][k][e];
            }
    }
}

template <int KIND, bool RES, bool SYM>
static cs_status launch_rep(const Level &L, const float *A, const float *lam, const float *b, const float *x, float *out,
                            const LamDeep *deep, cudaStream_t s) {
    const auto rep = make_rep<float, Sten<3, KIND>::NST>(L, deep);
    const uintptr_t m = (uintptr_t)lam | (uintptr_t)b | (uintptr_t)x | (uintptr_t)out;
    if (L.g.nx % 4 == 0 && m % 16 == 0) {
        const int64_t per = (int64_t)(L.g.nx / 4) * L.g.ny;
        const int64_t nbox = (per + 255) / 256 * ((L.g.nz + RZ - 1) / RZ);
        RowSet shell{};
        shell.on = 1;
        for (int d = 0; d < 3; ++d) { shell.lo[d] = L.clo[d]; shell.hi[d] = L.chi[d]; }
        shell.nshell = rowset_shell_count(L.g, L.clo, L.chi);
        CSX_CUDA(launch_if(L.settled, k_sweep_rep4<KIND, RES, SYM>, (unsigned)(nbox + (shell.nshell + 255) / 256), 256, 0, s,
                           L.g, A, lam, b, x, out, L.settled, (int)nbox, shell, rep));
        return CS_OK;
    }
    dim3 gr = node_grid(L.g);
    gr.z = (gr.z + RZ - 1) / RZ;
    CSX_CUDA(launch_if(L.settled, k_sweep_rep<KIND, RES, SYM>, gr, node_block(), 0, s, L.g, A, lam, b, x, out, L.settled, rep));
    return CS_OK;
}
// the kernels above where they apply (FP32, 3D, repeated rows, large enough); *done says whether one ran.  FP64 steps
// are bound by their arithmetic: a node per thread (k_sweep) with the same parameters takes 259 us on 256^3, RZ planes
// per thread 287
template <typename T, bool RES>
static cs_status try_rep(const Level &L, const T *A, const T *lam, const T *b, const T *x, T *out,
                         const LamDeep *deep, cudaStream_t s, bool *done) {
    *done = false;
    if constexpr (std::is_same<T, float>::value) {
        if (L.g.dim != 3 || !L.cbox || L.g.N < RZ_MIN_N || out == x) return CS_OK;
        *done = true;
        if (L.kind == STAR) return launch_rep<STAR, RES, false>(L, A, lam, b, x, out, deep, s);
        if (L.sym32) return launch_rep<BOX, RES, true>(L, A, lam, b, x, out, deep, s);
        return launch_rep<BOX, RES, false>(L, A, lam, b, x, out, deep, s);
    }
    return CS_OK;
}

__global__ void k_d2f_box_sym(int64_t N, const double *A, float *__restrict__ o) {
    pdl_trigger();
    pdl_wait();
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < 14 * N; t += (int64_t)gridDim.x * blockDim.x)
        o[t] = (float)A[13 * N + t];
}

cs_status launch_copy_box_sym32(const Level &L, float *o, cudaStream_t s) {
    if (!L.sym32) {
        set_error("internal: symmetric FP32 copy of a level without symmetric storage");
        return CS_ERR_ARG;
    }
    CSX_CUDA(launch_k(k_d2f_box_sym, 1216, 256, 0, s, L.g.N, L.A, o));
    CSX_CUDA(cudaGetLastError());
    count_launch();
    return CS_OK;
}

// ---- BF16 storage, 3D 7-point additive steps: two x-adjacent nodes per
// thread, every array read as bf16x2 pairs (nx even keeps the pairs 4-byte
// aligned).  With one 2-byte load per array and node the BF16 step issues as
// many requests as the FP32 one for half the bytes and stays request-bound;
// pairs halve the requests.  Per node the arithmetic is k_sweep's, in the
// same order.
__global__ void __launch_bounds__(TBX *TBY) k_sweep_bf16x2(Grid g, const __nv_bfloat16 *__restrict__ A,
                                                            const __nv_bfloat16 *__restrict__ lam,
                                                            const __nv_bfloat16 *b,
                                                            const __nv_bfloat16 *x,
                                                            __nv_bfloat16 *__restrict__ out, int xzero, int settled) {
    pdl_trigger();
    if (!settled) pdl_wait();
    const int ix = 2 * (blockIdx.x * TBX + threadIdx.x), iy = blockIdx.y * TBY + threadIdx.y, iz = blockIdx.z;
    const bool in = ix < g.nx && iy < g.ny;
    const int64_t N = g.N, i = ix + (int64_t)g.nx * (iy + (int64_t)g.ny * iz), sy = g.nx, sz = (int64_t)g.nx * g.ny;
    // the rows stay as they were read until x is requested too: converted here, the conversions waited for A
    // before the first read of x (256^3: 99 us, 72 with A kept raw, 67 with x too)
    auto raw = [](const __nv_bfloat16 *p) { return *reinterpret_cast<const unsigned *>(p); };
    auto two = [](unsigned v) { return make_float2(__uint_as_float(v << 16), __uint_as_float(v & 0xffff0000u)); };
    unsigned lraw = 0, araw[7] = {};
    if (in) {
        lraw = raw(lam + i);
        if (!xzero)
#pragma unroll
            for (int s2 = 0; s2 < 7; ++s2) araw[s2] = raw(A + (int64_t)s2 * N + i);
    }
    if (settled) pdl_wait();
    if (!in) return;
    const float2 ll = two(lraw);
    const unsigned braw = raw(b + i);
    float2 res;
    if (xzero) {
        const float2 bb = two(braw);
        res.x = 0.f - ll.x * (-bb.x);  // x = 0: 0 - lam (0 - b)
        res.y = 0.f - ll.y * (-bb.y);
    } else {
        const unsigned r[5] = {raw(x + i), iy > 0 ? raw(x + i - sy) : 0u, iy + 1 < g.ny ? raw(x + i + sy) : 0u,
                               iz > 0 ? raw(x + i - sz) : 0u, iz + 1 < g.nz ? raw(x + i + sz) : 0u};
        // the pairs beside this one hold the x neighbours
        const unsigned left = ix > 0 ? raw(x + i - 2) : 0u, right = ix + 2 < g.nx ? raw(x + i + 2) : 0u;
        const float2 bb = two(braw), xc = two(r[0]), ym = two(r[1]), yp = two(r[2]), zm = two(r[3]), zp = two(r[4]);
        const float xm = two(left).y, xp = two(right).x;
        float2 a[7];
#pragma unroll
        for (int s2 = 0; s2 < 7; ++s2) a[s2] = two(araw[s2]);
        // neighbours in k_sweep's order: centre, -x, +x, -y, +y, -z, +z
        const float n0[7] = {xc.x, xm, xc.y, ym.x, yp.x, zm.x, zp.x};
        const float n1[7] = {xc.y, xc.x, xp, ym.y, yp.y, zm.y, zp.y};
        float a0 = 0.f, a1 = 0.f;
#pragma unroll
        for (int s2 = 0; s2 < 7; ++s2) {
            a0 = fmaf(a[s2].x, n0[s2], a0);
            a1 = fmaf(a[s2].y, n1[s2], a1);
        }
        const float r0 = a0 - bb.x, r1 = a1 - bb.y;
        res.x = xc.x - ll.x * r0;
        res.y = xc.y - ll.y * r1;
    }
    *reinterpret_cast<__nv_bfloat162 *>(out + i) = __floats2bfloat162_rn(res.x, res.y);
}

// ---- FP32, 3D 7-point additive steps: two x-adjacent nodes per thread with
// float2 loads (nx even keeps the pairs 8-byte aligned): half the load
// requests of k_sweep for the same bytes.  Per node the arithmetic is
// k_sweep's, in the same order.
template <bool SYM>
__global__ void __launch_bounds__(TBX *TBY) k_sweep_f32x2(Grid g, const float *__restrict__ A,
                                                           const float *__restrict__ lam, const float *b,
                                                           const float *x, float *__restrict__ out,
                                                           int xzero, int settled) {
    pdl_trigger();
    if (!settled) pdl_wait();
    const int ix = 2 * (blockIdx.x * TBX + threadIdx.x), iy = blockIdx.y * TBY + threadIdx.y, iz = blockIdx.z;
    const bool in = ix < g.nx && iy < g.ny;
    const int64_t N = g.N, i = ix + (int64_t)g.nx * (iy + (int64_t)g.ny * iz), sy = g.nx, sz = (int64_t)g.nx * g.ny;
    auto pair = [](const float *p) { return *reinterpret_cast<const float2 *>(p); };
    float2 ll = make_float2(0.f, 0.f), a[7];
    if (in) {
        ll = pair(lam + i);
        if (!xzero) {
            if (SYM) {  // backward couplings from the neighbours' rows
#pragma unroll
                for (int s2 = 0; s2 < 7; s2 += 2) a[s2] = pair(A + (int64_t)s2 * N + i);
                a[1] = make_float2(ix > 0 ? A[2 * N + i - 1] : 0.f, a[2].x);
                a[3] = iy > 0 ? pair(A + 4 * N + i - sy) : make_float2(0.f, 0.f);
                a[5] = iz > 0 ? pair(A + 6 * N + i - sz) : make_float2(0.f, 0.f);
            } else {
#pragma unroll
                for (int s2 = 0; s2 < 7; ++s2) a[s2] = pair(A + (int64_t)s2 * N + i);
            }
        }
    }
    if (settled) pdl_wait();
    if (!in) return;
    const float2 bb = pair(b + i);
    float2 res;
    if (xzero) {
        res.x = 0.f - ll.x * (-bb.x);  // x = 0: 0 - lam (0 - b)
        res.y = 0.f - ll.y * (-bb.y);
    } else {
        const float2 xc = pair(x + i);
        const float xm = ix > 0 ? x[i - 1] : 0.f;
        const float xp = ix + 2 < g.nx ? x[i + 2] : 0.f;
        const float2 ym = iy > 0 ? pair(x + i - sy) : make_float2(0.f, 0.f);
        const float2 yp = iy + 1 < g.ny ? pair(x + i + sy) : make_float2(0.f, 0.f);
        const float2 zm = iz > 0 ? pair(x + i - sz) : make_float2(0.f, 0.f);
        const float2 zp = iz + 1 < g.nz ? pair(x + i + sz) : make_float2(0.f, 0.f);
        // neighbours in k_sweep's order: centre, -x, +x, -y, +y, -z, +z
        const float n0[7] = {xc.x, xm, xc.y, ym.x, yp.x, zm.x, zp.x};
        const float n1[7] = {xc.y, xc.x, xp, ym.y, yp.y, zm.y, zp.y};
        float a0 = 0.f, a1 = 0.f;
#pragma unroll
        for (int s2 = 0; s2 < 7; ++s2) {
            a0 = fmaf(a[s2].x, n0[s2], a0);
            a1 = fmaf(a[s2].y, n1[s2], a1);
        }
        const float r0 = a0 - bb.x, r1 = a1 - bb.y;
        res.x = xc.x - ll.x * r0;
        res.y = xc.y - ll.y * r1;
    }
    *reinterpret_cast<float2 *>(out + i) = res;
}

template <typename T, bool COLOURED>
static cs_status sweep_dispatch(const Level &L, const T *A, const T *lam, const T *b, const T *x, T *out,
                                int colour, bool xzero, cudaStream_t s, const LamDeep *deep) {
    dim3 gr = node_grid(L.g), bl = node_block();
    int xz = xzero ? 1 : 0;
    // the paired kernels load two values at once: every array must be aligned
    // to two elements (caller-given vectors may be views at an odd offset)
    auto pairs_aligned = [&](size_t bytes) {
        const uintptr_t m = (uintptr_t)A | (uintptr_t)lam | (uintptr_t)b | (uintptr_t)x | (uintptr_t)out;
        return (m % bytes) == 0;
    };
    bool done = false;
    if (!COLOURED && !xzero) CSX_TRY(try_rep<T, false>(L, A, lam, b, x, out, deep, s, &done));
    if (done) {
        count_launch();
        return CS_OK;
    }
    if constexpr (std::is_same<T, __nv_bfloat16>::value) {
        if (!COLOURED && L.g.dim == 3 && L.kind == STAR && L.g.nx % 2 == 0 && out != x && pairs_aligned(4)) {
            const dim3 g2((unsigned)((L.g.nx / 2 + TBX - 1) / TBX), gr.y, gr.z);
            CSX_CUDA(launch_if(L.settled, k_sweep_bf16x2, g2, bl, 0, s, L.g, A, lam, b, x, out, xz, L.settled));
            count_launch();
            return CS_OK;
        }
    }
    if (COLOURED) gr.x = (unsigned)(((L.g.nx + 1) / 2 + TBX - 1) / TBX);
#define CSX_SWEEP(DIM, KIND, SYM)                                                                                \
    CSX_CUDA(launch_if(L.settled, k_sweep<DIM, KIND, T, COLOURED, SYM>, gr, bl, 0, s, L.g, A, lam, b, x, out, colour, xz,   \
                      L.settled, make_rep<T, Sten<DIM, KIND>::NST>(L, deep)))
    if constexpr (std::is_same<T, float>::value) {
        if (!COLOURED && L.g.dim == 3 && L.kind == STAR && L.g.nx % 2 == 0 && out != x && pairs_aligned(8)) {
            const dim3 g2((unsigned)((L.g.nx / 2 + TBX - 1) / TBX), gr.y, gr.z);
            if (L.symstar) CSX_CUDA(launch_if(L.settled, k_sweep_f32x2<true>, g2, bl, 0, s, L.g, A, lam, b, x, out, xz, L.settled));
            else CSX_CUDA(launch_if(L.settled, k_sweep_f32x2<false>, g2, bl, 0, s, L.g, A, lam, b, x, out, xz, L.settled));
            count_launch();
            return CS_OK;
        }
        if (L.sym32 || L.symstar) {  // 27 points: stored symmetric; 7 points: half the couplings read
            if (L.sym32) CSX_SWEEP(3, BOX, true);
            else CSX_SWEEP(3, STAR, true);
            count_launch();
            return CS_OK;
        }
    }
    if (L.g.dim == 2) {
        if (L.kind == STAR) CSX_SWEEP(2, STAR, false);
        else CSX_SWEEP(2, BOX, false);
    } else {
        if (L.kind == STAR) CSX_SWEEP(3, STAR, false);
        else CSX_SWEEP(3, BOX, false);
    }
#undef CSX_SWEEP
    count_launch();
    return CS_OK;
}

template <typename T>
cs_status launch_sweep(const Level &L, const T *A, const T *lam, const T *b, const T *x, T *out, int colour,
                       bool x_is_zero, cudaStream_t s, const LamDeep *deep) {
    if (colour < 0) return sweep_dispatch<T, false>(L, A, lam, b, x, out, -1, x_is_zero, s, deep);
    return sweep_dispatch<T, true>(L, A, lam, b, x, out, colour, x_is_zero, s, deep);
}
template cs_status launch_sweep<double>(const Level &, const double *, const double *, const double *,
                                        const double *, double *, int, bool, cudaStream_t, const LamDeep *);
template cs_status launch_sweep<float>(const Level &, const float *, const float *, const float *, const float *,
                                       float *, int, bool, cudaStream_t, const LamDeep *);
template cs_status launch_sweep<__nv_bfloat16>(const Level &, const __nv_bfloat16 *, const __nv_bfloat16 *,
                                               const __nv_bfloat16 *, const __nv_bfloat16 *, __nv_bfloat16 *, int, bool,
                                               cudaStream_t, const LamDeep *);

// ------------------------------------------- a 2D cascade in one launch
// All nu x ncol steps of one application on a tile held in shared memory: a
// CTA reads its tile of x with a halo as wide as the step count, every step
// is valid on a region one node smaller than the last, and the tile's middle
// is written out.  Rows of A, Lambda and b stay in registers for all steps.
// The steps' arithmetic per node is k_sweep's, in the same order.  A step as a
// launch of its own is bound by the launch up to about 256^2 nodes and by L2
// above; the halo costs (TXT TYT) / ((TXT - 2 H)(TYT - 2 H)) times the work.
// Right GMRES on 1023^2 (FP32 cycles, red-black) went from 6.19 to 5.44 ms, a
// stationary FP64 solve on 64^2 from 780 to 675 us.
template <int KIND, typename T, bool MULT, int TXT, int TYT, int NPT>
__global__ void __launch_bounds__(TXT *TYT / NPT) k_cascade2d(Grid g, const T *__restrict__ A,
                                                            const T *__restrict__ lam, const T *b,
                                                            const T *x, T *__restrict__ out, int nu,
                                                            int reverse, int xzero, int settled) {
    constexpr int NST = Sten<2, KIND>::NST, RP = TYT / NPT;  // rows per pass over the tile
    constexpr int NU = 4;
    constexpr bool INPL = MULT && KIND == STAR;  // a colour's nodes read the other colour only
    __shared__ T xs[INPL ? 1 : 2][TYT][TXT + 1];
    pdl_trigger();
    if (!settled) pdl_wait();
    const int ncol = MULT ? 2 : 1, H = nu * ncol;
    const int tx = threadIdx.x % TXT, ty = threadIdx.x / TXT;
    const int gx = blockIdx.x * (TXT - 2 * H) + tx - H, gy0 = blockIdx.y * (TYT - 2 * H) + ty - H;
    T a[NPT][NST], lr[NPT][NU], bv[NPT];
#pragma unroll
    for (int k = 0; k < NPT; ++k) {
        const int gy = gy0 + RP * k;
        const bool in = (unsigned)gx < (unsigned)g.nx && (unsigned)gy < (unsigned)g.ny;
        const int64_t i = in ? gx + (int64_t)g.nx * gy : 0;
#pragma unroll
        for (int s = 0; s < NST; ++s) a[k][s] = in ? A[(int64_t)s * g.N + i] : T(0);
#pragma unroll
        for (int l = 0; l < NU; ++l) lr[k][l] = in && l < nu ? lam[(int64_t)l * g.N + i] : T(0);
    }
    if (settled) pdl_wait();
#pragma unroll
    for (int k = 0; k < NPT; ++k) {
        const int gy = gy0 + RP * k;
        const bool in = (unsigned)gx < (unsigned)g.nx && (unsigned)gy < (unsigned)g.ny;
        const int64_t i = in ? gx + (int64_t)g.nx * gy : 0;
        bv[k] = in ? b[i] : T(0);
        xs[0][ty + RP * k][tx] = in && !xzero ? x[i] : T(0);
        if (!INPL) xs[INPL ? 0 : 1][ty + RP * k][tx] = T(0);  // nodes outside the grid stay zero
    }
    __syncthreads();
    int cur = 0;
    for (int st = 0; st < H; ++st) {
        const int step = st / ncol, lv = reverse ? nu - 1 - step : step;
        const int colour = MULT ? (reverse ? 1 - (st & 1) : st & 1) : 0;
        const T(*src)[TXT + 1] = xs[cur];
        T(*dst)[TXT + 1] = xs[INPL ? 0 : cur ^ 1];
#pragma unroll
        for (int k = 0; k < NPT; ++k) {
            const int ly = ty + RP * k, gy = gy0 + RP * k;
            const bool in = (unsigned)gx < (unsigned)g.nx && (unsigned)gy < (unsigned)g.ny;
            if (!in || tx <= st || tx >= TXT - 1 - st || ly <= st || ly >= TYT - 1 - st) continue;
            const T xc = src[ly][tx];
            if (MULT && node_colour(2, gx, gy, 0) != colour) {
                if (!INPL) dst[ly][tx] = xc;
                continue;
            }
            T ax = T(0);
#pragma unroll
            for (int s = 0; s < NST; ++s) {
                int dx, dy, dz;
                Sten<2, KIND>::off(s, dx, dy, dz);
                ax = fma(a[k][s], src[ly + dy][tx + dx], ax);
            }
            T li = lr[k][0];
#pragma unroll
            for (int l = 1; l < NU; ++l)
                if (l == lv) li = lr[k][l];
            dst[ly][tx] = xc - li * (ax - bv[k]);
        }
        __syncthreads();
        if (!INPL) cur ^= 1;
    }
#pragma unroll
    for (int k = 0; k < NPT; ++k) {
        const int ly = ty + RP * k, gy = gy0 + RP * k;
        if ((unsigned)gx < (unsigned)g.nx && (unsigned)gy < (unsigned)g.ny && tx >= H && tx < TXT - H && ly >= H &&
            ly < TYT - H)
            out[gx + (int64_t)g.nx * gy] = xs[cur][ly][tx];
    }
}

// FP32: tiles of 64 x 48 on levels above 256^2 (1.6 times the work with six
// steps), 32 x 32 below, where more CTAs shorten the chain.  FP64 pays the
// halo's work at 1/64 of the FP32 rate: 16 x 16 tiles, while two per SM hold
// the level (tiles of 32 x 32 on 64^2 left all of it to nine SMs: a solve took
// 945 us, 780 with a launch per step, 675 with the small tiles).
template <typename T>
bool cascade2d_fits(const Level &L, int nu, int ncol) {
    if (std::is_same<T, __nv_bfloat16>::value || L.g.dim != 2 || L.bs != 1) return false;
    if (nu > 4 || nu * ncol < 2 || nu * ncol > 8) return false;
    const int H = nu * ncol, w = 16 - 2 * H;
    return std::is_same<T, float>::value ||
           (H <= 4 && (int64_t)((L.g.nx + w - 1) / w) * ((L.g.ny + w - 1) / w) <= 304);
}
template <typename T>
cs_status launch_cascade2d(const Level &L, const T *A, const T *lam, const T *b, const T *x, T *out, int nu, int ncol,
                           bool reverse, bool x_is_zero, cudaStream_t s) {
    if constexpr (!std::is_same<T, __nv_bfloat16>::value) {
        const int H = nu * ncol;
#define CSX_C2D(KIND, MULT, TX, TY, NP)                                                                             \
    CSX_CUDA(launch_if(L.settled, k_cascade2d<KIND, T, MULT, TX, TY, NP>,                                                       \
                      dim3((unsigned)((L.g.nx + TX - 2 * H - 1) / (TX - 2 * H)),                                    \
                           (unsigned)((L.g.ny + TY - 2 * H - 1) / (TY - 2 * H))),                                   \
                      TX * TY / NP, 0, s, L.g, A, lam, b, x, out, nu, reverse ? 1 : 0, x_is_zero ? 1 : 0, L.settled))
#define CSX_C2D_ALL(TX, TY, NP)                                                                                    \
    do {                                                                                                           \
        if (L.kind == STAR && ncol == 2) CSX_C2D(STAR, true, TX, TY, NP);                                          \
        else if (L.kind == STAR) CSX_C2D(STAR, false, TX, TY, NP);                                                 \
        else if (ncol == 2) CSX_C2D(BOX, true, TX, TY, NP);                                                        \
        else CSX_C2D(BOX, false, TX, TY, NP);                                                                      \
    } while (0)
        if constexpr (std::is_same<T, double>::value) {
            CSX_C2D_ALL(16, 16, 1);
        } else {
            if (L.g.N > 256 * 256) CSX_C2D_ALL(64, 48, 6);
            else CSX_C2D_ALL(32, 32, 2);
        }
#undef CSX_C2D_ALL
#undef CSX_C2D
        count_launch();
        return CS_OK;
    }
    set_error("internal: no fused cascade for this type");
    return CS_ERR_ARG;
}
#define CSX_C2D_INST(T)                                                                                             \
    template bool cascade2d_fits<T>(const Level &, int, int);                                                       \
    template cs_status launch_cascade2d<T>(const Level &, const T *, const T *, const T *, const T *, T *, int, int, \
                                           bool, bool, cudaStream_t);
CSX_C2D_INST(double)
CSX_C2D_INST(float)
CSX_C2D_INST(__nv_bfloat16)
#undef CSX_C2D_INST

// ------------------------------------------------------------ block steps
// Nodes of block (bx,by,bz): bs*b + l per axis, local position
// lp = lx + bs (ly + bs lz); partial blocks at the upper edges skip absent
// positions.  Lambda_b is nmax x nmax over local positions.
template <int DIM, int NMAX>
__device__ __forceinline__ int block_nodes(const Grid &g, int bs, int bx, int by, int bz, int *node, int *lpos,
                                           int (*co)[3]) {
    int np = 0;
    for (int lp = 0; lp < NMAX; ++lp) {
        const int lx = lp % bs, ly = (lp / bs) % bs, lz = DIM == 3 ? lp / (bs * bs) : 0;
        if (DIM == 2 && lp >= bs * bs) break;
        const int ix = bs * bx + lx, iy = bs * by + ly, iz = DIM == 3 ? bs * bz + lz : 0;
        if (ix >= g.nx || iy >= g.ny || (DIM == 3 && iz >= g.nz)) continue;
        node[np] = ix + g.nx * (iy + g.ny * iz);
        lpos[np] = lp;
        co[np][0] = ix; co[np][1] = iy; co[np][2] = iz;
        ++np;
    }
    return np;
}

// out_b = x_b - Lambda_b^(T) ((A x)_b - b_b), one thread per block
template <int DIM, int KIND, typename T, int NMAX, bool COLOURED>
__global__ void k_block_sweep(Grid g, int bs, int nbx, int nby, int64_t nblocks, const T *__restrict__ A,
                              const T *__restrict__ lam, const T *b, const T *x, T *out, int colour,
                              int transpose, int xzero) {
    pdl_trigger();
    pdl_wait();
    const int64_t blk = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (blk >= nblocks) return;
    const int bx = (int)(blk % nbx), by = (int)((blk / nbx) % nby), bz = (int)(blk / ((int64_t)nbx * nby));
    int node[NMAX], lpos[NMAX], co[NMAX][3];
    const int np = block_nodes<DIM, NMAX>(g, bs, bx, by, bz, node, lpos, co);
    if (COLOURED && ((((bx + 1) + (by + 1) + (DIM == 3 ? bz + 1 : 0)) & 1) != colour)) {
        for (int p = 0; p < np; ++p) {
            if (xzero) out[node[p]] = T(0);
            else if (out != x) out[node[p]] = x[node[p]];
        }
        return;
    }
    T r[NMAX];
    for (int p = 0; p < np; ++p)
        r[p] = (xzero ? T(0) : apply_row<DIM, KIND, T>(g, A, x, co[p][0], co[p][1], co[p][2], node[p])) - b[node[p]];
    const T *lb = lam + blk * (NMAX * NMAX);
    T xo[NMAX];
    for (int p = 0; p < np; ++p) {
        T acc = xzero ? T(0) : x[node[p]];
        for (int q = 0; q < np; ++q)
            acc = fma(-(transpose ? lb[lpos[q] * NMAX + lpos[p]] : lb[lpos[p] * NMAX + lpos[q]]), r[q], acc);
        xo[p] = acc;
    }
    for (int p = 0; p < np; ++p) out[node[p]] = xo[p];
}

template <typename T>
cs_status launch_block_sweep(const Level &L, const T *A, const T *lam, const T *b, const T *x, T *out, int colour,
                             bool transpose, bool xzero, cudaStream_t s) {
    const int threads = 128;
    const unsigned nblk = (unsigned)((L.nblocks + threads - 1) / threads);
    const int tr = transpose ? 1 : 0, xz = xzero ? 1 : 0;
#define CSX_BSW(DIM, KIND, NM)                                                                                   \
    if (colour < 0)                                                                                              \
        CSX_CUDA(launch_k(k_block_sweep<DIM, KIND, T, NM, false>, nblk, threads, 0, s, L.g, L.bs, L.nbx, L.nby, L.nblocks, A, lam, \
                                                                         b, x, out, colour, tr, xz));              \
    else                                                                                                         \
        CSX_CUDA(launch_k(k_block_sweep<DIM, KIND, T, NM, true>, nblk, threads, 0, s, L.g, L.bs, L.nbx, L.nby, L.nblocks, A, lam, \
                                                                        b, x, out, colour, tr, xz));
    if (L.g.dim == 2) {
        if (L.nmax <= 4) { if (L.kind == STAR) { CSX_BSW(2, STAR, 4) } else { CSX_BSW(2, BOX, 4) } }
        else { if (L.kind == STAR) { CSX_BSW(2, STAR, 9) } else { CSX_BSW(2, BOX, 9) } }
    } else {
        if (L.kind == STAR) { CSX_BSW(3, STAR, 8) } else { CSX_BSW(3, BOX, 8) }
    }
#undef CSX_BSW
    CSX_CUDA(cudaGetLastError());
    count_launch();
    return CS_OK;
}
template cs_status launch_block_sweep<double>(const Level &, const double *, const double *, const double *,
                                              const double *, double *, int, bool, bool, cudaStream_t);
template cs_status launch_block_sweep<float>(const Level &, const float *, const float *, const float *, const float *,
                                             float *, int, bool, bool, cudaStream_t);
// BF16 storage is implemented for point-block levels only
template <>
cs_status launch_block_sweep<__nv_bfloat16>(const Level &, const __nv_bfloat16 *, const __nv_bfloat16 *,
                                            const __nv_bfloat16 *, const __nv_bfloat16 *, __nv_bfloat16 *, int, bool,
                                            bool, cudaStream_t) {
    set_error("BF16 cycles are implemented for point-block levels only");
    return CS_ERR_UNSUPPORTED;
}

// The multi-RHS block step X_b <- X_b - Lambda_b^(T) (A X - B)_b.  One warp
// per node of a block (lane r = right-hand side r, so every load of X and B
// is a contiguous row of m values); the residual rows of a block meet in
// shared memory and, after one barrier, each warp forms its node's row of the
// n_b x m block product.  Per RHS and unknown this is nst + n_b FMAs against
// (nst + n_b + 3 m) words moved: HBM-bound, so plain FMAs, no tensor cores.
// BPC blocks adjacent in x share a CTA of 32 * NMAX * BPC threads; the grid
// spans the block grid (x tiles of BPC, y, z), so no index division is needed.
template <int DIM, int KIND, typename T, int BS, int BPC>
__global__ void __launch_bounds__(32 * (DIM == 3 ? BS * BS * BS : BS * BS) * BPC)
    k_block_sweep_m(Grid g, int nbx, const T *__restrict__ A, const T *__restrict__ lam, const T *B,
                    const T *X, T *out, int m, int colour, int transpose) {
    pdl_trigger();
    pdl_wait();
    using S = Sten<DIM, KIND>;
    constexpr int NMAX = DIM == 3 ? BS * BS * BS : BS * BS;
    __shared__ T rsm[BPC][NMAX][32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int bl = warp / NMAX, lp = warp % NMAX;  // compile-time divisors
    const int bx = blockIdx.x * BPC + bl, by = blockIdx.y, bz = blockIdx.z;
    const int lx = lp % BS, ly = (lp / BS) % BS, lz = DIM == 3 ? lp / (BS * BS) : 0;
    const int ix = BS * bx + lx, iy = BS * by + ly, iz = DIM == 3 ? BS * bz + lz : 0;
    const bool present = bx < nbx && ix < g.nx && iy < g.ny && (DIM == 2 || iz < g.nz);
    const bool active = colour < 0 || ((((bx + 1) + (by + 1) + (DIM == 3 ? bz + 1 : 0)) & 1) == colour);
    const bool work = present && lane < m;
    const int64_t i = ix + (int64_t)g.nx * (iy + (int64_t)g.ny * iz);
    T r = T(0);
    if (work && active) {
        T ax = T(0);
#pragma unroll
        for (int s = 0; s < S::NST; ++s) {
            int dx, dy, dz;
            S::off(s, dx, dy, dz);
            const int jx = ix + dx, jy = iy + dy, jz = iz + dz;
            const bool in = (unsigned)jx < (unsigned)g.nx && (unsigned)jy < (unsigned)g.ny &&
                            (DIM == 2 || (unsigned)jz < (unsigned)g.nz);
            const int64_t j = i + dx + (int64_t)g.nx * (dy + (int64_t)g.ny * dz);
            ax = fma(A[(int64_t)s * g.N + i], in ? X[j * m + lane] : T(0), ax);
        }
        r = ax - B[i * m + lane];
    }
    rsm[bl][lp][lane] = r;  // absent nodes contribute zero (their Lambda entries are zero too)
    __syncthreads();
    if (!work) return;
    if (!active) {
        if (out != X) out[i * m + lane] = X[i * m + lane];
        return;
    }
    const int64_t blk = bx + (int64_t)nbx * (by + (int64_t)gridDim.y * bz);
    const T *lb = lam + blk * (NMAX * NMAX);
    T acc = X[i * m + lane];
#pragma unroll
    for (int q = 0; q < NMAX; ++q)
        acc = fma(-(transpose ? lb[q * NMAX + lp] : lb[lp * NMAX + q]), rsm[bl][q][lane], acc);
    out[i * m + lane] = acc;
}

// The same block step in FP32 with four right-hand sides per lane (float4),
// for m = 4 LPN right-hand sides and blocks of NMAX nodes with NMAX LPN
// dividing 32: a warp holds 32 / (NMAX LPN) whole blocks, lane l takes node
// (l / LPN) % NMAX of its block and right-hand sides 4 (l % LPN) .. +3.  Every
// load of a step (coefficients, the x neighbourhood, b and the Lambda row) is
// issued before the first use, the block's residuals meet through warp
// shuffles (no CTA barrier), and warps stride over the blocks.  Per RHS and
// node the arithmetic and its order are those of k_block_sweep_m.
template <int DIM, int KIND, int BS, int LPN>
__global__ void __launch_bounds__(256) k_block_sweep_m4(Grid g, int nbx, int nby, int64_t nblocks,
                                                        const float *__restrict__ A, const float *__restrict__ lam,
                                                        const float4 *B, const float4 *X, float4 *out,
                                                        int colour, int transpose) {
    pdl_trigger();
    pdl_wait();
    using S = Sten<DIM, KIND>;
    constexpr int NMAX = DIM == 3 ? BS * BS * BS : BS * BS;
    constexpr int G = NMAX * LPN;  // lanes per block
    constexpr int BPW = 32 / G;    // blocks per warp
    const int lane = threadIdx.x & 31;
    const int gsub = lane / G, lp = (lane % G) / LPN, rg = lane % LPN;
    const int64_t warp0 = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const int lx = lp % BS, ly = (lp / BS) % BS, lz = DIM == 3 ? lp / (BS * BS) : 0;
    // block and node indices fit in 31 bits (the hierarchy checks N < 2^31): 32-bit index arithmetic
    for (int64_t w = warp0; w * BPW < nblocks; w += nwarps) {
        const int blk = (int)(w * BPW) + gsub;
        const bool valid = blk < nblocks;
        int bx = 0, by = 0, bz = 0;
        if (valid) {
            const int q = blk / nbx;
            bx = blk - q * nbx;
            if (DIM == 3) {
                bz = q / nby;
                by = q - bz * nby;
            } else {
                by = q;
            }
        }
        const int ix = BS * bx + lx, iy = BS * by + ly, iz = DIM == 3 ? BS * bz + lz : 0;
        const bool present = valid && ix < g.nx && iy < g.ny && (DIM == 2 || iz < g.nz);
        const bool active = colour < 0 || ((((bx + 1) + (by + 1) + (DIM == 3 ? bz + 1 : 0)) & 1) == colour);
        const int i = ix + g.nx * (iy + g.ny * iz);
        float4 r = make_float4(0.f, 0.f, 0.f, 0.f), xo = r;
        float lrow[NMAX];
        if (present && active) {
            const float *lb = lam + (int64_t)blk * (NMAX * NMAX);
#pragma unroll
            for (int q = 0; q < NMAX; ++q) lrow[q] = transpose ? lb[q * NMAX + lp] : lb[lp * NMAX + q];
            float4 ax = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int s = 0; s < S::NST; ++s) {
                int dx, dy, dz;
                S::off(s, dx, dy, dz);
                const bool in = (unsigned)(ix + dx) < (unsigned)g.nx && (unsigned)(iy + dy) < (unsigned)g.ny &&
                                (DIM == 2 || (unsigned)(iz + dz) < (unsigned)g.nz);
                const int j = i + dx + g.nx * (dy + g.ny * dz);
                const float a = A[(int64_t)s * g.N + i];
                const float4 xv = in ? X[(int64_t)j * LPN + rg] : make_float4(0.f, 0.f, 0.f, 0.f);
                if (dx == 0 && dy == 0 && dz == 0) xo = xv;
                ax.x = fmaf(a, xv.x, ax.x);
                ax.y = fmaf(a, xv.y, ax.y);
                ax.z = fmaf(a, xv.z, ax.z);
                ax.w = fmaf(a, xv.w, ax.w);
            }
            const float4 bv = B[(int64_t)i * LPN + rg];
            r = make_float4(ax.x - bv.x, ax.y - bv.y, ax.z - bv.z, ax.w - bv.w);
        } else if (present) {
            xo = X[(int64_t)i * LPN + rg];
        }
        // residuals of the block's nodes (absent nodes: 0, their Lambda entries are 0 too)
        float4 acc = xo;
        const int base = gsub * G + rg;
#pragma unroll
        for (int q = 0; q < NMAX; ++q) {
            const float rx = __shfl_sync(0xffffffffu, r.x, base + q * LPN);
            const float ry = __shfl_sync(0xffffffffu, r.y, base + q * LPN);
            const float rz = __shfl_sync(0xffffffffu, r.z, base + q * LPN);
            const float rw = __shfl_sync(0xffffffffu, r.w, base + q * LPN);
            if (present && active) {
                acc.x = fmaf(-lrow[q], rx, acc.x);
                acc.y = fmaf(-lrow[q], ry, acc.y);
                acc.z = fmaf(-lrow[q], rz, acc.z);
                acc.w = fmaf(-lrow[q], rw, acc.w);
            }
        }
        if (present && (active || out != X)) out[(int64_t)i * LPN + rg] = acc;
    }
}

// The steps on 2D levels of 2x2-node blocks: a thread takes a whole block, so
// that a block's residuals stay in registers and its rows share one read of
// the x neighbourhood (12 values for four 5-point rows instead of 20).
template <int KIND, typename T>
struct BlockRows {
    T a[4][Sten<2, KIND>::NST], lb[16];
    __device__ __forceinline__ void load(const Grid &g, int nbx, int bx, int by, const T *__restrict__ A,
                                         const T *__restrict__ lam) {
        const bool px = 2 * bx + 1 < g.nx, py = 2 * by + 1 < g.ny;
        const int64_t i0 = 2 * bx + (int64_t)g.nx * (2 * by);
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int s = 0; s < Sten<2, KIND>::NST; ++s)
                a[q][s] = ((q & 1) == 0 || px) && (q < 2 || py)
                              ? A[(int64_t)s * g.N + i0 + (q & 1) + (int64_t)g.nx * (q >> 1)]
                              : T(0);
        struct alignas(16) Q {
            T v[16 / sizeof(T)];
        };
        const Q *l = reinterpret_cast<const Q *>(lam + (bx + (int64_t)nbx * by) * 16);
#pragma unroll
        for (int e = 0; e < 16; ++e) lb[e] = l[e / (16 / sizeof(T))].v[e % (16 / sizeof(T))];
    }
};
// the step's arithmetic: residuals of the block's rows from x around it (w[y +
// 1][x + 1]) and b, then store(p, the new values of node p)
template <int KIND, typename T, int V, typename P, typename F>
__device__ __forceinline__ void block_step(const BlockRows<KIND, T> &c, const P (&w)[4][4], const P (&bq)[4],
                                           const bool (&pres)[4], int transpose, F &&store) {
    T r[4][V];
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int e = 0; e < V; ++e) {
            T ax = T(0);
#pragma unroll
            for (int s = 0; s < Sten<2, KIND>::NST; ++s) {
                int dx, dy, dz;
                Sten<2, KIND>::off(s, dx, dy, dz);
                ax = fma(c.a[q][s], w[(q >> 1) + 1 + dy][(q & 1) + 1 + dx].v[e], ax);
            }
            r[q][e] = pres[q] ? ax - bq[q].v[e] : T(0);
        }
#pragma unroll
    for (int p = 0; p < 4; ++p) {
        if (!pres[p]) continue;
        P o = w[(p >> 1) + 1][(p & 1) + 1];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const T l = -(transpose ? c.lb[4 * q + p] : c.lb[4 * p + q]);
#pragma unroll
            for (int e = 0; e < V; ++e) o.v[e] = fma(l, r[q][e], o.v[e]);
        }
        store(p, o);
    }
}
template <typename T, int V, bool VEC>
struct alignas(VEC ? sizeof(T) * V : sizeof(T)) Cols {
    T v[V];
};
// V right-hand sides per thread, x straight from memory, blocks in their
// order: for column counts without 16-byte copies.  VEC: the V are adjacent
// and come in one load; else they lie G apart, so that a warp's loads stay
// contiguous and A is read once for all V.  FP32 on 1024^2, us: a thread per
// node and 32 lanes per node took 205 (1 column), 207 (3), 228 (6), 243 (19)
// and 250 (30); here 9.6, 14, 21, 75 and 87
// (floor 7.4, 11, 17, 41 and 61).
template <int KIND, typename T, int V, bool VEC>
__global__ void __launch_bounds__(128) k_block_sweep_q(Grid g, int nbx, int nby, int m, int G, const T *__restrict__ A,
                                                       const T *__restrict__ lam, const T *B, const T *X, T *out,
                                                       int colour, int transpose, int settled) {
    using P = Cols<T, V, VEC>;
    pdl_trigger();
    if (!settled) pdl_wait();
    const unsigned t = blockIdx.x * 128u + threadIdx.x;
    // block rows along the grid's y and, beyond its 65,535, z
    const int bx = (int)(t / (unsigned)G), rg = (int)(t - (unsigned)bx * G), by = blockIdx.y + gridDim.y * blockIdx.z;
    const bool on = bx < nbx && by < nby;
    const bool px = 2 * bx + 1 < g.nx, py = 2 * by + 1 < g.ny;
    const int64_t i0 = 2 * bx + (int64_t)g.nx * (2 * by);
    const bool active = on && (colour < 0 || (((bx + 1) + (by + 1)) & 1) == colour);
    const bool pres[4] = {true, px, py, px && py};
    BlockRows<KIND, T> c;
    if (active) c.load(g, nbx, bx, by, A, lam);
    if (settled) pdl_wait();
    if (!on) return;
    auto get = [&](const T *p, int64_t node) {
        P o;
        if (VEC) {
            o = reinterpret_cast<const P *>(p)[node * G + rg];
        } else {
#pragma unroll
            for (int e = 0; e < V; ++e) o.v[e] = V == 1 || rg + e * G < m ? p[node * m + rg + e * G] : T(0);
        }
        return o;
    };
    auto put = [&](int64_t node, const P &o) {
        if (VEC) {
            reinterpret_cast<P *>(out)[node * G + rg] = o;
        } else {
#pragma unroll
            for (int e = 0; e < V; ++e)
                if (V == 1 || rg + e * G < m) out[node * m + rg + e * G] = o.v[e];
        }
    };
    auto at = [&](int q) { return i0 + (q & 1) + (int64_t)g.nx * (q >> 1); };
    if (!active) {
        if (out != X)
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (pres[q]) put(at(q), get(X, at(q)));
        return;
    }
    P w[4][4];  // x around the block: w[y + 1][x + 1]
#pragma unroll
    for (int wy = 0; wy < 4; ++wy)
#pragma unroll
        for (int wx = 0; wx < 4; ++wx) {
            if (KIND == STAR && (wx == 0 || wx == 3) && (wy == 0 || wy == 3)) continue;
            const int ix = 2 * bx + wx - 1, iy = 2 * by + wy - 1;
            if ((unsigned)ix < (unsigned)g.nx && (unsigned)iy < (unsigned)g.ny)
                w[wy][wx] = get(X, ix + (int64_t)g.nx * iy);
            else
#pragma unroll
                for (int e = 0; e < V; ++e) w[wy][wx].v[e] = T(0);
        }
    P bq[4];
#pragma unroll
    for (int q = 0; q < 4; ++q)
        if (pres[q]) bq[q] = get(B, at(q));
    block_step<KIND, T, V>(c, w, bq, pres, transpose, [&](int p, const P &o) { put(at(p), o); });
}

// Vectors of V = 16 bytes of right-hand sides per thread, tiles of bxc x byc
// blocks of x (with one node around) and b staged in shared memory by 16-byte
// asynchronous copies, a tile ahead, by CTAs that stride over the tiles; rows
// of A and Lambda come into registers meanwhile, where these suffice those of
// the next tile.  Bound by HBM: (nst + 4 + 3 m) words per node; loads straight
// into registers kept too little in flight.  FP32, 1024^2, 5-point, 32
// columns: 90.4 us with a thread per node and shuffles, 107 with a block per
// thread and x from memory, 86.4 here (floor 65); 16: 51, 50 and 47 (35).
template <int KIND, typename T>
__global__ void __launch_bounds__(128, sizeof(T) == 8 ? 2 : KIND == STAR ? 4 : 3) k_block_sweep_s(Grid g, int nbx, int nby, int m, int G, int bxc, int byc,
                                                          int tilesx, int ntiles, const T *__restrict__ A,
                                                          const T *__restrict__ lam, const T *B, const T *X, T *out,
                                                          int colour, int transpose, int settled) {
    constexpr int V = 16 / (int)sizeof(T);
    using P = Cols<T, V, true>;
    // two tiles: bxc byc G <= 128 blocks times vectors and m sizeof(T) <= 16 G, so that b's part of a tile
    // has at most 8 KB and x's, with its rim, 15 KB (4 x 2 blocks, G = 16)
    constexpr int XB = 15360, SB = XB + 8192;
    __shared__ __align__(16) unsigned char sm[2][SB];
    pdl_trigger();
    if (!settled) pdl_wait();
    const int wpx = (2 * bxc + 2) * m, wpb = 2 * bxc * m;  // words per staged row
    const int tb = (int)threadIdx.x / G, rg = (int)threadIdx.x - tb * G, ty = tb / bxc, tx = tb - ty * bxc;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // rows of a tile: 2 byc + 2 of x, then 2 byc of b; columns outside the grid are zero
    auto stage = [&](int t, int slot) {
        const int ty0 = t / tilesx, x0 = 2 * bxc * (t - ty0 * tilesx), y0 = 2 * byc * ty0;
        for (int r = warp; r < 4 * byc + 2; r += 4) {
            const bool isx = r < 2 * byc + 2;
            const int iy = isx ? y0 + r - 1 : y0 + r - (2 * byc + 2);
            const int xs = isx ? x0 - 1 : x0, n = isx ? wpx : wpb, cols = isx ? 2 * bxc + 2 : 2 * bxc;
            const bool row = (unsigned)iy < (unsigned)g.ny;
            // words [lo, hi) of the row lie in the grid
            const int lo = xs < 0 ? m : 0, hi = row ? min(cols, g.nx - xs) * m : 0;
            const T *src = (isx ? X : B) + (row ? ((int64_t)g.nx * iy + xs) * m : 0);
            const unsigned dst = (unsigned)__cvta_generic_to_shared(
                sm[slot] + (isx ? r * wpx * (int)sizeof(T) : XB + (r - (2 * byc + 2)) * wpb * (int)sizeof(T)));
            for (int w = lane * V; w < n; w += 32 * V) {
                const bool in = w >= lo && w < hi;
                const T *p = in ? src + w : X;
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst + w * (int)sizeof(T)), "l"(p),
                             "r"(in ? 16 : 0)
                             : "memory");
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    auto block = [&](int t, int &bx, int &by) {
        const int ty0 = t / tilesx;
        bx = bxc * (t - ty0 * tilesx) + tx;
        by = byc * ty0 + ty;
        return ty < byc && bx < nbx && by < nby;
    };
    auto is_active = [&](int bx, int by) { return colour < 0 || (((bx + 1) + (by + 1)) & 1) == colour; };
    constexpr bool AHEAD = sizeof(T) == 4 && KIND == STAR;  // where the registers hold a second set of rows
    BlockRows<KIND, T> c, cn;
    auto rows = [&](int t, BlockRows<KIND, T> &to) {
        int bx, by;
        if (block(t, bx, by) && is_active(bx, by)) to.load(g, nbx, bx, by, A, lam);
    };
    int t = blockIdx.x, bx, by;
    if (AHEAD) rows(t, c);
    if (settled) pdl_wait();
    stage(t, 0);
    for (int it = 0; t < ntiles; t += gridDim.x, ++it) {
        const int nt = t + gridDim.x;
        if (!AHEAD) rows(t, c);
        if (nt < ntiles) {
            if (AHEAD) rows(nt, cn);
            stage(nt, (it + 1) & 1);
            asm volatile("cp.async.wait_group 1;" ::: "memory");
        } else {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
        }
        __syncthreads();
        if (block(t, bx, by)) {
            const T *xs = reinterpret_cast<const T *>(sm[it & 1]) + (2 * ty) * wpx + (2 * tx) * m;
            const T *bs = reinterpret_cast<const T *>(sm[it & 1] + XB) + (2 * ty) * wpb + (2 * tx) * m;
            auto get = [&](const T *p) { return *reinterpret_cast<const P *>(p + rg * V); };
            auto put = [&](int64_t node, const P &o) { reinterpret_cast<P *>(out)[node * G + rg] = o; };
            const bool px = 2 * bx + 1 < g.nx, py = 2 * by + 1 < g.ny;
            const bool pres[4] = {true, px, py, px && py};
            const int64_t i0 = 2 * bx + (int64_t)g.nx * (2 * by);
            auto X4 = [&](int wy, int wx) { return get(xs + wy * wpx + wx * m); };  // x at (wy - 1, wx - 1)
            if (!is_active(bx, by)) {
                if (out != X)
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        if (pres[q]) put(i0 + (q & 1) + (int64_t)g.nx * (q >> 1), X4((q >> 1) + 1, (q & 1) + 1));
            } else {
                P w[4][4];
#pragma unroll
                for (int wy = 0; wy < 4; ++wy)
#pragma unroll
                    for (int wx = 0; wx < 4; ++wx) {
                        if (KIND == STAR && (wx == 0 || wx == 3) && (wy == 0 || wy == 3)) continue;
                        w[wy][wx] = X4(wy, wx);
                    }
                const P bq[4] = {get(bs), get(bs + m), get(bs + wpb), get(bs + wpb + m)};
                block_step<KIND, T, V>(c, w, bq, pres, transpose, [&](int p, const P &o) {
                    put(i0 + (p & 1) + (int64_t)g.nx * (p >> 1), o);
                });
            }
        }
        if (AHEAD) c = cn;
        __syncthreads();  // the slot is staged anew in the next pass
    }
}

template <int KIND, typename T>
static cs_status block_sweep_s(const Level &L, const T *A, const T *lam, const T *b, const T *x, T *out, int m,
                               int colour, int tr, cudaStream_t s) {
    const int G = m * (int)sizeof(T) / 16, nb = 128 / G, byc = nb >= 16 ? 4 : 2, bxc = nb / byc;
    int dev = 0, nsm = 0;
    CSX_CUDA(cudaGetDevice(&dev));
    CSX_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
    const int tilesx = (L.nbx + bxc - 1) / bxc, ntiles = tilesx * ((L.nby + byc - 1) / byc);
    const unsigned grid = (unsigned)std::min(ntiles, 4 * nsm);
    CSX_CUDA(launch_if(L.settled, k_block_sweep_s<KIND, T>, grid, 128, 0, s, L.g, L.nbx, L.nby, m, G, bxc, byc, tilesx,
                       ntiles, A, lam, b, x, out, colour, tr, L.settled));
    count_launch();
    return CS_OK;
}
template <int KIND, typename T, int V, bool VEC>
static cs_status block_sweep_q(const Level &L, const T *A, const T *lam, const T *b, const T *x, T *out, int m,
                               int colour, int tr, cudaStream_t s) {
    const int G = (m + V - 1) / V;
    const int gz = (L.nby + 65534) / 65535;
    const dim3 grid((unsigned)(((int64_t)L.nbx * G + 127) / 128), (unsigned)((L.nby + gz - 1) / gz), (unsigned)gz);
    CSX_CUDA(launch_if(L.settled, k_block_sweep_q<KIND, T, V, VEC>, grid, 128, 0, s, L.g, L.nbx, L.nby, m, G, A, lam, b, x,
                       out, colour, tr, L.settled));
    count_launch();
    return CS_OK;
}
// Columns in whole 16-byte vectors are staged; else pairs, and odd counts one
// or (from eight on, where reading A once for four columns pays) four at a
// time.  1024^2, FP32, 5 columns: 27 us one and 29 four at a time; 19: 101 and 84.  Staging with
// 8- or 4-byte copies was slower (30 columns: 145 us, 87 here).
template <int KIND, typename T>
static cs_status block_sweep_2x2(const Level &L, const T *A, const T *lam, const T *b, const T *x, T *out, int m,
                                 int colour, int tr, cudaStream_t s) {
    constexpr int V = 16 / (int)sizeof(T);
    const uintptr_t al = (uintptr_t)b | (uintptr_t)x | (uintptr_t)out | (m * sizeof(T));
    if (al % 16 == 0) return block_sweep_s<KIND, T>(L, A, lam, b, x, out, m, colour, tr, s);
    if constexpr (sizeof(T) == 4)
        if (al % 8 == 0) return block_sweep_q<KIND, T, 2, true>(L, A, lam, b, x, out, m, colour, tr, s);
    if (m < 8) return block_sweep_q<KIND, T, 1, false>(L, A, lam, b, x, out, m, colour, tr, s);
    return block_sweep_q<KIND, T, V, false>(L, A, lam, b, x, out, m, colour, tr, s);
}

template <typename T>
cs_status launch_block_sweep_m(const Level &L, const T *A, const T *lam, const T *b, const T *x, T *out, int m,
                               int colour, bool transpose, cudaStream_t s) {
    const int tr = transpose ? 1 : 0;
    // (m <= 32 and a 16-byte aligned Lambda: the entry point's limit and the cascade's own array)
    if (L.g.dim == 2 && L.bs == 2)
        return L.kind == STAR ? block_sweep_2x2<STAR, T>(L, A, lam, b, x, out, m, colour, tr, s)
                              : block_sweep_2x2<BOX, T>(L, A, lam, b, x, out, m, colour, tr, s);
    if (sizeof(T) == sizeof(float) && m % 4 == 0 && L.g.dim == 3 && L.bs == 2 && L.nmax * (m / 4) <= 32 &&
        32 % (L.nmax * (m / 4)) == 0 && ((uintptr_t)b | (uintptr_t)x | (uintptr_t)out) % 16 == 0) {
        const int lpn = m / 4, bpw = 32 / (L.nmax * lpn);
        const int64_t warps = (L.nblocks + bpw - 1) / bpw;
        int dev = 0, nsm = 0;
        CSX_CUDA(cudaGetDevice(&dev));
        CSX_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
        const float *Af = reinterpret_cast<const float *>(A), *lf = reinterpret_cast<const float *>(lam);
        const float4 *b4 = reinterpret_cast<const float4 *>(b), *x4 = reinterpret_cast<const float4 *>(x);
        float4 *o4 = reinterpret_cast<float4 *>(out);
        // one wave: as many CTAs as can be resident, so that no partial wave trails the strided loop
#define CSX_BSM4_LAUNCH(DIM, KIND, LPN)                                                                          \
    do {                                                                                                         \
        int per = 0;                                                                                             \
        CSX_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_block_sweep_m4<DIM, KIND, 2, LPN>, 256, 0)); \
        const unsigned grid = (unsigned)std::max<int64_t>(1, std::min<int64_t>((warps + 7) / 8,                 \
                                                                               (int64_t)nsm * std::max(per, 1))); \
        CSX_CUDA(launch_k(k_block_sweep_m4<DIM, KIND, 2, LPN>, grid, 256, 0, s, L.g, L.nbx, L.nby, L.nblocks, Af, lf, b4, x4, o4,  \
                                                                 colour, tr));                                    \
    } while (0)
#define CSX_BSM4(DIM, LPN)                                                                                       \
    do {                                                                                                         \
        if (L.kind == STAR) CSX_BSM4_LAUNCH(DIM, STAR, LPN);                                                     \
        else CSX_BSM4_LAUNCH(DIM, BOX, LPN);                                                                     \
    } while (0)
        if (lpn == 1) CSX_BSM4(3, 1);
        else if (lpn == 2) CSX_BSM4(3, 2);
        else CSX_BSM4(3, 4);
#undef CSX_BSM4
#undef CSX_BSM4_LAUNCH
        CSX_CUDA(cudaGetLastError());
        count_launch();
        return CS_OK;
    }
#define CSX_BSM(DIM, KIND, BS, BPC)                                                                              \
    CSX_CUDA(launch_k(k_block_sweep_m<DIM, KIND, T, BS, BPC>,                                                    \
                      dim3((unsigned)((L.nbx + BPC - 1) / BPC), (unsigned)L.nby, (unsigned)L.nbz),               \
                      32 * (DIM == 3 ? BS * BS * BS : BS * BS) * BPC, 0, s, L.g, L.nbx, A, lam, b, x, out, m,    \
                      colour, tr));
    if (L.g.dim == 2) {
        if (L.bs == 1) { if (L.kind == STAR) { CSX_BSM(2, STAR, 1, 8) } else { CSX_BSM(2, BOX, 1, 8) } }
        else { if (L.kind == STAR) { CSX_BSM(2, STAR, 3, 1) } else { CSX_BSM(2, BOX, 3, 1) } }
    } else {
        if (L.bs == 1) { if (L.kind == STAR) { CSX_BSM(3, STAR, 1, 8) } else { CSX_BSM(3, BOX, 1, 8) } }
        else { if (L.kind == STAR) { CSX_BSM(3, STAR, 2, 1) } else { CSX_BSM(3, BOX, 2, 1) } }
    }
#undef CSX_BSM
    CSX_CUDA(cudaGetLastError());
    count_launch();
    return CS_OK;
}
template cs_status launch_block_sweep_m<double>(const Level &, const double *, const double *, const double *,
                                                const double *, double *, int, int, bool, cudaStream_t);
template cs_status launch_block_sweep_m<float>(const Level &, const float *, const float *, const float *,
                                               const float *, float *, int, int, bool, cudaStream_t);

// rc_I = 2^-dim sum_f P_{f,I} (A x - b)_f.  Coarse node I sits on fine node
// 2I+1 (0-based); its fine neighbours 2I+1+d (d in {-1,0,1}) carry weight
// 1/2 per nonzero component of d (bilinear / trilinear interpolation).
template <int DIM, int KIND, typename T>
__global__ void __launch_bounds__(TBX *TBY) k_res_restrict(Grid gf, Grid gc, const T *__restrict__ A,
                                                            const T *b, const T *x,
                                                            T *__restrict__ rc) {
    pdl_trigger();
    pdl_wait();
    int cx = blockIdx.x * TBX + threadIdx.x;
    int cy = blockIdx.y * TBY + threadIdx.y;
    int cz = blockIdx.z;
    if (cx >= gc.nx || cy >= gc.ny) return;
    using C = typename AccT<T>::type;
    C acc = C(0);
    const int zlo = DIM == 3 ? -1 : 0, zhi = DIM == 3 ? 1 : 0;
    for (int dz = zlo; dz <= zhi; ++dz) {
        int fz = DIM == 3 ? 2 * cz + 1 + dz : 0;
        if (DIM == 3 && fz >= gf.nz) continue;
        for (int dy = -1; dy <= 1; ++dy) {
            int fy = 2 * cy + 1 + dy;
            if (fy >= gf.ny) continue;
#pragma unroll
            for (int dx = -1; dx <= 1; ++dx) {
                int fx = 2 * cx + 1 + dx;
                if (fx >= gf.nx) continue;
                C w = C((dx ? 0.5 : 1.0) * (dy ? 0.5 : 1.0) * (dz ? 0.5 : 1.0));
                int64_t f = fx + (int64_t)gf.nx * (fy + (int64_t)gf.ny * fz);
                C r = apply_row<DIM, KIND, T>(gf, A, x, fx, fy, fz, f) - ld<T>(b[f]);
                acc = fma(w, r, acc);
            }
        }
    }
    rc[cx + (int64_t)gc.nx * (cy + (int64_t)gc.ny * cz)] = st<T>(acc * C(DIM == 3 ? 0.125 : 0.25));
}

// Two-pass form of the same restriction for FP32 / FP64 storage: every fine
// residual (A x - b)_f once into a fine-level scratch vector, then each
// coarse node gathers its 3^dim window from it in the one-pass kernel's
// order.  The one-pass kernel recomputes a fine residual for each of the up
// to 2^dim coarse nodes whose window holds it; on 256^3 it ran at a third of
// the fine level's bandwidth.  FP64 residuals of 3D levels take repeated rows
// from the parameters, as k_sweep does (FP32 ones of large levels march,
// k_sweep_rep4): with the restriction 23.6 -> 21.8 us on the 27-point 63^3
// level of 127^3, 125 -> 118 on 128^3, 49.3 -> 48.3 and 343 -> 344 on the
// 7-point levels of 127^3 and 256^3, which the FP64 pipe bounds.
struct NoRep {};
template <int DIM, int KIND, typename T>
using FineRep = std::conditional_t<DIM == 3 && std::is_same<T, double>::value, Rep<T, Sten<DIM, KIND>::NST>, NoRep>;
template <int DIM, int KIND, typename T>
static FineRep<DIM, KIND, T> fine_rep(const Level &L) {
    if constexpr (std::is_same<FineRep<DIM, KIND, T>, NoRep>::value) return {};
    else return make_rep<T, Sten<DIM, KIND>::NST>(L, nullptr);
}
__device__ __forceinline__ bool rep_row(const NoRep &, int, int, int) { return false; }
template <typename T>
__device__ __forceinline__ void rep_coeff(const NoRep &, T *) {}
template <typename T, int NST>
__device__ __forceinline__ void rep_coeff(const Rep<T, NST> &rep, T *a) {
#pragma unroll
    for (int s = 0; s < NST; ++s) a[s] = rep.a[s];
}
template <int DIM, int KIND, typename T, bool SYM = false>
__global__ void __launch_bounds__(TBX *TBY) k_fine_residual(Grid g, const T *__restrict__ A, const T *b,
                                                             const T *x, T *__restrict__ r, int settled,
                                                             const __grid_constant__ FineRep<DIM, KIND, T> rep) {
    pdl_trigger();
    if (!settled) pdl_wait();
    const int ix = blockIdx.x * TBX + threadIdx.x, iy = blockIdx.y * TBY + threadIdx.y, iz = blockIdx.z;
    const bool in = ix < g.nx && iy < g.ny;
    const int64_t i = ix + (int64_t)g.nx * (iy + (int64_t)g.ny * iz);
    T a[Sten<DIM, KIND>::NST];
    if (in) {
        if (rep_row(rep, ix, iy, iz)) rep_coeff(rep, a);
        else load_coeff<DIM, KIND, T, SYM>(g, A, ix, iy, iz, i, a);
    }
    if (settled) pdl_wait();
    if (in) r[i] = apply_coeff<DIM, KIND, T>(g, a, x, ix, iy, iz, i) - b[i];
}

template <int DIM, typename T>
__global__ void __launch_bounds__(TBX *TBY) k_restrict_gather(Grid gf, Grid gc, const T *r,
                                                               T *__restrict__ rc) {
    pdl_trigger();
    pdl_wait();
    const int cx = blockIdx.x * TBX + threadIdx.x, cy = blockIdx.y * TBY + threadIdx.y, cz = blockIdx.z;
    if (cx >= gc.nx || cy >= gc.ny) return;
    T acc = T(0);
    const int zlo = DIM == 3 ? -1 : 0, zhi = DIM == 3 ? 1 : 0;
    for (int dz = zlo; dz <= zhi; ++dz) {
        const int fz = DIM == 3 ? 2 * cz + 1 + dz : 0;
        if (DIM == 3 && fz >= gf.nz) continue;
        for (int dy = -1; dy <= 1; ++dy) {
            const int fy = 2 * cy + 1 + dy;
            if (fy >= gf.ny) continue;
#pragma unroll
            for (int dx = -1; dx <= 1; ++dx) {
                const int fx = 2 * cx + 1 + dx;
                if (fx >= gf.nx) continue;
                const T w = T((dx ? 0.5 : 1.0) * (dy ? 0.5 : 1.0) * (dz ? 0.5 : 1.0));
                acc = fma(w, r[fx + (int64_t)gf.nx * (fy + (int64_t)gf.ny * fz)], acc);
            }
        }
    }
    rc[cx + (int64_t)gc.nx * (cy + (int64_t)gc.ny * cz)] = acc * T(DIM == 3 ? 0.125 : 0.25);
}

template <typename T>
cs_status launch_residual_restrict(const Level &f, const Level &c, const T *A, const T *b, const T *x, T *rc,
                                   T *scratch, cudaStream_t s) {
    dim3 gr = node_grid(c.g), bl = node_block();
    if (std::is_same<T, float>::value && f.sym32 && !scratch) {
        set_error("internal: the restriction from a symmetric FP32 level needs a scratch vector");
        return CS_ERR_ARG;
    }
    if constexpr (std::is_same<T, float>::value || std::is_same<T, double>::value) {
        if (scratch) {
            const dim3 gf = node_grid(f.g);
            bool done = false;
            CSX_TRY(try_rep<T, true>(f, A, nullptr, b, x, scratch, nullptr, s, &done));
            if (done) {
                CSX_CUDA(launch_k(k_restrict_gather<3, T>, gr, bl, 0, s, f.g, c.g, scratch, rc));
            } else {
#define CSX_FRES(DIM, KIND, SYM)                                                                                  \
    CSX_CUDA(launch_if(f.settled, k_fine_residual<DIM, KIND, T, SYM>, gf, bl, 0, s, f.g, A, b, x, scratch, f.settled, \
                       fine_rep<DIM, KIND, T>(f)))
                bool sym = false;  // half the couplings
                if constexpr (std::is_same<T, float>::value) {
                    sym = f.sym32 || f.symstar;
                    if (f.sym32) CSX_FRES(3, BOX, true);
                    else if (f.symstar) CSX_FRES(3, STAR, true);
                }
                if (!sym && f.g.dim == 2) {
                    if (f.kind == STAR) CSX_FRES(2, STAR, false);
                    else CSX_FRES(2, BOX, false);
                } else if (!sym) {
                    if (f.kind == STAR) CSX_FRES(3, STAR, false);
                    else CSX_FRES(3, BOX, false);
                }
#undef CSX_FRES
                if (f.g.dim == 2) CSX_CUDA(launch_k(k_restrict_gather<2, T>, gr, bl, 0, s, f.g, c.g, scratch, rc));
                else CSX_CUDA(launch_k(k_restrict_gather<3, T>, gr, bl, 0, s, f.g, c.g, scratch, rc));
            }
            CSX_CUDA(cudaGetLastError());
            count_launch(2);
            return CS_OK;
        }
    }
    if (f.g.dim == 2) {
        if (f.kind == STAR) CSX_CUDA(launch_k(k_res_restrict<2, STAR, T>, gr, bl, 0, s, f.g, c.g, A, b, x, rc));
        else CSX_CUDA(launch_k(k_res_restrict<2, BOX, T>, gr, bl, 0, s, f.g, c.g, A, b, x, rc));
    } else {
        if (f.kind == STAR) CSX_CUDA(launch_k(k_res_restrict<3, STAR, T>, gr, bl, 0, s, f.g, c.g, A, b, x, rc));
        else CSX_CUDA(launch_k(k_res_restrict<3, BOX, T>, gr, bl, 0, s, f.g, c.g, A, b, x, rc));
    }
    CSX_CUDA(cudaGetLastError());
    count_launch();
    return CS_OK;
}
template cs_status launch_residual_restrict<double>(const Level &, const Level &, const double *, const double *,
                                                    const double *, double *, double *, cudaStream_t);
template cs_status launch_residual_restrict<float>(const Level &, const Level &, const float *, const float *,
                                                   const float *, float *, float *, cudaStream_t);
template cs_status launch_residual_restrict<__nv_bfloat16>(const Level &, const Level &, const __nv_bfloat16 *,
                                                           const __nv_bfloat16 *, const __nv_bfloat16 *,
                                                           __nv_bfloat16 *, __nv_bfloat16 *, cudaStream_t);

// 1D interpolation weights of fine node f (0-based) from coarse nodes: an
// odd f coincides with coarse (f-1)/2; an even f takes half of coarse f/2-1
// and f/2 (those inside the coarse grid).
__device__ __forceinline__ int p1d(int f, int nc, int *c, float *w) {
    if (f & 1) {
        c[0] = (f - 1) >> 1; w[0] = 1.f;
        return 1;
    }
    int k = 0, lo = (f >> 1) - 1, hi = f >> 1;
    if (lo >= 0) { c[k] = lo; w[k] = 0.5f; ++k; }
    if (hi < nc) { c[k] = hi; w[k] = 0.5f; ++k; }
    return k;
}

// xo_f = x_f - sum_I P_{f,I} xc_I, one thread per coarse cell: cell j of an
// axis holds the fine nodes 2j (between coarse nodes j - 1 and j, weights
// 1/2, a node outside the grid dropped) and 2j + 1 (on coarse node j, weight
// 1).  The thread loads the cell's up to 2^d coarse corners once, all at
// once, and forms each of its up to 2^d fine nodes with the products in the
// order of the per-node definition (z outer, then y, then x; weight
// wx wy wz rounded once), so every fine value is the one a per-node loop
// gives.  A per-node thread issued its up to 2^d coarse reads one after the
// other and was latency bound.
template <int DIM, typename T>
__global__ void __launch_bounds__(TBX *TBY) k_prolong(Grid gf, Grid gc, const T *xc, const T *x,
                                                       T *xo) {
    pdl_trigger();
    pdl_wait();
    using C = typename AccT<T>::type;
    const int jx = blockIdx.x * TBX + threadIdx.x, jy = blockIdx.y * TBY + threadIdx.y, jz = blockIdx.z;
    if (2 * jx >= gf.nx || 2 * jy >= gf.ny) return;
    // corner d of an axis: coarse node j - 1 (d = 0) or j (d = 1)
    const int cx[2] = {jx - 1, jx}, cy[2] = {jy - 1, jy}, cz[2] = {DIM == 3 ? jz - 1 : 0, DIM == 3 ? jz : 0};
    auto okx = [&](int d) { return cx[d] >= 0 && cx[d] < gc.nx; };
    auto oky = [&](int d) { return cy[d] >= 0 && cy[d] < gc.ny; };
    auto okz = [&](int d) { return DIM == 3 ? (cz[d] >= 0 && cz[d] < gc.nz) : d == 1; };
    C v[2][2][2];
#pragma unroll
    for (int dz = 0; dz < 2; ++dz)
#pragma unroll
        for (int dy = 0; dy < 2; ++dy)
#pragma unroll
            for (int dx = 0; dx < 2; ++dx)
                v[dz][dy][dx] = (okx(dx) && oky(dy) && okz(dz))
                                    ? ld<T>(xc[cx[dx] + (int64_t)gc.nx * (cy[dy] + (int64_t)gc.ny * cz[dz])])
                                    : C(0);
    // fine node e of an axis (0: 2j, 1: 2j + 1) takes corner d when
    // e == 1 ? d == 1 : the corner is inside the grid, with weight 1 or 1/2;
    // the corners run in ascending d, as in the per-node definition
#pragma unroll
    for (int ez = 0; ez < (DIM == 3 ? 2 : 1); ++ez) {
        const int fz = DIM == 3 ? 2 * jz + ez : jz;
        if (fz >= gf.nz) continue;
#pragma unroll
        for (int ey = 0; ey < 2; ++ey) {
            const int fy = 2 * jy + ey;
            if (fy >= gf.ny) continue;
#pragma unroll
            for (int ex = 0; ex < 2; ++ex) {
                const int fx = 2 * jx + ex;
                if (fx >= gf.nx) continue;
                C acc = C(0);
#pragma unroll
                for (int dz = 0; dz < 2; ++dz) {
                    const bool uz = DIM == 3 ? (ez == 1 ? dz == 1 : okz(dz)) : dz == 1;
                    const float wz = (DIM == 3 && ez == 0) ? 0.5f : 1.f;
                    if (!uz) continue;
#pragma unroll
                    for (int dy = 0; dy < 2; ++dy) {
                        const bool uy = ey == 1 ? dy == 1 : oky(dy);
                        const float wy = ey == 0 ? 0.5f : 1.f;
                        if (!uy) continue;
#pragma unroll
                        for (int dx = 0; dx < 2; ++dx) {
                            const bool ux = ex == 1 ? dx == 1 : okx(dx);
                            const float wx = ex == 0 ? 0.5f : 1.f;
                            if (!ux) continue;
                            acc = fma(C(wx * wy * wz), v[dz][dy][dx], acc);
                        }
                    }
                }
                const int64_t f = fx + (int64_t)gf.nx * (fy + (int64_t)gf.ny * fz);
                xo[f] = st<T>(ld<T>(x[f]) - acc);
            }
        }
    }
}

template <typename T>
cs_status launch_prolong_correct(const Level &f, const Level &c, const T *xc, const T *x, T *xo, cudaStream_t s) {
    const int cxn = (f.g.nx + 1) / 2, cyn = (f.g.ny + 1) / 2, czn = f.g.dim == 3 ? (f.g.nz + 1) / 2 : f.g.nz;
    dim3 gr((unsigned)((cxn + TBX - 1) / TBX), (unsigned)((cyn + TBY - 1) / TBY), (unsigned)czn), bl = node_block();
    if (f.g.dim == 2) CSX_CUDA(launch_k(k_prolong<2, T>, gr, bl, 0, s, f.g, c.g, xc, x, xo));
    else CSX_CUDA(launch_k(k_prolong<3, T>, gr, bl, 0, s, f.g, c.g, xc, x, xo));
    CSX_CUDA(cudaGetLastError());
    count_launch();
    return CS_OK;
}
template cs_status launch_prolong_correct<double>(const Level &, const Level &, const double *, const double *,
                                                  double *, cudaStream_t);
template cs_status launch_prolong_correct<float>(const Level &, const Level &, const float *, const float *,
                                                 float *, cudaStream_t);
template cs_status launch_prolong_correct<__nv_bfloat16>(const Level &, const Level &, const __nv_bfloat16 *,
                                                         const __nv_bfloat16 *, __nv_bfloat16 *, cudaStream_t);

// block-wide deterministic sum (fixed tree order)
__device__ __forceinline__ double block_sum(double v, double *sm) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    int lane = (threadIdx.x + threadIdx.y * blockDim.x) & 31;
    int warp = (threadIdx.x + threadIdx.y * blockDim.x) >> 5;
    int nw = (blockDim.x * blockDim.y + 31) >> 5;
    if (lane == 0) sm[warp] = v;
    __syncthreads();
    double t = 0.0;
    if (warp == 0) {
        t = lane < nw ? sm[lane] : 0.0;
        for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
    }
    return t;
}

__device__ __forceinline__ float block_sum_f(float v, float *sm) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    int lane = (threadIdx.x + threadIdx.y * blockDim.x) & 31;
    int warp = (threadIdx.x + threadIdx.y * blockDim.x) >> 5;
    int nw = (blockDim.x * blockDim.y + 31) >> 5;
    if (lane == 0) sm[warp] = v;
    __syncthreads();
    float t = 0.f;
    if (warp == 0) {
        t = lane < nw ? sm[lane] : 0.f;
        for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
    }
    return t;
}

// r = b - A x in FP64; per-block partial sums of r^2 into red[block id],
// summed in FP64 or (N32: for a convergence test only, where the FP64 adds
// of the block tree would cost as much as the residual) in FP32
template <int DIM, int KIND, typename TL = float, bool N32 = false>
__global__ void __launch_bounds__(TBX *TBY) k_residual64(Grid g, const double *__restrict__ A,
                                                          const double *b, const double *x,
                                                          double *__restrict__ r, TL *__restrict__ r32,
                                                          double *__restrict__ red) {
    pdl_trigger();
    pdl_wait();
    __shared__ double sm[32];
    __shared__ float smf[32];
    int ix = blockIdx.x * TBX + threadIdx.x;
    int iy = blockIdx.y * TBY + threadIdx.y;
    int iz = blockIdx.z;
    double v = 0.0;
    if (ix < g.nx && iy < g.ny) {
        int64_t i = ix + (int64_t)g.nx * (iy + (int64_t)g.ny * iz);
        v = b[i] - apply_row<DIM, KIND, double>(g, A, x, ix, iy, iz, i);
        if (r) r[i] = v;
        if (r32) r32[i] = st<TL>((typename AccT<TL>::type)v);
    }
    if (red) {
        double t;
        if (N32) {
            const float vf = (float)v;
            t = (double)block_sum_f(vf * vf, smf);
        } else {
            t = block_sum(v * v, sm);
        }
        if (threadIdx.x == 0 && threadIdx.y == 0)
            red[blockIdx.x + gridDim.x * (blockIdx.y + (int64_t)gridDim.y * blockIdx.z)] = t;
    }
}

// The block sums of a value per thread and plane: each plane's in FP32, in the
// tree of block_sum_f, the planes' in FP64.  The lanes trade planes on the way
// (a lane keeps two of the four, then one), so the tree takes six shuffles,
// one more than that of a single plane; the FP64 additions go in pairs, since
// the CTA ends with them (a refinement iteration on 256^3: 1021.7 us with one
// after the other, 1019.4 in pairs, 1016.9 with all four planes in FP32).  The
// result is thread 0's.
__device__ __forceinline__ double block_sum_planes(const float (&v)[RZ], float *sm) {
    static_assert(RZ == 4 && TBX * TBY == 256, "four planes, eight warps");
    const int tid = threadIdx.x + TBX * threadIdx.y, lane = tid & 31, warp = tid >> 5;
    const bool h16 = lane & 16, h8 = lane & 8;
    const float p = (h16 ? v[2] : v[0]) + __shfl_xor_sync(0xffffffffu, h16 ? v[0] : v[2], 16);
    const float q = (h16 ? v[3] : v[1]) + __shfl_xor_sync(0xffffffffu, h16 ? v[1] : v[3], 16);
    float t = (h8 ? q : p) + __shfl_xor_sync(0xffffffffu, h8 ? p : q, 8);  // plane lane / 8
    for (int o = 4; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if ((lane & 7) == 0) sm[lane + warp] = t;  // [plane][warp]
    __syncthreads();
    double sum = 0.0;
    if (warp == 0) {
        t = sm[lane];
        for (int o = 4; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        sum = (double)t;
        sum += __shfl_xor_sync(0xffffffffu, sum, 8);
        sum += __shfl_xor_sync(0xffffffffu, sum, 16);
    }
    return sum;
}

// The same residual on a 3D level with a box of repeated rows (see
// k_sweep_rep): in the box only x, b and the outputs move, 20 B per node with
// an FP32 output where the general kernel moves 76.  Bound by the FP64 pipe
// then (8 operations per 7-point node).  The FP32 norm adds as many squares
// before FP64 takes over as the general kernel's, a CTA's of one plane.
template <int KIND, typename TL, bool N32>
__global__ void __launch_bounds__(TBX *TBY) k_residual64_rep(Grid g, const double *__restrict__ A,
                                                              const double *b,
                                                              const double *x, double *__restrict__ r,
                                                              TL *__restrict__ r32, double *__restrict__ red,
                                                              const __grid_constant__ Rep<double, Sten<3, KIND>::NST> rep) {
    constexpr int NST = Sten<3, KIND>::NST;
    pdl_trigger();
    pdl_wait();
    __shared__ double sm[32];
    __shared__ float smf[32];
    const int ix = blockIdx.x * TBX + threadIdx.x, iy = blockIdx.y * TBY + threadIdx.y, z0 = blockIdx.z * RZ;
    double v2 = 0.0;
    float v2f[RZ] = {};
    if (ix < g.nx && iy < g.ny) {
        const int64_t pl = (int64_t)g.nx * g.ny;
        int64_t i = ix + (int64_t)g.nx * iy + pl * z0;
        Column<KIND, double> col;
        col.start(g, x, ix, iy, z0, i);
#pragma unroll
        for (int k = 0; k < RZ; ++k, i += pl) {
            const int iz = z0 + k;
            if (iz < g.nz) {
                if (k > 0) col.advance(g, x, ix, iy, iz, i);
                double ax;
                if (rep_row(rep, ix, iy, iz)) {
                    ax = col.apply(rep.a);
                } else {
                    double a[NST];
                    load_row<3, KIND, double>(g, A, i, a);
                    ax = col.apply(a);
                }
                const double v = b[i] - ax;
                if (r) r[i] = v;
                if (r32) r32[i] = st<TL>((typename AccT<TL>::type)v);
                if (N32) v2f[k] = (float)v * (float)v;
                else v2 = fma(v, v, v2);
            }
        }
    }
    if (red) {
        const double t = N32 ? block_sum_planes(v2f, smf) : block_sum(v2, sm);
        if (threadIdx.x == 0 && threadIdx.y == 0)
            red[blockIdx.x + gridDim.x * (blockIdx.y + (int64_t)gridDim.y * blockIdx.z)] = t;
    }
}
static bool rep_residual(const Level &L) { return L.g.dim == 3 && L.cbox && L.g.N >= RZ_MIN_N; }
int residual_ctas(const Level &L) {
    const dim3 g = node_grid(L.g);
    return (int)(g.x * g.y * (rep_residual(L) ? (g.z + RZ - 1) / RZ : g.z));
}
template <typename TL, bool N32>
static cs_status launch_residual64_rep(const Level &L, const double *A, const double *b, const double *x, double *r,
                                       TL *r32, double *red, cudaStream_t s) {
    dim3 gr = node_grid(L.g);
    gr.z = (gr.z + RZ - 1) / RZ;
    if (L.kind == STAR)
        CSX_CUDA(launch_k(k_residual64_rep<STAR, TL, N32>, gr, node_block(), 0, s, L.g, A, b, x, r, r32, red,
                          make_rep<double, 7>(L, nullptr)));
    else
        CSX_CUDA(launch_k(k_residual64_rep<BOX, TL, N32>, gr, node_block(), 0, s, L.g, A, b, x, r, r32, red,
                          make_rep<double, 27>(L, nullptr)));
    count_launch();
    return CS_OK;
}

cs_status launch_residual64(const Level &L, const double *A, const double *b, const double *x, double *r,
                            float *r32, double *red, int nred, cudaStream_t s, bool norm32) {
    dim3 gr = node_grid(L.g), bl = node_block();
    if (red && residual_ctas(L) != nred) {
        set_error("internal: reduction size mismatch");
        return CS_ERR_ARG;
    }
    if (rep_residual(L))
        return norm32 ? launch_residual64_rep<float, true>(L, A, b, x, r, r32, red, s)
                      : launch_residual64_rep<float, false>(L, A, b, x, r, r32, red, s);
    if (norm32) {
        if (L.g.dim == 2) {
            if (L.kind == STAR) CSX_CUDA(launch_k(k_residual64<2, STAR, float, true>, gr, bl, 0, s, L.g, A, b, x, r, r32, red));
            else CSX_CUDA(launch_k(k_residual64<2, BOX, float, true>, gr, bl, 0, s, L.g, A, b, x, r, r32, red));
        } else {
            if (L.kind == STAR) CSX_CUDA(launch_k(k_residual64<3, STAR, float, true>, gr, bl, 0, s, L.g, A, b, x, r, r32, red));
            else CSX_CUDA(launch_k(k_residual64<3, BOX, float, true>, gr, bl, 0, s, L.g, A, b, x, r, r32, red));
        }
    } else if (L.g.dim == 2) {
        if (L.kind == STAR) CSX_CUDA(launch_k(k_residual64<2, STAR>, gr, bl, 0, s, L.g, A, b, x, r, r32, red));
        else CSX_CUDA(launch_k(k_residual64<2, BOX>, gr, bl, 0, s, L.g, A, b, x, r, r32, red));
    } else {
        if (L.kind == STAR) CSX_CUDA(launch_k(k_residual64<3, STAR>, gr, bl, 0, s, L.g, A, b, x, r, r32, red));
        else CSX_CUDA(launch_k(k_residual64<3, BOX>, gr, bl, 0, s, L.g, A, b, x, r, r32, red));
    }
    CSX_CUDA(cudaGetLastError());
    count_launch();
    return CS_OK;
}

__global__ void k_finish_sum(double *red, int n, double *host) {
    pdl_trigger();
    pdl_wait();
    __shared__ double sm[32];
    double v = 0.0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) v += red[i];
    double t = block_sum(v, sm);
    if (threadIdx.x == 0) {
        red[n] = t;
        if (host) *host = t;
    }
}
cs_status launch_finish_sum(double *red, int nred, cudaStream_t s, double *host) {
    CSX_CUDA(launch_k(k_finish_sum, 1, 1024, 0, s, red, nred, host));
    CSX_CUDA(cudaGetLastError());
    count_launch();
    return CS_OK;
}

__global__ void k_loop_in(int64_t N, const double *b, const double *x, double *hb, double *hx, LoopState *st,
                          double tol, int maxit) {
    pdl_trigger();
    pdl_wait();
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i == 0) {
        st->tol = tol;
        st->maxit = maxit;
    }
    if (i >= N) return;
    if (hb != b) hb[i] = b[i];
    if (hx != x) hx[i] = x[i];
}
cs_status launch_loop_in(int64_t N, const double *b, const double *x, double *hb, double *hx, LoopState *st, double tol,
                         int maxit, cudaStream_t s) {
    CSX_CUDA(launch_k(k_loop_in, (unsigned)((N + 255) / 256), 256, 0, s, N, b, x, hb, hx, st, tol, maxit));
    count_launch();
    return CS_OK;
}
// The host loop's tests, in its order and with its roundings.
__global__ void k_loop_decide(int start, LoopState *st, LoopState *host, const double *red, int n,
                              cudaGraphConditionalHandle cond) {
    pdl_trigger();
    pdl_wait();
    __shared__ double sm[32];
    double v = 0.0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) v += red[i];
    const double t = block_sum(v, sm);
    if (threadIdx.x != 0) return;
    if (start) {
        st->nb = sqrt(st->nb2);
        st->it = 0;
        st->nhist = 0;
        st->diverged = 0;
    } else {
        ++st->it;
    }
    const double rel = sqrt(t) / st->nb;
    if (start) st->rel0 = rel;
    else if (!isfinite(rel) || rel > 1e3 * fmax(st->rel0, 1.0)) st->diverged = 1;
    st->rel = rel;
    host->hist[st->nhist++] = rel;
    const bool more = st->nb > 0.0 && rel > st->tol && st->it < st->maxit && !st->diverged && st->nhist < 256;
    if (!more) {
        host->nb = st->nb;
        host->rel = rel;
        host->rel0 = st->rel0;
        host->it = st->it;
        host->diverged = st->diverged;
        host->nhist = st->nhist;
    }
    cudaGraphSetConditional(cond, more ? 1 : 0);
}
cs_status launch_loop_decide(bool start, LoopState *st, LoopState *host, const double *red, int nred,
                             cudaGraphConditionalHandle cond, cudaStream_t s) {
    CSX_CUDA(launch_k(k_loop_decide, 1, 1024, 0, s, start ? 1 : 0, st, host, red, nred, cond));
    count_launch();
    return CS_OK;
}

// One launch of a projection: w -= *hprev * prev (prev given), then
// *dst = <w, v> or, with v == nullptr, <w, w>.  The last CTA to arrive sums
// the CTAs' partials, in the order of k_finish_sum.  A Gram-Schmidt column
// took four launches (dot, its sum, a copy, the update), each shorter than
// its launch on vectors up to 1 M entries.
__global__ void __launch_bounds__(256) k_mgs(int64_t N, double *w, const double *prev,
                                             const double *hprev, const double *v, double *red,
                                             unsigned *ticket, double *dst, double *host) {
    pdl_trigger();
    pdl_wait();
    __shared__ double sm[32];
    __shared__ int last;
    double acc = 0.0;
    if (prev) {
        const double a = -*hprev;
        for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < N; i += (int64_t)gridDim.x * blockDim.x) {
            const double wi = fma(a, prev[i], w[i]);
            w[i] = wi;
            acc = fma(wi, v ? v[i] : wi, acc);
        }
    } else {
        for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < N; i += (int64_t)gridDim.x * blockDim.x) {
            const double wi = w[i];
            acc = fma(wi, v ? v[i] : wi, acc);
        }
    }
    const double t = block_sum(acc, sm);
    if (threadIdx.x == 0) {
        red[blockIdx.x] = t;
        __threadfence();
        last = atomicAdd(ticket, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int gq = warp; gq < 32; gq += 8) {
        const int k = 32 * gq + lane;
        double p = k < (int)gridDim.x ? __ldcg(red + k) : 0.0;
        for (int o = 16; o > 0; o >>= 1) p += __shfl_down_sync(0xffffffffu, p, o);
        if (lane == 0) sm[gq] = p;
    }
    __syncthreads();
    if (warp == 0) {
        double p = sm[lane];
        for (int o = 16; o > 0; o >>= 1) p += __shfl_down_sync(0xffffffffu, p, o);
        if (lane == 0) {
            *dst = p;
            if (host) *host = p;
            *ticket = 0;
        }
    }
}
cs_status launch_mgs(int64_t N, double *w, const double *prev, const double *hprev, const double *v, double *red,
                     unsigned *ticket, double *dst, double *host, cudaStream_t s) {
    const unsigned nb = (unsigned)std::max<int64_t>(1, std::min<int64_t>(NRED, (N + 255) / 256));
    CSX_CUDA(launch_k(k_mgs, nb, 256, 0, s, N, w, prev, hprev, v, red, ticket, dst, host));
    count_launch();
    return CS_OK;
}
cs_status launch_dot(int64_t N, const double *a, const double *b, double *red, unsigned *ticket, double *dst,
                     double *host, cudaStream_t s) {
    return launch_mgs(N, const_cast<double *>(a), nullptr, nullptr, b, red, ticket, dst, host, s);
}

__global__ void k_scale_dev(int64_t N, const double *num, double *y, const double *x) {
    pdl_trigger();
    pdl_wait();
    const double inv = *num > 0.0 ? 1.0 / sqrt(*num) : 1.0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < N; i += (int64_t)gridDim.x * blockDim.x)
        y[i] = x[i] * inv;
}
// y = x / sqrt(*num), or x where *num is 0
cs_status launch_scale_dev(int64_t N, const double *num, double *y, const double *x, cudaStream_t s) {
    CSX_CUDA(launch_k(k_scale_dev, 1216, 256, 0, s, N, num, y, x));
    CSX_CUDA(cudaGetLastError());
    count_launch();
    return CS_OK;
}

// One Arnoldi column in one cooperative launch: w stays in registers through
// all its projections, each V_i is read once (the next one while the grid
// meets for this one's sum) and the normalised vector is written.  As a launch
// per projection, w moved four times and V_i twice, and each waited for a
// launch: 15 columns of right GMRES on 1023^2 took 5.44 ms with the solve's
// cycles, 5.15 here; 18 columns of a general solve on 255^2 4.28 and 3.33.
template <int EPT>
__global__ void __launch_bounds__(256, EPT <= 8 ? 4 : 2) k_arnoldi(int64_t N, const double *V, int j, const double *w,
                                                                 double *out, double *red, double *hd, double *hh) {
    cooperative_groups::grid_group grid = cooperative_groups::this_grid();
    __shared__ double sm[32], total;
    const int64_t T = (int64_t)gridDim.x * 256, g = blockIdx.x * (int64_t)256 + threadIdx.x;
    double wr[EPT], v[EPT], vn[EPT];
    auto load = [&](const double *p, double *r) {
#pragma unroll
        for (int k = 0; k < EPT; ++k) r[k] = g + k * T < N ? p[g + k * T] : 0.0;
    };
    load(w, wr);
    load(V, v);
    for (int i = 0; i <= j + 1; ++i) {
        double acc = 0.0;
#pragma unroll
        for (int k = 0; k < EPT; ++k) acc = fma(wr[k], i <= j ? v[k] : wr[k], acc);
        const double part = block_sum(acc, sm);
        double *r = red + (i & 1) * NRED;  // the other half is still being read
        if (threadIdx.x == 0) r[blockIdx.x] = part;
        if (i < j) load(V + (int64_t)(i + 1) * N, vn);
        grid.sync();
        double q = 0.0;
        for (int k = threadIdx.x; k < (int)gridDim.x; k += 256) q += __ldcg(r + k);
        q = block_sum(q, sm);
        if (threadIdx.x == 0) total = q;
        __syncthreads();
        const double h = total;
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            hd[i] = h;
            hh[i] = h;
        }
        if (i <= j) {
#pragma unroll
            for (int k = 0; k < EPT; ++k) {
                wr[k] = fma(-h, v[k], wr[k]);
                v[k] = vn[k];
            }
        } else {
            const double inv = h > 0.0 ? 1.0 / sqrt(h) : 1.0;
#pragma unroll
            for (int k = 0; k < EPT; ++k)
                if (g + k * T < N) out[g + k * T] = wr[k] * inv;
        }
    }
}
// CTAs of k_arnoldi<EPT> that fit the current device at once (at most NRED)
template <int EPT>
static int arnoldi_ctas(int dev, int nsm) {
    static std::atomic<int> per[64];  // a constant of the device and the kernel; 0: not asked yet
    int p = per[dev].load(std::memory_order_relaxed);
    if (p == 0) {
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&p, k_arnoldi<EPT>, 256, 0) != cudaSuccess) p = -1;
        per[dev].store(p, std::memory_order_relaxed);
    }
    return std::min(NRED, std::max(0, p) * nsm);
}
template <int EPT>
static bool try_arnoldi(int dev, int nsm, int per_sm, int64_t N, const double *V, int j, double *w, double *out,
                        double *red, double *hd, double *hh, cudaStream_t s, cudaError_t *e) {
    const int ctas = (int)((N + 256 * EPT - 1) / (256 * EPT));
    if (ctas > std::min(arnoldi_ctas<EPT>(dev, nsm), per_sm * nsm)) return false;
    const double *wc = w;
    void *args[] = {&N, &V, &j, &wc, &out, &red, &hd, &hh};
    *e = cudaLaunchCooperativeKernel((const void *)k_arnoldi<EPT>, dim3((unsigned)ctas), dim3(256), args, 0, s);
    return true;
}
cs_status orthogonalise(int64_t N, const double *V, int j, double *w, double *out, double *red, unsigned *ticket,
                        double *hd, double *hh, cudaStream_t s) {
    int dev = 0, nsm = 0;
    CSX_CUDA(cudaGetDevice(&dev));
    CSX_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
    cudaError_t e = cudaSuccess;
    // as few CTAs as hold the vector: the meetings of the grid are the cost.
    // 1.2 M values fit the chip's registers; longer vectors take a launch per
    // projection, which moves them at the memory's rate
    if (dev < 64 && N <= (int64_t)NRED * 256 * 8 &&
        (try_arnoldi<2>(dev, nsm, 1, N, V, j, w, out, red, hd, hh, s, &e) ||
         try_arnoldi<4>(dev, nsm, 1, N, V, j, w, out, red, hd, hh, s, &e) ||
         try_arnoldi<8>(dev, nsm, 4, N, V, j, w, out, red, hd, hh, s, &e))) {
        CSX_CUDA(e);
        count_launch();
        return CS_OK;
    }
    for (int i = 0; i <= j + 1; ++i)
        CSX_TRY(launch_mgs(N, w, i > 0 ? V + (int64_t)(i - 1) * N : nullptr, i > 0 ? hd + i - 1 : nullptr,
                           i <= j ? V + (int64_t)i * N : nullptr, red, ticket, hd + i, hh + i, s));
    return launch_scale_dev(N, hd + j + 1, out, w, s);
}

// r = b - A x in FP64, stored in BF16 for the cycle (no reduction)
cs_status launch_residual64_bf16(const Level &L, const double *A, const double *b, const double *x,
                                 __nv_bfloat16 *r16, cudaStream_t s) {
    dim3 gr = node_grid(L.g), bl = node_block();
    if (rep_residual(L)) return launch_residual64_rep<__nv_bfloat16, false>(L, A, b, x, nullptr, r16, nullptr, s);
    if (L.g.dim == 2) {
        if (L.kind == STAR) CSX_CUDA(launch_k(k_residual64<2, STAR, __nv_bfloat16>, gr, bl, 0, s, L.g, A, b, x, nullptr, r16, nullptr));
        else CSX_CUDA(launch_k(k_residual64<2, BOX, __nv_bfloat16>, gr, bl, 0, s, L.g, A, b, x, nullptr, r16, nullptr));
    } else {
        if (L.kind == STAR) CSX_CUDA(launch_k(k_residual64<3, STAR, __nv_bfloat16>, gr, bl, 0, s, L.g, A, b, x, nullptr, r16, nullptr));
        else CSX_CUDA(launch_k(k_residual64<3, BOX, __nv_bfloat16>, gr, bl, 0, s, L.g, A, b, x, nullptr, r16, nullptr));
    }
    CSX_CUDA(cudaGetLastError());
    count_launch();
    return CS_OK;
}
__global__ void k_axpy_bf16(int64_t N, const __nv_bfloat16 *d, double *__restrict__ x) {
    pdl_trigger();
    pdl_wait();
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < N; i += (int64_t)gridDim.x * blockDim.x)
        x[i] += (double)__bfloat162float(d[i]);
}
cs_status launch_axpy_bf16(int64_t N, const __nv_bfloat16 *d, double *x, cudaStream_t s) {
    CSX_CUDA(launch_k(k_axpy_bf16, 1216, 256, 0, s, N, d, x));
    CSX_CUDA(cudaGetLastError());
    count_launch();
    return CS_OK;
}
__global__ void k_d2bf(int64_t N, const double *a, __nv_bfloat16 *__restrict__ o) {
    pdl_trigger();
    pdl_wait();
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < N; i += (int64_t)gridDim.x * blockDim.x)
        o[i] = __double2bfloat16(a[i]);
}
cs_status launch_copy_d2bf(int64_t N, const double *a, __nv_bfloat16 *o, cudaStream_t s) {
    CSX_CUDA(launch_k(k_d2bf, 1216, 256, 0, s, N, a, o));
    CSX_CUDA(cudaGetLastError());
    count_launch();
    return CS_OK;
}

__global__ void k_axpy_f32(int64_t N, const float *d, double *__restrict__ x) {
    pdl_trigger();
    pdl_wait();
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < N; i += (int64_t)gridDim.x * blockDim.x)
        x[i] += (double)d[i];
}
cs_status launch_axpy_f32(int64_t N, const float *d, double *x, cudaStream_t s) {
    CSX_CUDA(launch_k(k_axpy_f32, 1216, 256, 0, s, N, d, x));
    CSX_CUDA(cudaGetLastError());
    count_launch();
    return CS_OK;
}
__global__ void k_d2f(int64_t N, const double *a, float *__restrict__ o) {
    pdl_trigger();
    pdl_wait();
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < N; i += (int64_t)gridDim.x * blockDim.x)
        o[i] = (float)a[i];
}
cs_status launch_copy_d2f(int64_t N, const double *a, float *o, cudaStream_t s) {
    CSX_CUDA(launch_k(k_d2f, 1216, 256, 0, s, N, a, o));
    CSX_CUDA(cudaGetLastError());
    count_launch();
    return CS_OK;
}

__global__ void k_f2d(int64_t N, const float *a, double *__restrict__ o) {
    pdl_trigger();
    pdl_wait();
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < N; i += (int64_t)gridDim.x * blockDim.x)
        o[i] = 0.0 + (double)a[i];
}
cs_status launch_copy_f2d(int64_t N, const float *a, double *o, cudaStream_t s) {
    CSX_CUDA(launch_k(k_f2d, 1216, 256, 0, s, N, a, o));
    count_launch();
    return CS_OK;
}
__global__ void k_bf2d(int64_t N, const __nv_bfloat16 *a, double *__restrict__ o) {
    pdl_trigger();
    pdl_wait();
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < N; i += (int64_t)gridDim.x * blockDim.x)
        o[i] = 0.0 + (double)__bfloat162float(a[i]);
}
cs_status launch_copy_bf2d(int64_t N, const __nv_bfloat16 *a, double *o, cudaStream_t s) {
    CSX_CUDA(launch_k(k_bf2d, 1216, 256, 0, s, N, a, o));
    count_launch();
    return CS_OK;
}

// y = A x (FP64)
template <int DIM, int KIND>
__global__ void __launch_bounds__(TBX *TBY) k_matvec64(Grid g, const double *__restrict__ A,
                                                        const double *x, double *__restrict__ y) {
    pdl_trigger();
    pdl_wait();
    int ix = blockIdx.x * TBX + threadIdx.x, iy = blockIdx.y * TBY + threadIdx.y, iz = blockIdx.z;
    if (ix >= g.nx || iy >= g.ny) return;
    int64_t i = ix + (int64_t)g.nx * (iy + (int64_t)g.ny * iz);
    y[i] = apply_row<DIM, KIND, double>(g, A, x, ix, iy, iz, i);
}
cs_status launch_matvec64(const Level &L, const double *A, const double *x, double *y, cudaStream_t s) {
    dim3 gr = node_grid(L.g), bl = node_block();
    if (L.g.dim == 2) {
        if (L.kind == STAR) CSX_CUDA(launch_k(k_matvec64<2, STAR>, gr, bl, 0, s, L.g, A, x, y));
        else CSX_CUDA(launch_k(k_matvec64<2, BOX>, gr, bl, 0, s, L.g, A, x, y));
    } else {
        if (L.kind == STAR) CSX_CUDA(launch_k(k_matvec64<3, STAR>, gr, bl, 0, s, L.g, A, x, y));
        else CSX_CUDA(launch_k(k_matvec64<3, BOX>, gr, bl, 0, s, L.g, A, x, y));
    }
    CSX_CUDA(cudaGetLastError());
    count_launch();
    return CS_OK;
}

__global__ void k_add64(int64_t N, const double *d, double *__restrict__ x) {
    pdl_trigger();
    pdl_wait();
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < N; i += (int64_t)gridDim.x * blockDim.x)
        x[i] += d[i];
}
cs_status launch_add64(int64_t N, const double *d, double *x, cudaStream_t s) {
    CSX_CUDA(launch_k(k_add64, 1216, 256, 0, s, N, d, x));
    CSX_CUDA(cudaGetLastError());
    count_launch();
    return CS_OK;
}

// y += alpha_host * x with alpha from device memory slot
__global__ void k_axpy_vec(int64_t N, int m, const double *alpha, const double *V,
                           double *__restrict__ y) {
    pdl_trigger();
    pdl_wait();
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < N; i += (int64_t)gridDim.x * blockDim.x) {
        double s = y[i];
        for (int k = 0; k < m; ++k) s = fma(alpha[k], V[(int64_t)k * N + i], s);
        y[i] = s;
    }
}
// y += sum_k alpha[k] V[k]  (alpha: device array of m values)
cs_status launch_axpy_multi(int64_t N, int m, const double *alpha, const double *V, double *y, cudaStream_t s) {
    CSX_CUDA(launch_k(k_axpy_vec, 1216, 256, 0, s, N, m, alpha, V, y));
    CSX_CUDA(cudaGetLastError());
    count_launch();
    return CS_OK;
}

// x = Cinv b (bottom-level direct solve with the inverse formed at setup):
// one warp per row, FP64
template <typename T>
__global__ void k_coarse_solve(int n, const double *__restrict__ Cinv, const T *b, T *__restrict__ x) {
    pdl_trigger();
    pdl_wait();
    int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    int lane = threadIdx.x & 31;
    if (warp >= n) return;
    double s = 0.0;
    for (int j = lane; j < n; j += 32) s = fma(Cinv[(int64_t)warp * n + j], (double)ld<T>(b[j]), s);
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if (lane == 0) x[warp] = st<T>((typename AccT<T>::type)s);
}
cs_status launch_coarse_solve(const cs_hierarchy *h, const double *b, double *x, cudaStream_t s) {
    int threads = 256, blocks = (h->cn * 32 + threads - 1) / threads;
    CSX_CUDA(launch_k(k_coarse_solve<double>, blocks, threads, 0, s, h->cn, h->cinv, b, x));
    CSX_CUDA(cudaGetLastError());
    count_launch();
    return CS_OK;
}
cs_status launch_coarse_solve32(const cs_hierarchy *h, const float *b, float *x, cudaStream_t s) {
    int threads = 256, blocks = (h->cn * 32 + threads - 1) / threads;
    CSX_CUDA(launch_k(k_coarse_solve<float>, blocks, threads, 0, s, h->cn, h->cinv, b, x));
    CSX_CUDA(cudaGetLastError());
    count_launch();
    return CS_OK;
}

// ------------------------------------ the small levels of a 2D cycle at once
// The zero-guess cycle from the first level of at most TH nodes down to the
// coarsest, in one CTA with a node per thread: smoothing, restriction, the
// dense solve and the way back up, with CTA barriers between the steps and all
// vectors in shared memory; a level's rows come into registers once per
// application.  A launch each, these levels took 2 to 3 us a step whatever
// their size.  Arithmetic and its order are those of the single launches.
// A stationary FP64 solve on 64^2 went from 598 to 555 us, right GMRES on
// 1023^2 with FP32 cycles from 5.15 to 5.01 ms.
template <typename T, int TH>
__global__ void __launch_bounds__(TH) k_tail2d(const __grid_constant__ Tail2d<T> q) {
    constexpr int PAD = tail_pad<T>();
    __shared__ T xs[2][PAD], sb[PAD], sx[PAD];
    const int tid = threadIdx.x;
    pdl_trigger();
    if (!q.settled) pdl_wait();
    T a[9], lr[4];
    int nx = 0, ny = 0, N = 0, ix = 0, iy = 0, e = 0, sy = 0;
    bool in = false, star = false;
    auto level = [&](int l) {  // the thread's row of level l
        nx = q.nx[l];
        ny = q.ny[l];
        N = nx * ny;
        in = tid < N;
        iy = in ? tid / nx : 0;
        ix = in ? tid - iy * nx : 0;
        sy = nx + 2;
        e = ix + 1 + sy * (iy + 1);
        star = q.kind[l] == STAR;
#pragma unroll
        for (int s = 0; s < 9; ++s) a[s] = in && (s < 5 || !star) ? q.A[l][(int64_t)s * N + tid] : T(0);
#pragma unroll
        for (int k = 0; k < 4; ++k) lr[k] = in && k < q.nu ? q.lam[l][(int64_t)k * N + tid] : T(0);
    };
    auto apply = [&](const T *x) {
        T ax = T(0);
        if (star) {
            ax = fma(a[0], x[e], ax);
            ax = fma(a[1], x[e - 1], ax);
            ax = fma(a[2], x[e + 1], ax);
            ax = fma(a[3], x[e - sy], ax);
            ax = fma(a[4], x[e + sy], ax);
        } else {
#pragma unroll
            for (int s = 0; s < 9; ++s) ax = fma(a[s], x[e + s % 3 - 1 + sy * (s / 3 - 1)], ax);
        }
        return ax;
    };
    int cur = 0;
    auto smooth = [&](T b, bool reverse) {  // one application on xs[cur]; its border is zero
        const int H = q.nu * q.ncol;
        for (int st = 0; st < H; ++st) {
            const int step = st / q.ncol, lv = reverse ? q.nu - 1 - step : step;
            const int colour = q.ncol == 2 ? (reverse ? 1 - (st & 1) : st & 1) : -1;
            T li = lr[0];
#pragma unroll
            for (int k = 1; k < 4; ++k)
                if (k == lv) li = lr[k];
            if (in) {
                const T xc = xs[cur][e];
                xs[cur ^ 1][e] = colour >= 0 && node_colour(2, ix, iy, 0) != colour ? xc : xc - li * (apply(xs[cur]) - b);
            }
            cur ^= 1;
            __syncthreads();
        }
    };
    auto clear = [&]() {
        __syncthreads();  // the previous level's values have been read
        for (int k = tid; k < PAD; k += TH) xs[0][k] = xs[1][k] = T(0);
        cur = 0;
        __syncthreads();
    };
    level(0);
    if (q.settled) pdl_wait();
    if (in) sb[tid] = q.b[tid];
    for (int l = 0; l + 1 < q.n; ++l) {
        if (l > 0) level(l);
        clear();
        const T b = in ? sb[q.off[l] + tid] : T(0);
        for (int m = 0; m < q.mu_pre; ++m) smooth(b, q.rf != 0);
        if (in) {
            sx[q.off[l] + tid] = xs[cur][e];
            xs[cur ^ 1][e] = apply(xs[cur]) - b;
        }
        __syncthreads();
        const int cnx = q.nx[l + 1], cN = cnx * q.ny[l + 1];
        if (tid < cN) {
            const int cy = tid / cnx, cx = tid - cy * cnx;
            const T *r = xs[cur ^ 1];
            T acc = T(0);
#pragma unroll
            for (int t = 0; t < 9; ++t) {
                const int fx = 2 * cx + t % 3, fy = 2 * cy + t / 3;
                if (fx < nx && fy < ny)
                    acc = fma(T((t % 3 != 1 ? 0.5 : 1.0) * (t / 3 != 1 ? 0.5 : 1.0)), r[fx + 1 + sy * (fy + 1)], acc);
            }
            sb[q.off[l + 1] + tid] = acc * T(0.25);
        }
    }
    __syncthreads();
    for (int w = tid >> 5; w < q.cn; w += TH / 32) {
        const T *b = sb + q.off[q.n - 1];
        double v = 0.0;
        for (int j = tid & 31; j < q.cn; j += 32) v = fma(q.cinv[(int64_t)w * q.cn + j], (double)b[j], v);
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        if ((tid & 31) == 0) sx[q.off[q.n - 1] + w] = (T)v;
    }
    for (int l = q.n - 2; l >= 0; --l) {
        level(l);
        clear();
        if (in) {
            const int cnx = q.nx[l + 1], cny = q.ny[l + 1];
            const T *xc = sx + q.off[l + 1];
            T acc = T(0);
#pragma unroll
            for (int dy = 0; dy < 2; ++dy)
#pragma unroll
                for (int dx = 0; dx < 2; ++dx) {
                    // an odd node sits on coarse node (f - 1) / 2, an even one takes half of f / 2 - 1 and f / 2
                    const int cx = ix & 1 ? (ix - 1) / 2 : ix / 2 - 1 + dx, cy = iy & 1 ? (iy - 1) / 2 : iy / 2 - 1 + dy;
                    if ((ix & 1 && dx == 0) || (iy & 1 && dy == 0) || cx < 0 || cy < 0 || cx >= cnx || cy >= cny) continue;
                    acc = fma(T((ix & 1 ? 1.0 : 0.5) * (iy & 1 ? 1.0 : 0.5)), xc[cx + cnx * cy], acc);
                }
            xs[0][e] = sx[q.off[l] + tid] - acc;
        }
        __syncthreads();
        const T b = in ? sb[q.off[l] + tid] : T(0);
        for (int m = 0; m < q.mu_post; ++m) smooth(b, false);
        if (in) {
            if (l > 0) sx[q.off[l] + tid] = xs[cur][e];
            else q.x[tid] = xs[cur][e];
        }
    }
}
template <typename T>
cs_status launch_tail2d(const Tail2d<T> &q, cudaStream_t s) {
    constexpr int TH = tail_nodes<T>();
    CSX_CUDA(launch_if(q.settled != 0, k_tail2d<T, TH>, 1, TH, 0, s, q));
    count_launch();
    return CS_OK;
}
template cs_status launch_tail2d<double>(const Tail2d<double> &, cudaStream_t);
template cs_status launch_tail2d<float>(const Tail2d<float> &, cudaStream_t);
cs_status launch_coarse_solve16(const cs_hierarchy *h, const __nv_bfloat16 *b, __nv_bfloat16 *x, cudaStream_t s) {
    int threads = 256, blocks = (h->cn * 32 + threads - 1) / threads;
    CSX_CUDA(launch_k(k_coarse_solve<__nv_bfloat16>, blocks, threads, 0, s, h->cn, h->cinv, b, x));
    CSX_CUDA(cudaGetLastError());
    count_launch();
    return CS_OK;
}

}  // namespace csx
