// Internal declarations of the cascading-smoother multigrid library.
// Device data layout (HBM):
//   * every level stores its operator as structure-of-arrays stencil
//     coefficients A[s*N + i] (no index arrays: columns are implicit in the
//     structured grid); the canonical stencil of a level is either STAR
//     (2*dim+1 entries: C,-x,+x,-y,+y[,-z,+z]) or BOX (3^dim entries,
//     s = (dx+1) + 3(dy+1) + 9(dz+1));
//   * Lambda of a point-block cascade is one FP64 value per node per step,
//     lam[l*N + i]; FP32 copies sit beside it for low-precision cycles;
//   * vectors are contiguous N-arrays in natural (x fastest) order.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <atomic>
#include <cstdint>
#include <string>
#include <utility>
#include <vector>

#include "../../include/cascade_mg.h"

namespace csx {

enum StencilKind { STAR = 0, BOX = 1 };

struct Grid {
    int dim;
    int nx, ny, nz;
    int64_t N;
};

struct Level {
    Grid g;
    int kind = STAR;
    int nst = 0;
    int off[27][3];
    double *A = nullptr;  // [nst][N]
    // work vectors (FP64): b (rhs), x (iterate), t (ping-pong)
    double *b = nullptr, *x = nullptr, *t = nullptr;
    // every row at boundary distance >= margin has a coefficient row equal
    // (bitwise) to the grid-centre row; NO_MARGIN: no such region is used
    int margin = NO_MARGIN;
    static constexpr int NO_MARGIN = 1 << 30;
    // block partition: blocks of bs^dim nodes (partial at the upper edges),
    // block (bx,by,bz) = nodes bs*b .. bs*b+bs-1 per axis; nmax = bs^dim.
    // Lambda of a block level is stored [nu][nblocks][nmax][nmax] over the
    // local positions lp = lx + bs (ly + bs lz); absent positions are zero.
    int bs = 1, nbx = 0, nby = 0, nbz = 0, nmax = 1;
    int64_t nblocks = 0;
    // a 3D 27-point point-block level whose operator is symmetric (to 1e-12
    // of the diagonals): its FP32 copies keep the centre and the 13 forward
    // couplings only, [14][N] (entry k = 27-point entry 13 + k); a backward
    // coupling is the forward one stored at the neighbour
    int sym32 = 0;
    // a 3D 7-point point-block level whose operator is symmetric in FP32 (the
    // two couplings of a pair of nodes round to the same number): FP32 steps
    // read the centre and the three forward couplings, and a backward one from
    // the neighbour's row
    int symstar = 0;
    // the operator (and the Lambda of its cascades) belongs to a handle whose
    // setup has been waited for: no kernel of any stream writes it, so the
    // smoothing kernels may read it before their pdl_wait()
    int settled = 0;
    // box of rows (inclusive, per axis) whose couplings to nodes inside the
    // grid all equal (bitwise) the grid-centre row's, crow in the level's
    // stencil order; cbox = 0: no such box of at least half the rows
    int cbox = 0;
    int clo[3] = {0, 0, 0}, chi[3] = {0, 0, 0};
    double crow[27] = {0};
};

// Rows of a cascade step at boundary distance >= dist hold the Lambda of a
// representative row of their colour (NO_MARGIN: nothing is known)
struct LamDeep {
    int dist = Level::NO_MARGIN;
    int rep[2] = {0, 0};
};

// entries per node of a level's FP32 operator copy
inline int64_t lo_nst(const Level &L) { return L.sym32 ? 14 : L.nst; }

struct LowLevel {   // FP32 state of one level (owned by a cascade)
    float *A = nullptr;    // [nst][N]
    float *lam = nullptr;  // [nu][N]
    float *b = nullptr, *x = nullptr, *t = nullptr;
};

struct LowLevel16 {  // BF16 storage of one level (FP32 arithmetic; owned by a cascade)
    __nv_bfloat16 *A = nullptr;    // [nst][N]
    __nv_bfloat16 *lam = nullptr;  // [nu][N]
    __nv_bfloat16 *b = nullptr, *x = nullptr, *t = nullptr;
};

}  // namespace csx

namespace csx {
// A stationary solve whose loop runs on the device.  The host's copy receives
// the state and the residual history of a launch.
struct LoopState {
    double tol, nb2, nb, rel, rel0;
    int maxit, it, diverged, nhist;
    double hist[256];
};
}  // namespace csx

struct cs_hierarchy {
    int dim = 0;
    int nlev = 0;
    bool periodic = false;
    std::vector<csx::Level> lev;
    int cn = 0;                 // coarsest size
    double *cinv = nullptr;     // dense inverse of the coarsest operator, row-major
    double *fine_r = nullptr;   // FP64 residual scratch, finest level
    double *red = nullptr;      // reduction partials
    double *red_host = nullptr; // pinned host mirror of the reduction result
    unsigned *ticket = nullptr; // zeroed counter of the single-launch reductions
    double *hb = nullptr, *hx = nullptr; // device copies for host-buffer solves and solves in one graph
    csx::LoopState *loop = nullptr;      // device and pinned host state of a solve in one graph
    csx::LoopState *loop_host = nullptr;
    int64_t bytes = 0;
};

struct cs_cascade {
    cs_hierarchy *h = nullptr;
    int kind = CS_ADDITIVE;
    int nu = 1;
    int ncol = 1;
    int nlev = 0;               // smoothing levels
    bool lowp = false;
    std::vector<double *> lam;  // per level [nu][N]
    std::vector<std::vector<csx::LamDeep>> deep;  // per level and step
    std::vector<csx::LowLevel> lo;
    std::vector<csx::LowLevel16> lo16;  // BF16 copies (lowp = 2, point-block hierarchies)
    float *fine_b32 = nullptr, *fine_x32 = nullptr;
    // captured zero-initial-guess V-cycles, keyed by (precision, order, mu)
    struct Graph {
        int prec, order, mu_pre, mu_post;
        cudaGraphExec_t exec;
        int64_t kernels;
    };
    std::vector<Graph> graphs;
    std::vector<Graph> loops;  // whole stationary solves (kernels: of one iteration)
    cudaStream_t capture_stream = nullptr;
    // GMRES workspace (lazily allocated at first GMRES solve)
    int gm_restart = 0;
    double *gm_V = nullptr, *gm_h = nullptr;
    double *gm_host = nullptr;  // pinned mirror of gm_h's column
    double *gm_Z = nullptr;  // right-preconditioned GMRES: Z_j = M V_j
    int64_t bytes = 0;
    // learned setup of the finest level: 1 used (some blocks predicted), 0
    // fell back to the exact setup, -1 no model; level-1 Frobenius objectives
    // of the prediction and of the Lambda in use, over the exact one; block counts
    int learned_used = -1;
    double learned_ratio = 0.0, learned_ratio_used = 0.0;
    int64_t learned_blocks = 0, learned_full = 0, learned_accepted = 0;
};

namespace csx {

// error handling ----------------------------------------------------------
void set_error(const char *fmt, ...);
cs_status cuda_fail(cudaError_t e, const char *what, const char *file, int line);

#define CSX_CUDA(...)                                                   \
    do {                                                                \
        cudaError_t _e = (__VA_ARGS__);                                 \
        if (_e != cudaSuccess) return csx::cuda_fail(_e, #__VA_ARGS__, __FILE__, __LINE__); \
    } while (0)
// for functions that release their scratch at a `done:` label and return rc
#define CSX_CUDA_GOTO(call)                                             \
    do {                                                                \
        cudaError_t _e = (call);                                        \
        if (_e != cudaSuccess) { rc = csx::cuda_fail(_e, #call, __FILE__, __LINE__); goto done; } \
    } while (0)
#define CSX_TRY(...)                                                    \
    do {                                                                \
        cs_status _s = (__VA_ARGS__);                                   \
        if (_s != CS_OK) return _s;                                     \
    } while (0)

// Programmatic dependent launch: a kernel launched this way may become
// resident while the kernel before it in the stream (or captured graph) is
// still running.  Its threads call pdl_trigger() at once, which lets the
// next one in, load what no kernel of the stream writes (operators and Lambda
// of a finished setup), and then pdl_wait(), which returns when every earlier
// kernel has completed and its writes are visible; only then do they touch
// vectors.  Every kernel launched by launch_k calls pdl_wait(), so that
// completion carries over from kernel to kernel.  Inputs that another kernel
// of the stream may have written are plain pointers in these kernels: through
// a const __restrict__ parameter the compiler may take a load to be invariant
// and move it ahead of the wait.  Only the settled operators and tables, and
// outputs, are __restrict__.  The V-cycle's kernels below
// 128^3 (1024^2 in 2D) run for less time than a launch takes: a stationary
// solve on 64^2 went from 1.11 to 0.79 ms, right GMRES on 1023^2 from 9.66 to
// 7.00 ms, with the same kernels otherwise.
// launch_if: dependent only if `settled`; else it starts after everything ahead
// of it has completed (operators that the caller may just have written).
template <typename... KArgs, typename... Args>
inline cudaError_t launch_if(bool settled, void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem,
                             cudaStream_t s, Args &&...args) {
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = at;
    cfg.numAttrs = settled ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}
template <typename... KArgs, typename... Args>
inline cudaError_t launch_k(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                            Args &&...args) {
    return launch_if(true, kernel, grid, block, smem, s, std::forward<Args>(args)...);
}
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

extern std::atomic<int64_t> g_launches;
inline void count_launch(int64_t n = 1) { g_launches.fetch_add(n, std::memory_order_relaxed); }

// Device memory comes from a library-owned stream-ordered pool per device
// (cudaMallocFromPoolAsync / cudaFreeAsync) that keeps freed memory mapped,
// so repeated setups of multi-GB residual buffers cost no driver calls.
cs_status dalloc(void **p, size_t bytes, int64_t *acct, cudaStream_t s = 0);
void dfree(void *p, cudaStream_t s = 0);
template <typename T>
cs_status dalloc_t(T **p, size_t count, int64_t *acct, cudaStream_t s = 0) {
    return dalloc(reinterpret_cast<void **>(p), count * sizeof(T), acct, s);
}

inline Grid make_grid(int dim, int nx, int ny, int nz) {
    Grid g;
    g.dim = dim; g.nx = nx; g.ny = ny; g.nz = dim == 3 ? nz : 1;
    g.N = (int64_t)g.nx * g.ny * g.nz;
    return g;
}

// The rows a reuse-enabled kernel computes: the grid minus an inner box of
// deep rows (lo..hi inclusive per axis), enumerated densely so that warps
// hold only rows with work, followed by nrep representative rows.
struct RowSet {
    int on;
    int lo[3], hi[3];
    int64_t nshell;
    int nrep;
    int rep[2][3];
};

inline int64_t rowset_shell_count(const Grid &g, const int *lo, const int *hi) {
    const int64_t nxi = hi[0] - lo[0] + 1, nyi = hi[1] - lo[1] + 1;
    const int64_t nzi = g.dim == 3 ? hi[2] - lo[2] + 1 : 1;
    return g.N - nxi * nyi * nzi;
}

// coordinates of the t-th row of the set; false past its end
__device__ __forceinline__ bool rowset_coord(const RowSet &rs, const Grid &g, int64_t t, int &ix, int &iy, int &iz) {
    if (t >= rs.nshell) {
        const int r = (int)(t - rs.nshell);
        if (r >= rs.nrep) return false;
        ix = rs.rep[r][0]; iy = rs.rep[r][1]; iz = rs.rep[r][2];
        return true;
    }
    const int nxi = rs.hi[0] - rs.lo[0] + 1, nyi = rs.hi[1] - rs.lo[1] + 1;
    const int nxo = g.nx - nxi, nyo = g.ny - nyi;
    int zlo = 0, nzi = 1;
    if (g.dim == 3) {  // whole outer z-planes first
        nzi = rs.hi[2] - rs.lo[2] + 1;
        zlo = rs.lo[2];
        const int64_t plane = (int64_t)g.nx * g.ny;
        const int64_t pz = (int64_t)(g.nz - nzi) * plane;
        if (t < pz) {
            const int k = (int)(t / plane);
            const int64_t rem = t - (int64_t)k * plane;
            iz = k < rs.lo[2] ? k : k + nzi;
            iy = (int)(rem / g.nx);
            ix = (int)(rem - (int64_t)iy * g.nx);
            return true;
        }
        t -= pz;
    }
    const int64_t pery = (int64_t)nyo * g.nx;  // outer y-rows of the inner z-range
    const int64_t py = (int64_t)nzi * pery;
    if (t < py) {
        const int zz = (int)(t / pery);
        const int64_t rem = t - (int64_t)zz * pery;
        const int k = (int)(rem / g.nx);
        iz = zlo + zz;
        iy = k < rs.lo[1] ? k : k + nyi;
        ix = (int)(rem - (int64_t)k * g.nx);
        return true;
    }
    t -= py;  // outer x-columns of the inner y- and z-range
    const int64_t perz = (int64_t)nyi * nxo;
    const int zz = (int)(t / perz);
    const int64_t rem = t - (int64_t)zz * perz;
    const int yy = (int)(rem / nxo);
    const int k = (int)(rem - (int64_t)yy * nxo);
    iz = zlo + zz;
    iy = rs.lo[1] + yy;
    ix = k < rs.lo[0] ? k : k + nxi;
    return true;
}

// launch geometry: one thread per node, x fastest
constexpr int TBX = 64, TBY = 4;
inline dim3 node_grid(const Grid &g) {
    return dim3((unsigned)((g.nx + TBX - 1) / TBX), (unsigned)((g.ny + TBY - 1) / TBY), (unsigned)g.nz);
}
inline dim3 node_block() { return dim3(TBX, TBY, 1); }

// ---- stencil kernels (cs_stencil.cu)
// out = x - lam_l (A x - b) over all nodes (additive step), or over colour
// `colour` only (multiplicative step; other nodes copied when out != x).
template <typename T>
cs_status launch_sweep(const Level &L, const T *A, const T *lam, const T *b, const T *x, T *out,
                       int colour, bool x_is_zero, cudaStream_t s, const LamDeep *deep = nullptr);
// The small 2D levels of a cycle in one launch: n levels from the first with
// at most tail_nodes() nodes to the coarsest, whose dense inverse is cinv.
// FP64, at 1/64 of the FP32 rate, keeps levels of more than 16^2 nodes on
// several SMs.
constexpr int TAIL_LEV = 8;
template <typename T>
constexpr int tail_nodes() {
    return sizeof(T) == 8 ? 256 : 1024;
}
template <typename T>  // nodes of a level with its border, and of all levels together, that shared memory holds
constexpr int tail_pad() {
    return tail_nodes<T>() * 3 / 2;
}
template <typename T>
struct Tail2d {
    int n, nu, ncol, mu_pre, mu_post, rf, cn, settled;
    int nx[TAIL_LEV], ny[TAIL_LEV], kind[TAIL_LEV], off[TAIL_LEV];
    const T *A[TAIL_LEV], *lam[TAIL_LEV];
    const T *b;
    T *x;
    const double *cinv;
};
template <typename T>
cs_status launch_tail2d(const Tail2d<T> &q, cudaStream_t s);
// One whole application of a point cascade on a 2D level in one launch: out
// receives the iterate after nu steps (of ncol colours each) from x; out != x.
// cascade2d_fits: the launch exists for this level, depth and type and beats
// the single steps.
template <typename T>
bool cascade2d_fits(const Level &L, int nu, int ncol);
template <typename T>
cs_status launch_cascade2d(const Level &L, const T *A, const T *lam, const T *b, const T *x, T *out, int nu, int ncol,
                           bool reverse, bool x_is_zero, cudaStream_t s);
// rc = R (A x - b) (full weighting, 2^-dim P^T); with a fine-level scratch
// vector (FP32 / FP64) in two passes, else in one
template <typename T>
cs_status launch_residual_restrict(const Level &f, const Level &c, const T *A, const T *b, const T *x,
                                   T *rc, T *scratch, cudaStream_t s);
template <typename T>
cs_status launch_prolong_correct(const Level &f, const Level &c, const T *xc, const T *x, T *xo,
                                 cudaStream_t s);
// r = b - A x (FP64) with FP64 or FP32-stored coefficients; optional FP32
// copy of r and per-block partial sums of r^2 into red (nblocks entries;
// norm32: the block sums in FP32, enough for a convergence test).
cs_status launch_residual64(const Level &L, const double *A, const double *b, const double *x,
                            double *r, float *r32, double *red, int nred, cudaStream_t s, bool norm32 = false);
// CTAs of launch_residual64 on a level: the partial sums it writes
int residual_ctas(const Level &L);
cs_status launch_coarse_solve(const cs_hierarchy *h, const double *b, double *x, cudaStream_t s);
cs_status launch_coarse_solve32(const cs_hierarchy *h, const float *b, float *x, cudaStream_t s);
cs_status launch_axpy_f32(int64_t N, const float *d, double *x, cudaStream_t s);  // x += d
cs_status launch_copy_d2f(int64_t N, const double *a, float *o, cudaStream_t s);
cs_status launch_copy_d2bf(int64_t N, const double *a, __nv_bfloat16 *o, cudaStream_t s);
cs_status launch_axpy_bf16(int64_t N, const __nv_bfloat16 *d, double *x, cudaStream_t s);  // x += d
cs_status launch_residual64_bf16(const Level &L, const double *A, const double *b, const double *x,
                                 __nv_bfloat16 *r16, cudaStream_t s);
cs_status launch_coarse_solve16(const cs_hierarchy *h, const __nv_bfloat16 *b, __nv_bfloat16 *x, cudaStream_t s);
// sum of red[0..nred) into red[nred] (one block, fixed order), and into pinned host memory if given
cs_status launch_finish_sum(double *red, int nred, cudaStream_t s, double *host = nullptr);
// The parts of a solve in one graph (LoopState): st takes tol and maxit, hb
// and hx copies of b and x; then, after red has the nred partial sums of the
// residual and st->nb2 = <b, b>, `start` or `step` of the loop, which sets the
// condition and writes the host's copy.
cs_status launch_loop_in(int64_t N, const double *b, const double *x, double *hb, double *hx, LoopState *st, double tol,
                         int maxit, cudaStream_t s);
cs_status launch_loop_decide(bool start, LoopState *st, LoopState *host, const double *red, int nred,
                             cudaGraphConditionalHandle cond, cudaStream_t s);
// *dst = <a, b> (and *host, pinned, if given), in one launch; red: NRED
// partials, ticket: a zeroed counter that the launch leaves zero
cs_status launch_dot(int64_t N, const double *a, const double *b, double *red, unsigned *ticket, double *dst,
                     double *host, cudaStream_t s);
// one step of modified Gram-Schmidt in one launch: w -= *hprev * prev (if
// prev), then *dst = <w, v> (v == nullptr: <w, w>)
cs_status launch_mgs(int64_t N, double *w, const double *prev, const double *hprev, const double *v, double *red,
                     unsigned *ticket, double *dst, double *host, cudaStream_t s);
cs_status launch_copy_f2d(int64_t N, const float *a, double *o, cudaStream_t s);
cs_status launch_copy_bf2d(int64_t N, const __nv_bfloat16 *a, double *o, cudaStream_t s);
cs_status launch_scale_dev(int64_t N, const double *num, double *y, const double *x, cudaStream_t s); // y = x / *num
cs_status launch_matvec64(const Level &L, const double *A, const double *x, double *y, cudaStream_t s);
cs_status launch_add64(int64_t N, const double *d, double *x, cudaStream_t s);  // x += d
cs_status launch_axpy_multi(int64_t N, int m, const double *alpha, const double *V, double *y, cudaStream_t s);
constexpr int NRED = 1024;  // partial sums of a reduction
// w against V_0 .. V_j by modified Gram-Schmidt: hd (device) and hh (pinned
// host) receive the j + 1 projections and ||w||^2 after them, out (may be w)
// the normalised vector, or w itself where the norm is 0.  red: 2 NRED values.
cs_status orthogonalise(int64_t N, const double *V, int j, double *w, double *out, double *red, unsigned *ticket,
                        double *hd, double *hh, cudaStream_t s);
// (re)allocates the pinned host column of a Krylov solve
cs_status krylov_host(double **p, int n);

// ---- setup kernels (cs_setup.cu)
cs_status galerkin_level(const Level &f, Level &c, bool reuse, cudaStream_t s);
cs_status level_margin(Level &L, bool periodic, cudaStream_t s);
// zeroes the coefficients of couplings to nodes outside a Dirichlet grid
cs_status drop_outside_couplings(const Level &L, cudaStream_t s);
// sets L.sym32 / L.symstar (3D point-block levels; synchronises the stream)
cs_status check_symmetric(Level &L, cudaStream_t s);
// the FP32 copy of a sym32 level's operator ([14][N])
cs_status launch_copy_box_sym32(const Level &L, float *o, cudaStream_t s);
cs_status coarse_factor(cs_hierarchy *h, cudaStream_t s);
// dense inverse of M (Cholesky, else LU with partial pivoting; W: n x n scratch, piv: n) by one CTA; *status 1: singular
cs_status launch_factor_inverse(int n, double *M, double *W, double *Inv, int *piv, int *status, cudaStream_t s);
// fp32: form the residual rows R and the error propagator E in FP32 (the
// row products summed in FP64 over chunks of 8, or as pairs of FP32 numbers);
// lambda is stored in FP64
cs_status cascade_setup_level(const cs_hierarchy *h, int l, int kind, int nu, int prescale, bool reuse, int alpha,
                              bool fp32, double *lam, cudaStream_t s, int64_t *peak_bytes,
                              std::vector<LamDeep> *deep = nullptr);
cs_status cascade_setup_level_sketch(const cs_hierarchy *h, int l, int kind, int nu, int prescale, int s,
                                     uint64_t seed, int exact_first, bool fp32, double *lam, cudaStream_t st);
cs_status cascade_setup_level_blocks(const cs_hierarchy *h, int l, int kind, int nu, int prescale, int alpha, bool fp32, double *lam,
                                     cudaStream_t s);
cs_status learned_setup_level0(const cs_hierarchy *h, cs_cascade *c, cs_mlp *M, double tol, double *lam,
                               const double *lam_exact1, cudaStream_t s);
// block cascade step (bs > 1): out_b = x_b - Lambda_b^(T) (A x - b)_b over all
// blocks or the blocks of one colour
template <typename T>
cs_status launch_block_sweep(const Level &L, const T *A, const T *lam, const T *b, const T *x, T *out, int colour,
                             bool transpose, bool x_is_zero, cudaStream_t s);
template <>
cs_status launch_block_sweep<__nv_bfloat16>(const Level &, const __nv_bfloat16 *, const __nv_bfloat16 *,
                                            const __nv_bfloat16 *, const __nv_bfloat16 *, __nv_bfloat16 *, int, bool,
                                            bool, cudaStream_t);
// the same with m right-hand sides, vectors RHS-contiguous (X[i*m + r], m <= 32)
template <typename T>
cs_status launch_block_sweep_m(const Level &L, const T *A, const T *lam, const T *b, const T *x, T *out, int m,
                               int colour, bool transpose, cudaStream_t s);

}  // namespace csx
