// Dense BF16 GEMM on the 5th-generation tensor cores (tcgen05) for the
// learned-setup network: C[M x N] (FP32) = A[M x K] B[N x K]^T with A and B
// BF16, K contiguous (row-major A and B, "TN"), FP32 accumulation in tensor
// memory.
//
// One CTA computes a 128 x BN tile of C, BN = 128, or 256 where that fills half
// the SMs (grid
// x: N tiles, y: M tiles, z: K splits).  Operand boxes of 128 rows x 64 BF16
// (128 B per row) are staged by TMA into shared memory with the 128-byte
// swizzle, three or four stages deep; one thread issues the TMA copies and the
// tcgen05.mma instructions (M = 128, N = BN, K = 16 each) and commits each
// stage back to its "empty" barrier; the accumulator lives in BN TMEM
// columns; the warps read it back with
// tcgen05.ld (warp w owns TMEM lanes 32w .. 32w + 31, i.e. rows of C) for the
// epilogue (bias, ReLU, mask, packed copy) or for a split-K partial.
//
// Every wait on an mbarrier is bounded: on expiry the kernel raises *err,
// stops issuing, waits (bounded again) for its copies in flight, frees its
// TMEM and returns; the host reports CS_ERR_TIMEOUT.
//
// FP32 operands enter as BF16 pairs (hi = bf16(x), lo = bf16(x - hi)) laid
// side by side along K, so that one GEMM over the concatenated K forms
// a_hi b_hi + a_lo b_hi + a_hi b_lo: the products of FP32 values to about
// 2^-16 relative (the bf16x3 scheme of Henry, Tang and Heinecke 2019), while
// BF16 weights enter once per segment unsplit.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cudaTypedefs.h>

#include <cstring>
#include <mutex>

#include "cs_internal.cuh"
#include "cs_tcgemm.cuh"

namespace csx {

namespace {

constexpr int TC_BM = 128, TC_BK = 64;  // tile rows; BK: BF16 elements per 128-byte row
// operand stages of a kernel with EW epilogue warps: what the warps' chunks
// leave of the shared memory
template <int BN, int EW>
constexpr int tc_stages() {
    return BN == 256 && EW == 8 ? 3 : 4;
}
constexpr int TC_TILE_BYTES = TC_BM * TC_BK * 2;  // 16 KB: one 128-row operand box
// dynamic shared memory for a tile of BN columns: per stage one A box and
// BN / 128 B boxes, plus alignment and slack
template <int BN, int EW>
constexpr int tc_smem() {
    return tc_stages<BN, EW>() * TC_TILE_BYTES * (1 + BN / 128) + 1024;
}
constexpr long long TC_SPIN = 1ll << 24;  // try_wait rounds before a wait is declared expired

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}

// bounded wait for the phase with the given parity to complete
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity) {
    for (long long it = 0; it < TC_SPIN; ++it) {
        uint32_t ok;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
            : "=r"(ok)
            : "r"(bar), "r"(parity)
            : "memory");
        if (ok) return true;
    }
    return false;
}

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap *map, int x, int y, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
            dst),
        "l"((uint64_t)map), "r"(x), "r"(y), "r"(bar)
        : "memory");
}

// shared-memory matrix descriptor of a K-major tile with the 128-byte
// swizzle: 8-row core groups 1024 B apart (stride byte offset), the leading
// byte offset unused for this layout (1), descriptor version 1 (bits 46-48),
// swizzle mode 2 (128 B) in bits 61-63
__device__ __forceinline__ uint64_t sw128_desc(uint32_t addr) {
    return (uint64_t)((addr & 0x3FFFF) >> 4) | ((uint64_t)1 << 16) | ((uint64_t)(1024 >> 4) << 32) |
           ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}

// instruction descriptor of kind::f16: D F32 (bits 4-5 = 1), A and B BF16
// (bits 7-9, 10-12 = 1), both K-major, N >> 3 in bits 17-22, M >> 4 in 24-28
template <int BN>
constexpr uint32_t tc_idesc() {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(TC_BM >> 4) << 24);
}

__device__ __forceinline__ void mma_bf16(uint32_t tmem_d, uint64_t da, uint64_t db, uint32_t idesc,
                                         uint32_t accumulate) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(tmem_d),
        "l"(da), "l"(db), "r"(idesc), "r"(accumulate)
        : "memory");
}

__device__ __forceinline__ void mma_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float *v) {
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ uint32_t pack_bf16(__nv_bfloat16 a, __nv_bfloat16 b) {
    return (uint32_t)__bfloat16_as_ushort(a) | ((uint32_t)__bfloat16_as_ushort(b) << 16);
}

// the result's hi / lo pairs of four adjacent columns
__device__ __forceinline__ void store_packed4(const TcArgs &a, int row, int n, const float *x) {
    uint32_t hi[2], lo[2];
#pragma unroll
    for (int e = 0; e < 2; ++e) {  // two conversions per instruction
        const __nv_bfloat162 h = __floats2bfloat162_rn(x[2 * e], x[2 * e + 1]);
        const float2 f = __bfloat1622float2(h);
        const __nv_bfloat162 l = __floats2bfloat162_rn(x[2 * e] - f.x, x[2 * e + 1] - f.y);
        hi[e] = pack_bf16(h.x, h.y);
        lo[e] = pack_bf16(l.x, l.y);
    }
    __nv_bfloat16 *h = a.H + (int64_t)row * a.hkw + n;
    *reinterpret_cast<uint2 *>(h) = make_uint2(hi[0], hi[1]);
    *reinterpret_cast<uint2 *>(h + a.hseg) = make_uint2(lo[0], lo[1]);
}
// mask: the mask's value there, 1 without a mask
__device__ __forceinline__ float finish(const TcArgs &a, float mask, float bias, float x) {
    if (a.bias) x += bias;
    if (a.relu) x = fmaxf(x, 0.f);
    return mask > 0.f ? x : 0.f;
}

// A 32 x 32 chunk of sums, one row per lane in v, to its rows row0.. and
// columns n0.. of the result.  It goes through shared memory so that rows
// leave in full 128-byte segments: as float4 with eight lanes to a row, four
// rows per store (vec), else a column per lane and a row per store.  One row
// per store instruction was 32 rounds of a chunk's epilogue; with the
// network's K of 512 that took longer than the products.
constexpr int TC_TS = 36;  // row stride of the chunk: 16-byte rows, conflict-free float4 both ways
__device__ __forceinline__ void store_chunk(const TcArgs &a, float (*tile)[TC_TS], const float *v, float *C, int ldc,
                                            int row0, int n0, int lane) {
#pragma unroll
    for (int i = 0; i < 32; i += 4)
        *reinterpret_cast<float4 *>(&tile[lane][i]) = make_float4(v[i], v[i + 1], v[i + 2], v[i + 3]);
    __syncwarp();
    // the whole chunk is read before the first store: the compiler cannot tell that the stores leave the tile
    // alone, and each read in its turn waited for shared memory
    if (a.vec) {
        const int n = n0 + 4 * (lane & 7);
        const bool on = n < a.N;  // N is a multiple of 4
        float4 x4[8], m4[8];
        float bv[4];
#pragma unroll
        for (int it = 0; it < 8; ++it) {
            const int r = 4 * it + (lane >> 3);
            x4[it] = *reinterpret_cast<const float4 *>(&tile[r][4 * (lane & 7)]);
            m4[it] = !a.partial && a.mask && on && row0 + r < a.M
                         ? *reinterpret_cast<const float4 *>(a.mask + (int64_t)(row0 + r) * a.ldc + n)
                         : make_float4(1.f, 1.f, 1.f, 1.f);
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) bv[e] = !a.partial && a.bias && on ? a.bias[n + e] : 0.f;
#pragma unroll
        for (int it = 0; it < 8; ++it) {
            const int row = row0 + 4 * it + (lane >> 3);
            if (row >= a.M || !on) continue;
            float x[4] = {x4[it].x, x4[it].y, x4[it].z, x4[it].w};
            if (!a.partial) {
                const float m[4] = {m4[it].x, m4[it].y, m4[it].z, m4[it].w};
#pragma unroll
                for (int e = 0; e < 4; ++e) x[e] = finish(a, m[e], bv[e], x[e]);
                if (a.H) store_packed4(a, row, n, x);
            }
            if (C) *reinterpret_cast<float4 *>(C + (int64_t)row * ldc + n) = make_float4(x[0], x[1], x[2], x[3]);
        }
    } else {
        const int n = n0 + lane;
        const bool on = n < a.N;
        const float bn = !a.partial && a.bias && on ? a.bias[n] : 0.f;
#pragma unroll
        for (int g = 0; g < 32; g += 16) {
            float xr[16], m[16];
#pragma unroll
            for (int r = 0; r < 16; ++r) {
                xr[r] = tile[g + r][lane];
                m[r] = !a.partial && a.mask && on && row0 + g + r < a.M
                           ? a.mask[(int64_t)(row0 + g + r) * a.ldc + n]
                           : 1.f;
            }
#pragma unroll
            for (int r = 0; r < 16; ++r) {
                const int row = row0 + g + r;
                if (row >= a.M || !on) continue;
                float x = xr[r];
                if (!a.partial) {
                    x = finish(a, m[r], bn, x);
                    if (a.H) {
                        const __nv_bfloat16 hi = __float2bfloat16_rn(x);
                        a.H[(int64_t)row * a.hkw + n] = hi;
                        a.H[(int64_t)row * a.hkw + a.hseg + n] = __float2bfloat16_rn(x - __bfloat162float(hi));
                    }
                }
                if (C) C[(int64_t)row * ldc + n] = x;
            }
        }
    }
    __syncwarp();
}

}  // namespace

// C (+ bias, ReLU, mask, packed copy) = A B^T over the K blocks
// [z kps, min(nkb, (z + 1) kps)) of this CTA's split, or, with partial set,
// the split's raw sum into C + z M N (row stride N).  BN = 128 or 256 columns
// per tile: the B tile is BN / 128 stacked 128-row boxes, one MMA of N = BN
// per 16-wide K step, BN TMEM columns.
template <int BN>
__global__ void __launch_bounds__(256, 1) k_tc_gemm(const __grid_constant__ CUtensorMap ma,
                                                    const __grid_constant__ CUtensorMap mb, TcArgs a) {
    constexpr int TC_STAGES = tc_stages<BN, 8>();
    constexpr int NB = BN / 128;                         // B boxes per stage
    constexpr int BTILE = NB * TC_TILE_BYTES;            // B bytes per stage
    constexpr uint32_t IDESC = tc_idesc<BN>();
    extern __shared__ uint8_t tc_smem_raw[];
    __shared__ __align__(8) uint64_t full[TC_STAGES], empty[TC_STAGES], done;
    __shared__ uint32_t tmem_slot;
    __shared__ int failed;
    __shared__ __align__(16) float stile[8][32][TC_TS];  // per warp: a 32 x 32 chunk of C
    const uint32_t raw = smem_u32(tc_smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;  // the 128-byte swizzle wants 1024-byte aligned tiles
    const uint32_t sA = base, sB = base + TC_STAGES * TC_TILE_BYTES;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int n0 = blockIdx.x * BN, m0 = blockIdx.y * TC_BM;
    const int kb0 = blockIdx.z * a.kps;
    const int nk = min(a.nkb, kb0 + a.kps) - kb0;
    if (threadIdx.x == 0) {
        for (int s = 0; s < TC_STAGES; ++s) {
            mbar_init(smem_u32(&full[s]), 1);
            mbar_init(smem_u32(&empty[s]), 1);
        }
        mbar_init(smem_u32(&done), 1);
        failed = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                     "r"(a.run > 0 ? 4 * BN : BN)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_slot;
    const int run = a.run > 0 ? a.run : nk, nrun = (nk + run - 1) / run;
    pdl_trigger();
    pdl_wait();  // barriers and tensor memory are set up; the operands may now be read

    // warp 0 is the issuing warp: lane 0 runs the copy / product loop and the
    // other lanes park at __syncwarp (a spinning lane of the same warp would
    // share its issue slots and stall the loop); warps 1-7 wait on "done"
    if (threadIdx.x == 0) {
        bool ok = true;
        int issued = 0, consumed = 0;
        auto load = [&](int k) {
            const int s = k % TC_STAGES;
            const uint32_t fb = smem_u32(&full[s]);
            mbar_expect_tx(fb, TC_TILE_BYTES + BTILE);
            tma_load_2d(sA + s * TC_TILE_BYTES, &ma, (kb0 + k) * TC_BK, m0, fb);
#pragma unroll
            for (int h = 0; h < NB; ++h)  // 128-row boxes stacked: 8-row groups stay 1024 B apart
                tma_load_2d(sB + s * BTILE + h * TC_TILE_BYTES, &mb, (kb0 + k) * TC_BK, n0 + 128 * h, fb);
        };
        for (int k = 0; k < nk && k < TC_STAGES; ++k) {
            load(k);
            ++issued;
        }
        for (int k = 0; k < nk; ++k) {
            const int s = k % TC_STAGES;
            if (!mbar_wait(smem_u32(&full[s]), (uint32_t)(k / TC_STAGES) & 1u)) { ok = false; break; }
            ++consumed;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
            for (int j = 0; j < TC_BK / 16; ++j)  // K = 16 per instruction: 32 bytes along the swizzled row
                mma_bf16(tmem + (uint32_t)(k / run * BN), sw128_desc(sA + s * TC_TILE_BYTES + 32 * j),
                         sw128_desc(sB + s * BTILE + 32 * j), IDESC, (k % run > 0 || j > 0) ? 1u : 0u);
            mma_commit(smem_u32(&empty[s]));
            // refill the stage of the previous K block once its products are done
            if (k >= 1 && k - 1 + TC_STAGES < nk) {
                const int sp = (k - 1) % TC_STAGES;
                if (!mbar_wait(smem_u32(&empty[sp]), (uint32_t)((k - 1) / TC_STAGES) & 1u)) { ok = false; break; }
                load(k - 1 + TC_STAGES);
                ++issued;
            }
        }
        mma_commit(smem_u32(&done));  // arrives once every product issued above has completed
        if (!ok) {
            atomicExch(a.err, 1);
            failed = 1;
            for (int k = consumed; k < issued; ++k)  // copies still in flight land before the CTA exits
                mbar_wait(smem_u32(&full[k % TC_STAGES]), (uint32_t)(k / TC_STAGES) & 1u);
        }
    }
    if (warp == 0) __syncwarp();
    const bool got = mbar_wait(smem_u32(&done), 0u);
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const int all_ok = __syncthreads_and(got ? 1 : 0);
    if (!all_ok && threadIdx.x == 0) atomicExch(a.err, 1);
    if (all_ok && !failed && nk > 0) {
        float *C = a.partial ? a.C + (int64_t)blockIdx.z * a.M * a.N : a.C;
        const int quad = warp & 3;  // its quarter of the tensor memory's lanes; two warps share a quarter's columns
        for (int c = 32 * (warp >> 2); c < BN && n0 + c < a.N; c += 64) {
            float v[32];
            tmem_ld32(tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)c, v);
            for (int r = 1; r < nrun; ++r) {
                float u[32];
                tmem_ld32(tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(r * BN + c), u);
#pragma unroll
                for (int i = 0; i < 32; ++i) v[i] += u[i];
            }
            store_chunk(a, stile[warp], v, C, a.partial ? a.N : a.ldc, m0 + quad * 32, n0 + c, lane);
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(a.run > 0 ? 4 * BN : BN) : "memory");
    }
}

// Persistent form for large products (no K split): one CTA per SM walks the
// 128 x BN tiles in a grid-stride loop, in groups of 16 M blocks with the M
// block fastest inside a group (the tiles in flight share their A and B panels
// in L2), with three roles.  Warp 0 lane 0 streams the operand boxes of every
// (tile, K block) through the ring of stages; warp 1 lane 0 issues the MMAs
// into one of two TMEM accumulators (2 BN columns) and commits each stage
// to its "empty" barrier and each finished tile to its accumulator's "full"
// barrier; the other warps read a finished accumulator back (warp w owns TMEM
// lanes 32 (w mod 4) ..), apply the epilogue and release the accumulator, so
// the epilogue of one tile overlaps the products of the next.  Every wait is
// bounded: on expiry *err is raised and the role stops, and all roles reach
// the final barrier.
// tile t -> (M block, N block) in groups of TC_GROUP M blocks
constexpr int TC_GROUP = 16;
__device__ __forceinline__ void tc_tile(int t, int tn, int tm, int &mb, int &nb) {
    const int per = TC_GROUP * tn, grp = t / per, first = grp * TC_GROUP;
    const int gsize = min(TC_GROUP, tm - first), r = t - grp * per;
    mb = first + r % gsize;
    nb = r / gsize;
}

template <int BN, int EW>
__global__ void __launch_bounds__(64 + 32 * EW, 1) k_tc_gemm_persistent(const __grid_constant__ CUtensorMap ma,
                                                               const __grid_constant__ CUtensorMap mb, TcArgs a,
                                                               int tn, int ntiles) {
    constexpr int TC_STAGES = tc_stages<BN, EW>();
    constexpr int NB = BN / 128;
    constexpr int BTILE = NB * TC_TILE_BYTES;
    constexpr uint32_t IDESC = tc_idesc<BN>();
    extern __shared__ uint8_t tc_smem_raw[];
    __shared__ __align__(8) uint64_t full[TC_STAGES], empty[TC_STAGES], tfull[2], tempty[2], done;
    __shared__ uint32_t tmem_slot;
    __shared__ __align__(16) float stile[EW][32][TC_TS];  // per epilogue warp: a 32 x 32 chunk
    const uint32_t raw = smem_u32(tc_smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    const uint32_t sA = base, sB = base + TC_STAGES * TC_TILE_BYTES;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < TC_STAGES; ++s) {
            mbar_init(smem_u32(&full[s]), 1);
            mbar_init(smem_u32(&empty[s]), 1);
        }
        for (int c = 0; c < 2; ++c) {
            mbar_init(smem_u32(&tfull[c]), 1);
            mbar_init(smem_u32(&tempty[c]), EW);  // one arrival per epilogue warp
        }
        mbar_init(smem_u32(&done), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                     "r"(2 * BN)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_slot;
    pdl_trigger();
    pdl_wait();
    const int nkb = a.nkb;
    if (warp == 0) {
        if (lane == 0) {  // producer
            int64_t it = 0;
            bool ok = true;
            for (int t = blockIdx.x; t < ntiles && ok; t += gridDim.x) {
                int mbk, nbk;
                tc_tile(t, tn, ntiles / tn, mbk, nbk);
                const int m0 = mbk * TC_BM, n0 = nbk * BN;
                for (int kb = 0; kb < nkb; ++kb, ++it) {
                    const int s = (int)(it % TC_STAGES);
                    if (it >= TC_STAGES &&
                        !mbar_wait(smem_u32(&empty[s]), (uint32_t)((it / TC_STAGES - 1) & 1))) { ok = false; break; }
                    const uint32_t fb = smem_u32(&full[s]);
                    mbar_expect_tx(fb, TC_TILE_BYTES + BTILE);
                    tma_load_2d(sA + s * TC_TILE_BYTES, &ma, kb * TC_BK, m0, fb);
#pragma unroll
                    for (int h = 0; h < NB; ++h)
                        tma_load_2d(sB + s * BTILE + h * TC_TILE_BYTES, &mb, kb * TC_BK, n0 + 128 * h, fb);
                }
            }
            if (!ok) atomicExch(a.err, 1);
            // the copies of the last stages land before the CTA exits
            for (int64_t k = std::max<int64_t>(0, it - TC_STAGES); k < it; ++k)
                mbar_wait(smem_u32(&full[k % TC_STAGES]), (uint32_t)((k / TC_STAGES) & 1));
        }
        __syncwarp();
    } else if (warp == 1) {
        if (lane == 0) {  // MMA issue
            int64_t it = 0;
            int tc = 0;
            bool ok = true;
            for (int t = blockIdx.x; t < ntiles && ok; t += gridDim.x, ++tc) {
                const int c = tc & 1;
                if (tc >= 2 && !mbar_wait(smem_u32(&tempty[c]), (uint32_t)(((tc >> 1) - 1) & 1))) { ok = false; break; }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t acc = tmem + (uint32_t)(c * BN);
                for (int kb = 0; kb < nkb; ++kb, ++it) {
                    const int s = (int)(it % TC_STAGES);
                    if (!mbar_wait(smem_u32(&full[s]), (uint32_t)((it / TC_STAGES) & 1))) { ok = false; break; }
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
                    for (int j = 0; j < TC_BK / 16; ++j)
                        mma_bf16(acc, sw128_desc(sA + s * TC_TILE_BYTES + 32 * j), sw128_desc(sB + s * BTILE + 32 * j),
                                 IDESC, (kb > 0 || j > 0) ? 1u : 0u);
                    mma_commit(smem_u32(&empty[s]));
                }
                mma_commit(smem_u32(&tfull[c]));
            }
            if (!ok) atomicExch(a.err, 1);
            // every product issued has completed before the accumulators are freed
            mma_commit(smem_u32(&done));
            if (!mbar_wait(smem_u32(&done), 0u)) atomicExch(a.err, 1);
        }
        __syncwarp();
    } else {  // epilogue warps 2 .. EW + 1
        const int quad = warp & 3;
        int tc = 0;
        for (int t = blockIdx.x; t < ntiles; t += gridDim.x, ++tc) {
            const int c = tc & 1;
            const bool got = mbar_wait(smem_u32(&tfull[c]), (uint32_t)((tc >> 1) & 1));
            if (!__all_sync(0xffffffffu, got)) {
                if (lane == 0) atomicExch(a.err, 1);
                break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            int mbk, nbk;
            tc_tile(t, tn, ntiles / tn, mbk, nbk);
            const int m0 = mbk * TC_BM, n0 = nbk * BN;
            for (int cc = 32 * ((warp - 2) >> 2); cc < BN && n0 + cc < a.N; cc += 8 * EW) {
                float v[32];
                tmem_ld32(tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(c * BN + cc), v);
                store_chunk(a, stile[warp - 2], v, a.C, a.ldc, m0 + quad * 32, n0 + cc, lane);
            }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&tempty[c])) : "memory");
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 1) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2 * BN) : "memory");
    }
}

// sum of the split partials in split order, then the epilogue; a.partial is
// 0 here and P holds the partials
__global__ void __launch_bounds__(256) k_tc_reduce(TcArgs a, int splits, const float *P) {
    pdl_trigger();
    pdl_wait();
    const int64_t MN = (int64_t)a.M * a.N;
    if (a.vec) {
        for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; 4 * q < MN; q += (int64_t)gridDim.x * blockDim.x) {
            const int row = (int)(4 * q / a.N), n = (int)(4 * q - (int64_t)row * a.N);
            float x[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 8
            for (int z = 0; z < splits; ++z) {
                const float4 t = *reinterpret_cast<const float4 *>(P + z * MN + 4 * q);
                x[0] += t.x; x[1] += t.y; x[2] += t.z; x[3] += t.w;
            }
#pragma unroll
            for (int e = 0; e < 4; ++e)
                x[e] = finish(a, a.mask ? a.mask[(int64_t)row * a.ldc + n + e] : 1.f, a.bias ? a.bias[n + e] : 0.f, x[e]);
            if (a.H) store_packed4(a, row, n, x);
            if (a.C) *reinterpret_cast<float4 *>(a.C + (int64_t)row * a.ldc + n) = make_float4(x[0], x[1], x[2], x[3]);
        }
        return;
    }
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < MN; e += (int64_t)gridDim.x * blockDim.x) {
        const int row = (int)(e / a.N), n = (int)(e - (int64_t)row * a.N);
        float x = 0.f;
#pragma unroll 8
        for (int z = 0; z < splits; ++z) x += P[z * MN + e];
        x = finish(a, a.mask ? a.mask[(int64_t)row * a.ldc + n] : 1.f, a.bias ? a.bias[n] : 0.f, x);
        if (a.H) {
            const __nv_bfloat16 hi = __float2bfloat16_rn(x);
            a.H[(int64_t)row * a.hkw + n] = hi;
            a.H[(int64_t)row * a.hkw + a.hseg + n] = __float2bfloat16_rn(x - __bfloat162float(hi));
        }
        if (a.C) a.C[(int64_t)row * a.ldc + n] = x;
    }
}

// dst[r kw + g kseg + k] = part_g(src[r ld + k]) for r < R, segment g < nseg,
// k < kseg (zero for k >= K); part code 0: hi = bf16(x), 1: lo = bf16(x - hi).
// A warp per row, two columns per lane: one thread per element with a 64-bit
// division each took 30 us for 29 k rows of 225 from cold caches, 17 us here.
__global__ void __launch_bounds__(256) k_tc_pack(int64_t R, int K, int kseg, int nseg, uint32_t codes,
                                                 const float *src, int64_t ld,
                                                 __nv_bfloat16 *__restrict__ dst, int64_t kw) {
    pdl_trigger();
    pdl_wait();
    const int lane = threadIdx.x & 31;
    for (int64_t r = blockIdx.x * (int64_t)8 + (threadIdx.x >> 5); r < R; r += (int64_t)gridDim.x * 8) {
        const float *s = src + r * ld;
        __nv_bfloat16 *d = dst + r * kw;
#pragma unroll 4
        for (int k = 2 * lane; k < kseg; k += 64) {
            const float x0 = k < K ? s[k] : 0.f, x1 = k + 1 < K ? s[k + 1] : 0.f;
            const __nv_bfloat16 h0 = __float2bfloat16_rn(x0), h1 = __float2bfloat16_rn(x1);
            const uint32_t hi = pack_bf16(h0, h1), lo = pack_bf16(__float2bfloat16_rn(x0 - __bfloat162float(h0)),
                                                                  __float2bfloat16_rn(x1 - __bfloat162float(h1)));
            for (int g = 0; g < nseg; ++g)
                *reinterpret_cast<uint32_t *>(d + (int64_t)g * kseg + k) = ((codes >> (2 * g)) & 3u) ? lo : hi;
        }
    }
}

// The transposed pack, element (r, k) = src[k ld + r]: tiles of 64 k x 32 r
// through shared memory, read along r and written as eight k (16 bytes) per
// thread and segment.  csum (or null): the tile's column sums, into
// csum[(k / 64) R + r], for the bias gradients, which read the same matrix.
__global__ void __launch_bounds__(256) k_tc_pack_t(int R, int K, int kseg, int nseg, uint32_t codes,
                                                   const float *src, int64_t ld,
                                                   __nv_bfloat16 *__restrict__ dst, int64_t kw,
                                                   float *__restrict__ csum) {
    __shared__ float tile[64][33];
    pdl_trigger();
    pdl_wait();
    const int k0 = blockIdx.x * 64, r0 = blockIdx.y * 32, tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int k = k0 + ty + 8 * i, r = r0 + tx;
        tile[ty + 8 * i][tx] = k < K && r < R ? src[(int64_t)k * ld + r] : 0.f;
    }
    __syncthreads();
    const int rr = threadIdx.x >> 3, j = threadIdx.x & 7, r = r0 + rr;
    float x[8], sum = 0.f;
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        x[e] = tile[8 * j + e][rr];
        sum += x[e];
    }
    if (csum) {
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
        if (j == 0 && r < R && k0 < K) csum[(int64_t)blockIdx.x * R + r] = sum;
    }
    if (r >= R) return;
    uint32_t hi[4], lo[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const __nv_bfloat16 h0 = __float2bfloat16_rn(x[2 * e]), h1 = __float2bfloat16_rn(x[2 * e + 1]);
        hi[e] = pack_bf16(h0, h1);
        lo[e] = pack_bf16(__float2bfloat16_rn(x[2 * e] - __bfloat162float(h0)),
                          __float2bfloat16_rn(x[2 * e + 1] - __bfloat162float(h1)));
    }
    __nv_bfloat16 *d = dst + (int64_t)r * kw + k0 + 8 * j;
    for (int g = 0; g < nseg; ++g)
        *reinterpret_cast<uint4 *>(d + (int64_t)g * kseg) =
            ((codes >> (2 * g)) & 3u) ? make_uint4(lo[0], lo[1], lo[2], lo[3]) : make_uint4(hi[0], hi[1], hi[2], hi[3]);
}

namespace {
PFN_cuTensorMapEncodeTiled_v12000 g_encode = nullptr;
std::once_flag g_encode_once;
std::once_flag g_attr_once;
cudaError_t g_attr_err = cudaSuccess;

template <int BN>
cs_status tc_launch(const TcOperand &A, const TcOperand &B, const TcArgs &a, int tn, int tm, int splits,
                    cudaStream_t s) {
    const int ntiles = tn * tm;
    if (splits == 1 && ntiles > 152) {  // more tiles than SMs: a CTA per SM overlaps its epilogues
        // An epilogue of 128 x 256 results by four warps, one a scheduler, waits for its own instructions (ncu: 0.5
        // of a warp instruction per cycle and SM): it took longer than a product of 8 K blocks.  Eight warps share
        // it there; long products hide it and want the fourth stage instead.
        if (a.nkb <= 32)
            CSX_CUDA(launch_k(k_tc_gemm_persistent<BN, 8>, 152, 320, tc_smem<BN, 8>(), s, A.map, B.map, a, tn, ntiles));
        else
            CSX_CUDA(launch_k(k_tc_gemm_persistent<BN, 4>, 152, 192, tc_smem<BN, 4>(), s, A.map, B.map, a, tn, ntiles));
    } else
        CSX_CUDA(launch_k(k_tc_gemm<BN>, dim3(tn, tm, splits), 256, tc_smem<BN, 8>(), s, A.map, B.map, a));
    count_launch();
    return CS_OK;
}
}  // namespace

cs_status tc_map(CUtensorMap *map, const __nv_bfloat16 *ptr, int64_t rows, int64_t kw) {
    std::call_once(g_encode_once, [] {
        cudaDriverEntryPointQueryResult q;
        void *fn = nullptr;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            g_encode = (PFN_cuTensorMapEncodeTiled_v12000)fn;
    });
    if (!g_encode) {
        set_error("cuTensorMapEncodeTiled is not available from the driver");
        return CS_ERR_CUDA;
    }
    if (((uintptr_t)ptr & 15) || kw % 8 || rows < 1 || kw < 1) {
        set_error("tensor-core operand: base not 16-byte aligned or K width not a multiple of 8");
        return CS_ERR_ARG;
    }
    const cuuint64_t dims[2] = {(cuuint64_t)kw, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)kw * 2};
    const cuuint32_t box[2] = {(cuuint32_t)TC_BK, (cuuint32_t)TC_BM};
    const cuuint32_t es[2] = {1, 1};
    std::memset(map, 0, sizeof(*map));
    const CUresult r = g_encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, (void *)ptr, dims, strides, box, es,
                                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                                CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) {
        set_error("cuTensorMapEncodeTiled failed (%d)", (int)r);
        return CS_ERR_CUDA;
    }
    return CS_OK;
}

cs_status tc_operand_init(TcOperand &op, int64_t rows, int64_t kw, int64_t *acct) {
    op.rows = rows;
    op.kw = kw;
    CSX_TRY(dalloc_t(&op.p, (size_t)(rows * kw), acct));
    CSX_CUDA(cudaMemset(op.p, 0, sizeof(__nv_bfloat16) * (size_t)(rows * kw)));
    return tc_map(&op.map, op.p, rows, kw);
}

static cs_status pack_codes(const TcOperand &op, int64_t R, int K, int kseg, const char *parts, int *nseg,
                            uint32_t *codes) {
    *nseg = (int)std::strlen(parts);
    if (R > op.rows || (int64_t)*nseg * kseg > op.kw || kseg % TC_BK || K > kseg) {
        set_error("tensor-core operand too small for the pack");
        return CS_ERR_ARG;
    }
    *codes = 0;
    for (int g = 0; g < *nseg; ++g) *codes |= (parts[g] == 'l' ? 1u : 0u) << (2 * g);
    return CS_OK;
}

cs_status tc_pack(TcOperand &op, int64_t R, int K, int kseg, const char *parts, const float *src, int64_t ld,
                  bool trans, cudaStream_t s) {
    if (trans) return tc_pack_sum(op, R, K, kseg, parts, src, ld, nullptr, s);
    int nseg;
    uint32_t codes;
    CSX_TRY(pack_codes(op, R, K, kseg, parts, &nseg, &codes));
    CSX_CUDA(launch_k(k_tc_pack, (unsigned)std::max<int64_t>(1, std::min<int64_t>((R + 7) / 8, 152 * 8)), 256, 0, s, R,
                      K, kseg, nseg, codes, src, ld, op.p, op.kw));
    count_launch();
    return CS_OK;
}

cs_status tc_pack_sum(TcOperand &op, int64_t R, int K, int kseg, const char *parts, const float *src, int64_t ld,
                      float *csum, cudaStream_t s) {
    int nseg;
    uint32_t codes;
    CSX_TRY(pack_codes(op, R, K, kseg, parts, &nseg, &codes));
    CSX_CUDA(launch_k(k_tc_pack_t, dim3((unsigned)(kseg / 64), (unsigned)((R + 31) / 32)), 256, 0, s, (int)R, K, kseg,
                      nseg, codes, src, ld, op.p, op.kw, csum));
    count_launch();
    return CS_OK;
}

cs_status tc_gemm(const TcOperand &A, const TcOperand &B, int M, int N, int64_t K, float *C, int ldc,
                  const TcEpilogue &ep, float *partial, int64_t partial_cap, int *err, cudaStream_t s) {
    if (M < 1 || N < 1 || K < 1 || M > A.rows || N > B.rows || K > A.kw || K > B.kw) {
        set_error("tensor-core GEMM: shape exceeds its operands");
        return CS_ERR_ARG;
    }
    if (ep.packed && (M > ep.packed->rows || 2 * (int64_t)ep.kseg > ep.packed->kw || N > ep.kseg)) {
        set_error("tensor-core GEMM: packed result exceeds its operand");
        return CS_ERR_ARG;
    }
    std::call_once(g_attr_once, [] {
        const auto allow = [](auto *kernel, int bytes) {
            if (g_attr_err == cudaSuccess)
                g_attr_err = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
        };
        allow(k_tc_gemm<128>, tc_smem<128, 8>());
        allow(k_tc_gemm<256>, tc_smem<256, 8>());
        allow(k_tc_gemm_persistent<128, 4>, tc_smem<128, 4>());
        allow(k_tc_gemm_persistent<128, 8>, tc_smem<128, 8>());
        allow(k_tc_gemm_persistent<256, 4>, tc_smem<256, 4>());
        allow(k_tc_gemm_persistent<256, 8>, tc_smem<256, 8>());
    });
    CSX_CUDA(g_attr_err);
    // 128 x 256 tiles (one MMA of N = 256 per K step) where they fill half the SMs,
    // else 128 x 128 ones.
    const int nkb = (int)((K + TC_BK - 1) / TC_BK), tm = (M + TC_BM - 1) / TC_BM;
    const int t256 = (N > 128 ? (N + 255) / 256 : 1) * tm;
    const int bn = N > 128 && t256 >= 76 ? 256 : 128, tn = (N + bn - 1) / bn;
    // K is summed in runs whose length depends on the 256-wide tiles, never on
    // how the product is cut: the rounding error stays that of short runs, and a
    // unit whose input rounds to about zero falls on the same side of the ReLU.
    int runs = t256 >= 76 ? 1 : std::min(nkb, (152 + t256 - 1) / t256);
    int run = (nkb + runs - 1) / runs;
    runs = (nkb + run - 1) / run;
    if (runs > 1 && (!partial || (int64_t)runs * M * N > partial_cap)) {
        runs = 1;
        run = nkb;
    }
    // A CTA keeps up to four runs, an accumulator each in tensor memory: a split
    // costs a write and a read of C, which for the network's layers (8 K blocks)
    // took longer than the products.  More runs than that are splits, of as
    // many runs as leave a CTA for every SM (of one for a layer, whose sums keep
    // their order).
    const int per = runs <= 4 ? runs : ep.bias ? 1 : std::min(4, (runs * tn * tm + 151) / 152);
    const int kps = run * per, splits = (nkb + kps - 1) / kps;
    TcArgs a{};
    a.M = M; a.N = N; a.nkb = nkb; a.kps = kps;
    a.run = per > 1 ? run : 0;
    a.C = C;
    a.ldc = ldc;
    a.bias = ep.bias; a.relu = ep.relu ? 1 : 0; a.mask = ep.mask;
    if (ep.packed) { a.H = ep.packed->p; a.hkw = ep.packed->kw; a.hseg = ep.kseg; }
    a.vec = N % 4 == 0 && ldc % 4 == 0 && (((uintptr_t)C | (uintptr_t)ep.mask) & 15) == 0;
    a.err = err;
    TcArgs g = a;
    if (splits > 1) {
        g.partial = 1;
        g.C = partial;
        g.vec = N % 4 == 0;
    }
    CSX_TRY(bn == 256 ? tc_launch<256>(A, B, g, tn, tm, splits, s) : tc_launch<128>(A, B, g, tn, tm, splits, s));
    if (splits > 1) {
        const int64_t items = a.vec ? (int64_t)M * N / 4 : (int64_t)M * N;
        CSX_CUDA(launch_k(k_tc_reduce, (unsigned)std::max<int64_t>(1, std::min<int64_t>((items + 255) / 256, 152 * 8)),
                          256, 0, s, a, splits, (const float *)partial));
        count_launch();
    }
    return CS_OK;
}

}  // namespace csx

extern "C" {

cs_status cs_tc_gemm_bf16(int M, int N, int K, const void *A, const void *B, float *C, cs_stream stream) {
    using namespace csx;
    if (M < 1 || N < 1 || K < 8 || K % 8 || !A || !B || !C) {
        set_error("cs_tc_gemm_bf16: M, N >= 1, K a positive multiple of 8, non-null operands");
        return CS_ERR_ARG;
    }
    cudaStream_t s = (cudaStream_t)stream;
    int dev = 0;
    CSX_CUDA(cudaGetDevice(&dev));
    const void *ptrs[3] = {A, B, C};
    const char *names[3] = {"A", "B", "C"};
    for (int k = 0; k < 3; ++k) {  // the operands must be memory of the current device
        cudaPointerAttributes at{};
        if (cudaPointerGetAttributes(&at, ptrs[k]) != cudaSuccess) {
            cudaGetLastError();
            set_error("cs_tc_gemm_bf16: %s is not a CUDA device pointer", names[k]);
            return CS_ERR_ARG;
        }
        if ((at.type != cudaMemoryTypeDevice && at.type != cudaMemoryTypeManaged) || at.device != dev) {
            set_error("cs_tc_gemm_bf16: %s must be device memory of the current device %d", names[k], dev);
            return CS_ERR_ARG;
        }
    }
    // one wait-expiry flag per device, allocated on first use there
    static int *errs[64] = {};
    static std::mutex mu;
    if (dev < 0 || dev >= 64) { set_error("device ordinal %d unsupported", dev); return CS_ERR_UNSUPPORTED; }
    int *err = nullptr;
    {
        std::lock_guard<std::mutex> g(mu);
        if (!errs[dev]) CSX_CUDA(cudaMalloc(&errs[dev], sizeof(int)));
        err = errs[dev];
    }
    TcOperand a, b;
    a.p = (__nv_bfloat16 *)A; a.rows = M; a.kw = K;
    b.p = (__nv_bfloat16 *)B; b.rows = N; b.kw = K;
    CSX_TRY(tc_map(&a.map, a.p, M, K));
    CSX_TRY(tc_map(&b.map, b.p, N, K));
    CSX_CUDA(cudaMemsetAsync(err, 0, sizeof(int), s));
    CSX_TRY(tc_gemm(a, b, M, N, K, C, N, TcEpilogue{}, nullptr, 0, err, s));
    int h = 0;
    CSX_CUDA(cudaMemcpyAsync(&h, err, sizeof(int), cudaMemcpyDeviceToHost, s));
    CSX_CUDA(cudaStreamSynchronize(s));
    if (h) {
        set_error("a tensor-core GEMM wait expired");
        return CS_ERR_TIMEOUT;
    }
    return CS_OK;
}

}  // extern "C"
