// Tensor-core (tcgen05) BF16 GEMM C = A B^T used by the learned-setup
// network; see cs_tcgemm.cu.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>

#include "cs_internal.cuh"

namespace csx {

struct TcArgs {
    int M, N, nkb, kps;  // rows and columns of C, 64-wide K blocks in all, K blocks per split
    int run;             // > 0: K blocks per accumulator, at most four, added in order (BN = 128 only)
    float *C;            // C (row stride ldc) or null, or the split partials [split][M][N]
    int ldc;
    const float *bias;   // [N] or null
    int relu;
    const float *mask;   // values (row stride ldc) or null: C is 0 where mask is not > 0
    __nv_bfloat16 *H;    // the result as a packed operand, or null: hi at [m hkw + n], lo at [m hkw + hseg + n]
    int64_t hkw;
    int hseg;
    int partial;
    int vec;             // rows leave as float4: N, ldc multiples of 4 and C, mask 16-byte aligned
    int *err;            // set to 1 when a bounded wait expires
};

// A BF16 operand in HBM, K contiguous: rows x kw (kw a multiple of 8), with
// its TMA tensor map (128 x 64 boxes, 128-byte swizzle, zero fill outside).
struct TcOperand {
    __nv_bfloat16 *p = nullptr;
    int64_t rows = 0, kw = 0;
    CUtensorMap map;
};

cs_status tc_map(CUtensorMap *map, const __nv_bfloat16 *ptr, int64_t rows, int64_t kw);
// allocate (zeroed) and describe a rows x kw operand
cs_status tc_operand_init(TcOperand &op, int64_t rows, int64_t kw, int64_t *acct);
// pack R rows of an FP32 matrix as K-segments of kseg columns (K valid, the
// rest zero): parts[g] = 'h' (bf16(x)) or 'l' (bf16(x - bf16(x))) for
// segment g; trans: element (r, k) is src[k ld + r], else src[r ld + k]
cs_status tc_pack(TcOperand &op, int64_t R, int K, int kseg, const char *parts, const float *src, int64_t ld,
                  bool trans, cudaStream_t s);
// What a GEMM does with its sums: + bias, ReLU, zero where mask is not > 0;
// then C (FP32, unless null) and, with `packed`, the hi / lo segments of that
// operand ("hl" of tc_pack, segments of kseg columns; columns from N on stay
// as they are: zero).  As passes of their own, bias, activation, mask and the
// packing for the next GEMM moved each layer's output four times: prediction
// of 29 k blocks of 225 inputs went from 255 to 180 us (130 with the epilogue
// shared by eight warps), gradients of 4096 samples (with the packing below)
// from 530 to 239 (222).
struct TcEpilogue {
    const float *bias = nullptr;
    bool relu = false;
    const float *mask = nullptr;
    TcOperand *packed = nullptr;
    int kseg = 0;
};
// the same with the sums over the K rows of src, element (r, k) = src[k ld + r]
// (trans only): csum[(k / 64) R + r] = sum of the 64 rows' src[k ld + r]
cs_status tc_pack_sum(TcOperand &op, int64_t R, int K, int kseg, const char *parts, const float *src, int64_t ld,
                      float *csum, cudaStream_t s);
// C[M x N] = epilogue(A[M x K] B[N x K]^T) on the tensor cores, split along K
// when the tile grid is small (partials in partial[0 .. partial_cap), reduced
// in split order)
cs_status tc_gemm(const TcOperand &A, const TcOperand &B, int M, int N, int64_t K, float *C, int ldc,
                  const TcEpilogue &ep, float *partial, int64_t partial_cap, int *err, cudaStream_t s);

}  // namespace csx
