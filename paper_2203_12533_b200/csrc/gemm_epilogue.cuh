// What the two GEMM kernels share: the epilogue's operands, its element-wise steps on 8-column
// groups, and the tensor-map encoder.
#pragma once

#include "pw_kernels.h"

namespace pw {

struct GemmEpilogue {
    int M, N;
    void* C; int ldc;
    const __nv_bfloat16* bias;
    const __nv_bfloat16* aux_in; int ld_aux;
    void* aux_out;                           // kEpiBiasGelu: GeLU of the pre-activation, pitch ldc
    int accumulate, act;
    float* row_dot; int head_dim, seq_len;   // kEpiRowDot: per (row, head) dot products with aux_in, [B, H, S]
};

// f = GeLU(f) and f *= GeLU'(u); one uniform branch on the activation per group, not per pair.
__device__ __forceinline__ void gelu8(float* f, int act)
{
    if (act == 0) {
#pragma unroll
        for (int j = 0; j < 8; j += 2) gelu2_erf(f[j], f[j + 1]);
    } else {
#pragma unroll
        for (int j = 0; j < 8; j += 2) gelu2(f[j], f[j + 1], act);
    }
}
__device__ __forceinline__ void gelu_grad_mul8(float* f, const float* u, int act)
{
    if (act == 0) {
#pragma unroll
        for (int j = 0; j < 8; j += 2) gelu_grad_mul2_erf(f[j], f[j + 1], u[j], u[j + 1]);
    } else {
#pragma unroll
        for (int j = 0; j < 8; j += 2) gelu_grad_mul2(f[j], f[j + 1], u[j], u[j + 1], act);
    }
}

// 2-D tensor map (bf16, or fp32 when f32 is set): `inner` contiguous elements per row, `outer`
// rows, row pitch ld elements; 128-byte swizzle, so box_inner * element size must be 128 bytes
// (64 bytes with swizzle64).
inline const char* encode_2d(Runtime* rt, CUtensorMap* map, const void* ptr, uint64_t inner, uint64_t outer, uint64_t ld,
                             uint32_t box_inner, uint32_t box_outer, bool f32 = false, bool swizzle64 = false)
{
    typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                      const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                      CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
    cuuint64_t dims[2] = {inner, outer};
    cuuint64_t strides[1] = {ld * (f32 ? 4 : 2)};
    cuuint32_t box[2] = {box_inner, box_outer};
    cuuint32_t estr[2] = {1, 1};
    CUresult r = reinterpret_cast<EncodeTiledFn>(rt->encode_tiled)(
        map, f32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(ptr), dims, strides, box, estr,
        CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle64 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? nullptr : "cuTensorMapEncodeTiled failed";
}

}  // namespace pw
