// Host side of the copy engine: tensor maps of bf16 tensors.
#pragma once
#include <cuda.h>  // CUtensorMap and its enums; the encoder is reached through the runtime's entry-point query

#include "common.cuh"

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

inline EncodeTiledFn encode_fn() {
    // (an initialiser and no flag: a second thread's first call waits for the query of the first one)
    static const EncodeTiledFn fn = []() -> EncodeTiledFn {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) != cudaSuccess || q != cudaDriverEntryPointSuccess)
            return nullptr;
        return reinterpret_cast<EncodeTiledFn>(p);
    }();
    return fn;
}

inline CUtensorMapSwizzle swizzle_of_row(int row_bytes) {
    return row_bytes == 128 ? CU_TENSOR_MAP_SWIZZLE_128B : (row_bytes == 64 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B);
}

// Map of a bf16 tensor with the given extents (innermost first), byte strides of dimensions 1 .. rank-1, and box; the
// box's innermost row (128, 64 or 32 bytes) selects the swizzle.
inline int make_map_strided(CUtensorMap *m, const void *base, int rank, const long long *dims, const long long *stride_bytes,
                            const int *box) {
    EncodeTiledFn fn = encode_fn();
    if (!fn) return PPO_ERR_CUDA;
    cuuint64_t gd[5], gs[4];
    cuuint32_t bx[5], es[5];
    for (int i = 0; i < rank; ++i) {
        if (box[i] < 1 || box[i] > 256 || dims[i] < 1) return PPO_ERR_UNSUPPORTED;
        gd[i] = (cuuint64_t)dims[i];
        bx[i] = (cuuint32_t)box[i];
        es[i] = 1;
        if (i + 1 < rank) {
            if (stride_bytes[i] % 16 != 0 || stride_bytes[i] >= (1ll << 40)) return PPO_ERR_UNSUPPORTED;
            gs[i] = (cuuint64_t)stride_bytes[i];
        }
    }
    const int rb = box[0] * 2;
    if ((rb != 128 && rb != 64 && rb != 32) || !ppo_aligned(base, 16)) return PPO_ERR_UNSUPPORTED;
    const CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, (cuuint32_t)rank, const_cast<void *>(base), gd, gs, bx, es,
                          CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle_of_row(rb), CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? PPO_OK : PPO_ERR_CUDA;
}
