// Tensor maps: rows of 16-bit elements in device memory, fetched in boxes of whole or part rows.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>

namespace ckv {

// `rows` rows of `width` 16-bit elements at `base`, boxes of box_rows x box_width.  false if the driver cannot encode it.
inline bool encode_rows(CUtensorMap* map, const void* base, int width, int64_t rows, int box_width, int box_rows,
                        CUtensorMapSwizzle swizzle, CUtensorMapL2promotion l2)
{
    typedef CUresult (*EncodeFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                 const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                 CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
    static const EncodeFn encode = [] {
        void* fn = nullptr;
        cudaDriverEntryPointQueryResult q;
        const bool ok = cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &q) == cudaSuccess &&
                        q == cudaDriverEntryPointSuccess;
        if (!ok) cudaGetLastError();
        return ok ? reinterpret_cast<EncodeFn>(fn) : nullptr;
    }();
    if (!encode) return false;
    const cuuint64_t dims[2] = {(cuuint64_t)width, (cuuint64_t)rows}, strides[1] = {(cuuint64_t)width * 2};
    const cuuint32_t box[2] = {(cuuint32_t)box_width, (cuuint32_t)box_rows}, estr[2] = {1, 1};
    auto go = [&] {
        return encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
                      CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle, l2, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    };
    CUresult r = go();
    if (r == CUDA_ERROR_INVALID_CONTEXT) {
        // A driver call, which does not make a context current by itself as a launch does: a thread that has launched,
        // allocated and copied nothing yet has none.
        int device;
        if (cudaGetDevice(&device) != cudaSuccess || cudaSetDevice(device) != cudaSuccess) {
            cudaGetLastError();
            return false;
        }
        r = go();
    }
    return r == CUDA_SUCCESS;
}

}  // namespace ckv
