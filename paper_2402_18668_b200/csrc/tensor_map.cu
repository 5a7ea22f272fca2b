// Tensor maps of the library's TMA tiles: rows of a bf16 [BH][L][width] array.
#include <cuda.h>

#include "common.cuh"
#include "sm100.cuh"

namespace based {

namespace {
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiledFn encode_fn() {
    static std::atomic<EncodeTiledFn> cached{nullptr};
    EncodeTiledFn fn = cached.load(std::memory_order_acquire);
    if (!fn) {
        void* ptr = nullptr;
        cudaDriverEntryPointQueryResult qres;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &ptr, cudaEnableDefault, &qres) == cudaSuccess &&
            qres == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(ptr);
        cached.store(fn, std::memory_order_release);
    }
    return fn;
}
}  // namespace

static bool encode_map(CUtensorMap* m, const void* base, int rank, const cuuint64_t* dims, const cuuint64_t* strides, const cuuint32_t* box,
                       CUtensorMapSwizzle sw) {
    EncodeTiledFn enc = encode_fn();
    if (!enc) return false;
    cuuint32_t estr[4] = {1, 1, 1, 1};
    auto encode = [&] {
        return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, rank, const_cast<void*>(base), dims, strides, box, estr,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, sw, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
    };
    if (encode()) return true;
    // The encoder is a driver call and fails in a thread that no runtime call has bound to the device's context yet,
    // such as autograd's worker thread when its allocations come out of the allocator's cache.  Bind it and try again.
    int dev = -1;
    return cudaGetDevice(&dev) == cudaSuccess && cudaSetDevice(dev) == cudaSuccess && encode();
}

bool make_rows_map_bf16(CUtensorMap* m, const void* base, int BH, int L, int width, int box_w, int box_rows,
                        CUtensorMapSwizzle sw) {
    const cuuint64_t dims[3] = {(cuuint64_t)width, (cuuint64_t)L, (cuuint64_t)BH};
    const cuuint64_t strides[2] = {(cuuint64_t)width * 2, (cuuint64_t)L * width * 2};
    const cuuint32_t box[3] = {(cuuint32_t)box_w, (cuuint32_t)box_rows, 1};
    return encode_map(m, base, 3, dims, strides, box, sw);
}

bool make_head_rows_map_bf16(CUtensorMap* m, const void* base, int BH, int H, int L, int width, int box_w, int box_rows,
                             CUtensorMapSwizzle sw) {
    if (H == 0) return make_rows_map_bf16(m, base, BH, L, width, box_w, box_rows, sw);
    const cuuint64_t row = (cuuint64_t)width * 2, heads = H;
    const cuuint64_t dims[4] = {(cuuint64_t)width, heads, (cuuint64_t)L, (cuuint64_t)(BH / H)};
    const cuuint64_t strides[3] = {row, heads * row, heads * L * row};
    const cuuint32_t box[4] = {(cuuint32_t)box_w, 1, (cuuint32_t)box_rows, 1};
    return encode_map(m, base, 4, dims, strides, box, sw);
}

}  // namespace based
