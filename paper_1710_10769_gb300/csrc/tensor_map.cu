// Host-side TMA descriptor encoding through the driver entry point (no link
// dependency on libcuda).
#include <cuda.h>
#include <cudaTypedefs.h>

#include <mutex>

#include "internal.cuh"
#include "ptx.cuh"

namespace hpc {

namespace {
PFN_cuTensorMapEncodeTiled_v12000 tiled_fn() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(f);
    });
    return fn;
}
}  // namespace

namespace {
bool encode(CUtensorMap* map, const void* base, int elem_bytes, uint64_t inner, uint64_t outer,
            uint64_t row_stride_bytes, uint32_t box_inner, uint32_t box_outer, CUtensorMapSwizzle swz) {
    auto fn = tiled_fn();
    if (!fn) return false;
    const CUtensorMapDataType dt = elem_bytes == 8 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT64
                                   : elem_bytes == 4 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32
                                                     : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16;
    cuuint64_t dims[2] = {(cuuint64_t)inner, (cuuint64_t)outer};
    cuuint64_t strides[1] = {(cuuint64_t)row_stride_bytes};
    cuuint32_t box[2] = {box_inner, box_outer};
    cuuint32_t estr[2] = {1, 1};
    return fn(map, dt, 2, const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, swz,
              CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}
}  // namespace

bool encode_tensor_map_2d(CUtensorMap* map, const void* base, int elem_bytes, uint64_t inner, uint64_t outer,
                          uint64_t row_stride_bytes, uint32_t box_inner, uint32_t box_outer) {
    return encode(map, base, elem_bytes, inner, outer, row_stride_bytes, box_inner, box_outer,
                  CU_TENSOR_MAP_SWIZZLE_NONE);
}

bool encode_tensor_map_2d_sw128(CUtensorMap* map, const void* base, int elem_bytes, uint64_t inner, uint64_t outer,
                                uint64_t row_stride_bytes, uint32_t box_inner, uint32_t box_outer) {
    return encode(map, base, elem_bytes, inner, outer, row_stride_bytes, box_inner, box_outer,
                  CU_TENSOR_MAP_SWIZZLE_128B);
}

bool device_readable(const void* q, size_t bytes, size_t align) {
    using Range = CUresult (*)(CUdeviceptr*, size_t*, CUdeviceptr);
    static const Range range = [] {
        void* fn = nullptr;
        cudaDriverEntryPointQueryResult st = cudaDriverEntryPointSymbolNotFound;
        const cudaError_t e = cudaGetDriverEntryPointByVersion("cuMemGetAddressRange", &fn, 12000, cudaEnableDefault, &st);
        if (e != cudaSuccess) (void)cudaGetLastError();
        return e == cudaSuccess && st == cudaDriverEntryPointSuccess ? reinterpret_cast<Range>(fn) : nullptr;
    }();
    int dev = 0;
    cudaPointerAttributes a{};
    if (reinterpret_cast<uintptr_t>(q) % align != 0 || !range) return false;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaPointerGetAttributes(&a, q) != cudaSuccess) {
        (void)cudaGetLastError();
        return false;
    }
    if (!(a.type == cudaMemoryTypeManaged || (a.type == cudaMemoryTypeDevice && a.device == dev))) return false;
    CUdeviceptr base = 0;
    size_t size = 0;
    const CUdeviceptr at = reinterpret_cast<CUdeviceptr>(q);
    return range(&base, &size, at) == CUDA_SUCCESS && at >= base && at - base <= size && bytes <= size - (at - base);
}

cudaError_t set_smem_once(const void* func, int bytes, int slot) {
    static std::mutex mu;
    static bool done[64][kSmemSlots] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64 || slot < 0 || slot >= kSmemSlots)
        return cudaFuncSetAttribute(func, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    std::lock_guard<std::mutex> lock(mu);
    if (done[dev][slot]) return cudaSuccess;
    e = cudaFuncSetAttribute(func, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess) done[dev][slot] = true;
    return e;
}

}  // namespace hpc
