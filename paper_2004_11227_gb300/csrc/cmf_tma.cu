// Host-side TMA tensor-map encoding.  The driver function is looked up once
// through the runtime's entry-point query, so libcmf does not link libcuda.
#include <cudaTypedefs.h>

#ifdef CMF_FAULT_INJECTION
#include <atomic>
#endif

#include "cmf_tma.cuh"

namespace cmf {

static PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    if (!fn) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000,
                                             cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (PFN_cuTensorMapEncodeTiled_v12000)p;
    }
    return fn;
}

#ifdef CMF_FAULT_INJECTION
static std::atomic<long long> g_encodings{0};
#endif

bool tma_available() { return encode_fn() != nullptr; }

cudaError_t encode_tma_3d(CUtensorMap* map, const void* base, int elem_bytes, int cols, int rows,
                          int planes, int pitch, int box_x, int box_y, int box_z) {
    PFN_cuTensorMapEncodeTiled_v12000 fn = encode_fn();
    if (!fn) return cudaErrorInvalidValue;
    // plain bit copies: unsigned types of the element width (out-of-range
    // fill is all-zero bits, i.e. +0.0 for float32, float16 and bfloat16)
    const CUtensorMapDataType dt =
        elem_bytes == 4 ? CU_TENSOR_MAP_DATA_TYPE_UINT32 : CU_TENSOR_MAP_DATA_TYPE_UINT16;
    const cuuint64_t dims[3] = {(cuuint64_t)cols, (cuuint64_t)rows, (cuuint64_t)planes};
    const cuuint64_t strides[2] = {(cuuint64_t)pitch * elem_bytes,
                                   (cuuint64_t)pitch * elem_bytes * (cuuint64_t)rows};
    const cuuint32_t box[3] = {(cuuint32_t)box_x, (cuuint32_t)box_y,
                               (cuuint32_t)box_z};
    const cuuint32_t estr[3] = {1u, 1u, 1u};
#ifdef CMF_FAULT_INJECTION
    ++g_encodings;
#endif
    CUresult r = fn(map, dt, 3, const_cast<void*>(base), dims, strides, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                    CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

}  // namespace cmf

#ifdef CMF_FAULT_INJECTION
// Test build only: tensor maps encoded by the process so far.
extern "C" long long cmf_debug_map_encodings(void) { return cmf::g_encodings.load(); }
#endif
