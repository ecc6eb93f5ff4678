// Tensor-memory-accelerator (TMA) staging helpers for sm_103a: mbarrier and
// cp.async.bulk.tensor wrappers in inline PTX, bounded waits, and host-side
// tensor-map encoding through the driver entry point (no libcuda link).
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#ifdef CMF_FAULT_INJECTION
#include <vector>
#endif

namespace cmf {

#ifdef CMF_FAULT_INJECTION
// Fault-injection test build only (never in the library the product loads):
// extra bytes every row barrier of this translation unit expects beyond what its
// copies deliver.  With a non-zero value no such phase can complete, the bounded
// waits run out, and the kernels record kErrWaitTimeout and return; nothing
// faults and no copy is left in flight.
static __device__ unsigned int g_inject_row_tx = 0;
static cudaError_t inject_row_tx(unsigned int bytes) {
    return cudaMemcpyToSymbol(g_inject_row_tx, &bytes, sizeof(bytes));
}
inline std::vector<cudaError_t (*)(unsigned int)>& inject_hooks() {  // one per unit
    static std::vector<cudaError_t (*)(unsigned int)> hooks;
    return hooks;
}
static const bool g_inject_hooked = (inject_hooks().push_back(inject_row_tx), true);
#define CMF_ROW_EXTRA_TX g_inject_row_tx
#else
#define CMF_ROW_EXTRA_TX 0u
#endif

// ---- device side -----------------------------------------------------------

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count)
                 : "memory");
}

// Make mbarrier initialisation visible to the async proxy (the TMA unit).
__device__ __forceinline__ void fence_mbar_init() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

// Order this thread's earlier shared-memory accesses (generic proxy) before
// later async-proxy (TMA) accesses to the same buffers.
__device__ __forceinline__ void fence_proxy_async_smem() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
                 "r"(bytes + CMF_ROW_EXTRA_TX)
                 : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// Wait for phase `parity` of the barrier to complete, giving up after about
// `limit_cycles` SM clock cycles.  Returns false on timeout.
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* bar, uint32_t parity,
                                                  long long limit_cycles) {
    if (mbar_try_wait(bar, parity)) return true;
    const long long t0 = clock64();
    while (!mbar_try_wait(bar, parity)) {
        if (clock64() - t0 > limit_cycles) return false;
    }
    return true;
}

// 2D / 3D tiled loads global -> shared, completing on `bar` (transaction
// bytes).  Coordinates are element indices, innermost first; the innermost
// coordinate times the element size must be a multiple of 16 bytes.
__device__ __forceinline__ void tma_load_2d(void* dst, const CUtensorMap* map, uint64_t* bar,
                                            int x, int y) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3}], [%4];" ::"r"(smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(smem_u32(bar))
        : "memory");
}

__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* map, uint64_t* bar,
                                            int x, int y, int z) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(smem_u32(bar))
        : "memory");
}

#ifdef CMF_FAULT_INJECTION
// Fault-injection test build only: about 50 microseconds, so a test can make
// a wait run out quickly (see cmf_debug_inject_tx_mismatch).
constexpr long long kWaitLimitCycles = 100000ll;
#else
// About one second at the GB300's 2.07 GHz maximum SM clock.
constexpr long long kWaitLimitCycles = 2000000000ll;
#endif

// (kErrWaitTimeout, the value a timed-out wait records, is in cmf_kernels.cuh.)

// ---- host side -------------------------------------------------------------

// Whether tensor maps can be encoded (the driver has the function).
bool tma_available();

// Encode a row-major [planes][rows][cols] tensor of `elem_bytes` elements with
// a row stride of `pitch` elements and a plane stride of rows * pitch; box
// {box_x, box_y, box_z}; out-of-range elements read as zero.  Returns
// cudaErrorInvalidValue when the driver rejects the description.
cudaError_t encode_tma_3d(CUtensorMap* map, const void* base, int elem_bytes, int cols, int rows,
                          int planes, int pitch, int box_x, int box_y, int box_z = 1);

}  // namespace cmf
