// Batches on the kernels of the single solves: Potts instances with the labels
// side by side, binary ones by chains of warps.  A block takes its item from a
// table of (instance, base band) pairs, takes *merge base bands where its own is
// the first of them, and its instance's problem, state and tensor
// maps from device memory, and leaves at once when the instance has converged.
// The tables hold one class of label counts each, so that small instances do
// not pay for the largest block.
//
// What bounds it.  The problem's and the state's pointers come from memory and not
// from the parameter bank: with two iterations a launch 118 registers for at most 4
// labels (three blocks of 5 warps an SM instead of four), and 104 to 148 bytes a
// thread spilled for 8 and 16 labels, where the single solves' kernel spills 4.  16
// instances of 512^2, L = 4, float32: 286 us per launch (ncu, cold L2), 36% of the
// issue slots, DRAM at 28%; the latency of loads and of a row's chain of shuffles is
// the rest.
#pragma once

#include "cmf_binary_chain.cuh"
#include "cmf_potts_rows.cuh"

namespace cmf {

// Tensor maps in global memory: order the host's copy of them before their
// use by this thread.
__device__ __forceinline__ void acquire_maps(const CUtensorMap* m, int n) {
    for (int i = 0; i < n; ++i)
        asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;" ::"l"(
                         reinterpret_cast<uint64_t>(m + i))
                     : "memory");
}

template <typename S, bool ANISO, int T, int LC>
__global__ void __launch_bounds__(32 * (LC + rows::service_warps(T, LC)),
                                  LC == 4 ? 3 : (LC == 8 ? 2 : 1))
    k_batch_potts_rows(const BatchDesc* __restrict__ desc, const BatchMaps* __restrict__ maps,
                       const int2* __restrict__ items, AdmmCoef K, int parity, int first,
                       const int* merge, int* err) {
    const int2 e = items[blockIdx.x];
    const BatchDesc* D = desc + e.x;
    const int band = e.y / D->sp_nstrips, take = *merge;
    if (!D->active || band % take != 0) return;
    const PottsRowsMaps* M = &maps[D->tile_base].set[parity].potts;
    acquire_maps(&M->qx, sizeof(PottsRowsMaps) / sizeof(CUtensorMap));
    K.inv_a2 = D->ak.inv_a2;
    const PottsProblem P = D->pp;
    const PottsState<S> s1 = (parity ? D->pu : D->pw).as<S>();
    const int r0 = band * D->sp_rows;
    potts_rows_block<S, ANISO, true, T, LC, false>(
        *M, P, s1, K, first ? 0.f : K.cu, r0, min(r0 + take * D->sp_rows, P.g.H),
        (e.y % D->sp_nstrips) * D->sp_out - (T == 2 ? 4 : 2), 0, err);
}

template <typename S, bool ANISO>
__global__ void __launch_bounds__(32 * (chain::kMaxIters + 1), 4)
    k_batch_binary_chain(const BatchDesc* __restrict__ desc, const BatchMaps* __restrict__ maps,
                         const int2* __restrict__ items, AdmmCoef K, int T, int parity,
                         const int* merge, int* err) {
    const int2 e = items[blockIdx.x];
    const BatchDesc* D = desc + e.x;
    const int band = e.y / D->sp_nstrips, take = *merge;
    if (!D->active || band % take != 0) return;
    const BinChainMaps* M = &maps[D->tile_base].set[parity].binary;
    acquire_maps(&M->qx, sizeof(BinChainMaps) / sizeof(CUtensorMap));
    const BinProblem P = D->bp;
    const BinState<S> s1 = (parity ? D->bu : D->bw).as<S>();
    const int r0 = band * D->sp_rows;
    constexpr int hl = chain::left_cols(chain::kMaxIters),
                  hr = chain::right_cols(chain::kMaxIters, false);
    DF a = {0.f, 0.f}, b = a, c = a;
    binary_chain_block<S, ANISO, true, false, false>(
        *M, P, s1, K, T, 0, r0, min(r0 + take * D->sp_rows, P.g.H),
        (e.y % D->sp_nstrips) * D->sp_out - hl, hl, hr, a, b, c, err);
}

template <typename S, bool ANISO, int T, int LC>
static cudaError_t launch_batch_rows(int nlab, const BatchDesc* desc, const BatchMaps* maps,
                                     const int2* items, int nitems, const AdmmCoef& K, int parity,
                                     int first, const int* merge, int* err, cudaStream_t st) {
    auto kern = k_batch_potts_rows<S, ANISO, T, LC>;
    constexpr size_t dyn = rows::Layout<LC, (int)sizeof(S), false>::bytes;
    static std::atomic<long long> limit[kMaxDevices];
    const cudaError_t e = raise_dyn_smem(limit, kern, dyn);
    if (e != cudaSuccess) return e;
    kern<<<nitems, 32 * (nlab + rows::service_warps(T, LC)), dyn, st>>>(desc, maps, items, K,
                                                                       parity, first, merge,
                                                                       err);
    return cudaGetLastError();
}

template <typename S>
static cudaError_t batch_rows_s(bool aniso, int lc, int nlab, int iters, const BatchDesc* desc,
                                const BatchMaps* maps, const int2* items, int nitems,
                                const AdmmCoef& K, int parity, int first, const int* merge, int* err,
                                cudaStream_t st) {
#define CMF_ROWS(AN, IT, LC) \
    launch_batch_rows<S, AN, IT, LC>(nlab, desc, maps, items, nitems, K, parity, first, merge,      \
                                     err, st)
#define CMF_ROWS_LC(AN, IT) \
    (lc == 4 ? CMF_ROWS(AN, IT, 4) : (lc == 8 ? CMF_ROWS(AN, IT, 8) : CMF_ROWS(AN, IT, 16)))
    if (iters == 2) return aniso ? CMF_ROWS_LC(true, 2) : CMF_ROWS_LC(false, 2);
    return aniso ? CMF_ROWS_LC(true, 1) : CMF_ROWS_LC(false, 1);
#undef CMF_ROWS_LC
#undef CMF_ROWS
}

template <typename S, bool ANISO>
static cudaError_t launch_batch_chain(int T, const BatchDesc* desc, const BatchMaps* maps,
                                      const int2* items, int nitems, const AdmmCoef& K,
                                      int parity, const int* merge, int* err, cudaStream_t st) {
    auto kern = k_batch_binary_chain<S, ANISO>;
    const size_t dyn = chain::Layout<(int)sizeof(S)>::bytes(T - 1);
    static std::atomic<long long> limit[kMaxDevices];
    const cudaError_t e = raise_dyn_smem(limit, kern, dyn);
    if (e != cudaSuccess) return e;
    kern<<<nitems, 32 * (T + 1), dyn, st>>>(desc, maps, items, K, T, parity, merge, err);
    return cudaGetLastError();
}

template <typename S>
static cudaError_t batch_chain_s(bool aniso, int T, const BatchDesc* desc, const BatchMaps* maps,
                                 const int2* items, int nitems, const AdmmCoef& K, int parity,
                                 const int* merge, int* err, cudaStream_t st) {
    return aniso ? launch_batch_chain<S, true>(T, desc, maps, items, nitems, K, parity, merge, err,
                                               st)
                 : launch_batch_chain<S, false>(T, desc, maps, items, nitems, K, parity, merge,
                                                err, st);
}

}  // namespace cmf
