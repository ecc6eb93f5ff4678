// Batch kernels of the Potts rows and binary chains: __half flows.
#include "cmf_batch_rows.cuh"

namespace cmf {

cudaError_t batch_rows_f16(
    bool aniso, int lc, int nlab, int iters, const BatchDesc* desc, const BatchMaps* maps,
    const int2* items, int nitems, const AdmmCoef& K, int parity, int first,
    const int* merge, int* err, cudaStream_t st) {
    return batch_rows_s<__half>(aniso, lc, nlab, iters, desc, maps, items, nitems, K, parity, first,
                             merge, err, st);
}

cudaError_t batch_chain_f16(
    bool aniso, int T, const BatchDesc* desc, const BatchMaps* maps, const int2* items, int nitems,
    const AdmmCoef& K, int parity, const int* merge, int* err,
    cudaStream_t st) {
    return batch_chain_s<__half>(aniso, T, desc, maps, items, nitems, K, parity, merge, err, st);
}

}  // namespace cmf
