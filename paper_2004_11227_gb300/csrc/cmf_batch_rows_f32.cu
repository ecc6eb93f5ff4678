// Batch kernels of the Potts rows and binary chains: float flows.
#include "cmf_batch_rows.cuh"

namespace cmf {

cudaError_t batch_rows_f32(
    bool aniso, int lc, int nlab, int iters, const BatchDesc* desc, const BatchMaps* maps,
    const int2* items, int nitems, const AdmmCoef& K, int parity, int first,
    const int* merge, int* err, cudaStream_t st) {
    return batch_rows_s<float>(aniso, lc, nlab, iters, desc, maps, items, nitems, K, parity, first,
                             merge, err, st);
}

cudaError_t batch_chain_f32(
    bool aniso, int T, const BatchDesc* desc, const BatchMaps* maps, const int2* items, int nitems,
    const AdmmCoef& K, int parity, const int* merge, int* err,
    cudaStream_t st) {
    return batch_chain_s<float>(aniso, T, desc, maps, items, nitems, K, parity, merge, err, st);
}

}  // namespace cmf
