// Dispatch of the batch kernels to the storage type's translation unit.
#include "cmf_batch_rows.cuh"

namespace cmf {

cudaError_t batch_rows_f32(
    bool aniso, int lc, int nlab, int iters, const BatchDesc* desc, const BatchMaps* maps,
    const int2* items, int nitems, const AdmmCoef& K, int parity, int first,
    const int* merge, int* err, cudaStream_t st);
cudaError_t batch_chain_f32(
    bool aniso, int T, const BatchDesc* desc, const BatchMaps* maps, const int2* items, int nitems,
    const AdmmCoef& K, int parity, const int* merge, int* err, cudaStream_t st);
cudaError_t batch_rows_f16(
    bool aniso, int lc, int nlab, int iters, const BatchDesc* desc, const BatchMaps* maps,
    const int2* items, int nitems, const AdmmCoef& K, int parity, int first,
    const int* merge, int* err, cudaStream_t st);
cudaError_t batch_chain_f16(
    bool aniso, int T, const BatchDesc* desc, const BatchMaps* maps, const int2* items, int nitems,
    const AdmmCoef& K, int parity, const int* merge, int* err, cudaStream_t st);
cudaError_t batch_rows_bf16(
    bool aniso, int lc, int nlab, int iters, const BatchDesc* desc, const BatchMaps* maps,
    const int2* items, int nitems, const AdmmCoef& K, int parity, int first,
    const int* merge, int* err, cudaStream_t st);
cudaError_t batch_chain_bf16(
    bool aniso, int T, const BatchDesc* desc, const BatchMaps* maps, const int2* items, int nitems,
    const AdmmCoef& K, int parity, const int* merge, int* err, cudaStream_t st);

int batch_chain_cols() {
    return chain::kCols - chain::left_cols(chain::kMaxIters) -
           chain::right_cols(chain::kMaxIters, false);
}

cudaError_t batch_potts_rows_step(int storage, bool aniso, int lc, int nlab, int iters,
                                  const BatchDesc* desc, const BatchMaps* maps, const int2* items,
                                  int nitems, const AdmmCoef& K, int parity, int first,
                                  const int* merge, int* err, cudaStream_t st) {
    if (nitems <= 0) return cudaSuccess;
    auto f = storage == CMF_F32 ? batch_rows_f32
                                : (storage == CMF_F16 ? batch_rows_f16 : batch_rows_bf16);
    return f(aniso, lc, nlab, iters, desc, maps, items, nitems, K, parity, first, merge, err, st);
}

cudaError_t batch_binary_chain_step(int storage, bool aniso, int T, const BatchDesc* desc,
                                    const BatchMaps* maps, const int2* items, int nitems,
                                    const AdmmCoef& K, int parity, const int* merge,
                                    int* err, cudaStream_t st) {
    if (nitems <= 0) return cudaSuccess;
    auto f = storage == CMF_F32 ? batch_chain_f32
                                : (storage == CMF_F16 ? batch_chain_f16 : batch_chain_bf16);
    return f(aniso, T, desc, maps, items, nitems, K, parity, merge, err, st);
}

}  // namespace cmf
