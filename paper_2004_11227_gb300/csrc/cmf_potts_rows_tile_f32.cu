// Potts ADMM with the labels side by side: float flows, odd widths (the
// roundings of the TMA tile kernel).
#include "cmf_potts_rows.cuh"

namespace cmf {

cudaError_t potts_rows_tile_step_f32(const PottsProblem& P, const PottsStateV& b, bool aniso,
                                     const AdmmCoef& K, float cu_in, int iters,
                                     const PottsRowsMaps& M, int fused, int* err,
                                     cudaStream_t st) {
    return potts_rows_step_s<float, true, true>(P, b, aniso, K, cu_in, iters, M, fused, err, st);
}

}  // namespace cmf
