// Potts ADMM with the labels side by side: __nv_bfloat16 flows, even widths.
#include "cmf_potts_rows.cuh"

namespace cmf {

cudaError_t potts_rows_step_bf16(const PottsProblem& P, const PottsStateV& b, bool aniso,
                                 const AdmmCoef& K, float cu_in, int iters,
                                 const PottsRowsMaps& M, int* err, cudaStream_t st) {
    return K.ty || K.cp ? potts_rows_step_s<__nv_bfloat16, false, false>(P, b, aniso, K, cu_in, iters, M, 0,
                                                               err, st)
                        : potts_rows_step_s<__nv_bfloat16, true, false>(P, b, aniso, K, cu_in, iters, M, 0,
                                                              err, st);
}

}  // namespace cmf
