// Potts rPDRQ with the labels side by side: __half flows.
#include "cmf_potts_dr_rows.cuh"

namespace cmf {

cudaError_t potts_dr_rows_f16(const PottsProblem& P, const PottsStateV& b, bool aniso,
                              const DrCoef& D, const PottsRowsMaps& M, int* err, cudaStream_t st) {
    return potts_dr_rows_s<__half>(P, b, aniso, D, M, err, st);
}

}  // namespace cmf
