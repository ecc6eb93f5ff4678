// Potts certificates with the labels side by side: float flows.
#include "cmf_potts_cert.cuh"

namespace cmf {

cudaError_t potts_cert_f32(const PottsProblem& P, const PottsRowsMaps& M, bool aniso, bool dr,
                           float tau, double* partials, const EvalTail& T, int* err,
                           cudaStream_t st) {
    return potts_cert_s<float>(P, M, aniso, dr, tau, partials, T, err, st);
}

}  // namespace cmf
