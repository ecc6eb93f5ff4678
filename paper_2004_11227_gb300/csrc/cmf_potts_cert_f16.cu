// Potts certificates with the labels side by side: __half flows.
#include "cmf_potts_cert.cuh"

namespace cmf {

cudaError_t potts_cert_f16(const PottsProblem& P, const PottsRowsMaps& M, bool aniso, bool dr,
                           float tau, double* partials, const EvalTail& T, int* err,
                           cudaStream_t st) {
    return potts_cert_s<__half>(P, M, aniso, dr, tau, partials, T, err, st);
}

}  // namespace cmf
