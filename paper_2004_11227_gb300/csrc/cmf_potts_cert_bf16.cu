// Potts certificates with the labels side by side: __nv_bfloat16 flows.
#include "cmf_potts_cert.cuh"

namespace cmf {

cudaError_t potts_cert_bf16(const PottsProblem& P, const PottsRowsMaps& M, bool aniso, bool dr,
                            float tau, double* partials, const EvalTail& T, int* err,
                            cudaStream_t st) {
    return potts_cert_s<__nv_bfloat16>(P, M, aniso, dr, tau, partials, T, err, st);
}

}  // namespace cmf
