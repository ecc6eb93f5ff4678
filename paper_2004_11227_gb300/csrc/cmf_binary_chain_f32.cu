// Binary ADMM by chains of warps: float flows.
#include "cmf_binary_chain.cuh"

namespace cmf {

cudaError_t binary_chain_step_f32(
    const BinProblem& P, const BinStateV& b, bool aniso,
    const AdmmCoef& K, int T, int iter0, const BinChainMaps& M, double* partials, int max_blocks,
    const EvalTail* cert, int* err, cudaStream_t st) {
    const bool simple = !K.ty && !K.cp;
#define CMF_CHAIN(SI, EV)                                                                   \
    binary_chain_step_s<float, SI, EV>(P, b, aniso, K, T, iter0, M, partials, max_blocks, cert, err, st)
    if (P.g.W % 2) return simple ? CMF_CHAIN(true, false) : CMF_CHAIN(false, false);
    return simple ? CMF_CHAIN(true, true) : CMF_CHAIN(false, true);
#undef CMF_CHAIN
}

}  // namespace cmf
