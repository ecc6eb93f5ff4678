// Host side of the binary ADMM kernel that chains warps (cmf_binary_chain.cuh):
// which layouts it takes, its tensor maps, and the dispatch to the storage
// type's translation unit.
#include "cmf_binary_chain.cuh"

namespace cmf {

cudaError_t binary_chain_step_f32(
    const BinProblem& P, const BinStateV& b, bool aniso,
    const AdmmCoef& K, int T, int iter0, const BinChainMaps& M, double* partials, int max_blocks,
    const EvalTail* cert, int* err, cudaStream_t st);
cudaError_t binary_chain_step_f16(
    const BinProblem& P, const BinStateV& b, bool aniso,
    const AdmmCoef& K, int T, int iter0, const BinChainMaps& M, double* partials, int max_blocks,
    const EvalTail* cert, int* err, cudaStream_t st);
cudaError_t binary_chain_step_bf16(
    const BinProblem& P, const BinStateV& b, bool aniso,
    const AdmmCoef& K, int T, int iter0, const BinChainMaps& M, double* partials, int max_blocks,
    const EvalTail* cert, int* err, cudaStream_t st);

int binary_chain_max_iters(bool cert) { return cert ? chain::kMaxCert : chain::kMaxIters; }

bool binary_chain_eligible(const BinProblem& P, int storage, const BinStateV& a,
                           const BinStateV& b, const BinStateV& c) {
    const Grid& G = P.g;
    if (G.plane > (size_t)INT_MAX) return false;
    const size_t es = dtype_size(storage);
    if ((G.pitch * es) % 16 || (G.pitch * 4) % 16) return false;
    auto al = [](const void* p) { return ((uintptr_t)p % 16) == 0; };
    if (!al(P.Cs) || !al(P.Ct) || (P.alpha.plane && !al(P.alpha.plane))) return false;
    for (const BinStateV* s : {&a, &b, &c})
        if (!al(s->u) || !al(s->qx) || !al(s->qy) || !al(s->ps) || !al(s->pt)) return false;
    return true;
}

bool binary_chain_certifies(const Grid& G, int max_blocks) {
    const int out = chain::kCols - chain::left_cols(chain::kMaxCert) -
                    chain::right_cols(chain::kMaxCert, true);
    return (G.W + out - 1) / out <= max_blocks;
}

cudaError_t binary_chain_maps(const BinProblem& P, int storage, const BinStateV& s,
                              BinChainMaps& m, const BinChainMaps* planes) {
    return binary_row_maps(
        P, storage, s, dtype_size(storage) == 4 ? chain::Seg<4>::cols : chain::Seg<2>::cols,
        chain::Seg<4>::cols, m, planes);
}

cudaError_t binary_row_maps(const BinProblem& P, int storage, const BinStateV& s, int cs, int c4,
                            BinChainMaps& m, const BinChainMaps* planes) {
    const Grid& G = P.g;
    const int es = (int)dtype_size(storage);
    const struct {
        CUtensorMap* map;
        const void* base;
        int es, box;
    } f[] = {{&m.qx, s.qx, es, cs}, {&m.qy, s.qy, es, cs}, {&m.ps, s.ps, es, cs},
              {&m.pt, s.pt, es, cs}, {&m.u, s.u, 4, c4},    {&m.Cs, P.Cs, 4, c4},
              {&m.Ct, P.Ct, 4, c4},  {&m.al, P.alpha.plane, 4, c4}};
    for (const auto& q : f) {
        if (planes && q.map == &m.Cs) {
            m.Cs = planes->Cs;
            m.Ct = planes->Ct;
            m.al = planes->al;
            break;
        }
        if (!q.base) {  // constant alpha: its map is never read
            *q.map = m.u;
            continue;
        }
        const cudaError_t e =
            encode_tma_3d(q.map, q.base, q.es, G.W, G.H, 1, G.pitch, q.box, 1);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t binary_chain_step(
    int storage, const BinProblem& P, const BinStateV& b, bool aniso,
    const AdmmCoef& K, int T, int iter0, const BinChainMaps& M, double* partials, int max_blocks,
    const EvalTail* cert, int* err, cudaStream_t st) {
    switch (storage) {
        case CMF_F32:
            return binary_chain_step_f32(P, b, aniso, K, T, iter0, M, partials, max_blocks, cert, err, st);
        case CMF_F16:
            return binary_chain_step_f16(P, b, aniso, K, T, iter0, M, partials, max_blocks, cert, err, st);
        default:
            return binary_chain_step_bf16(P, b, aniso, K, T, iter0, M, partials, max_blocks, cert, err,
                                          st);
    }
}

}  // namespace cmf
