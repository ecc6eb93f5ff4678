// Host side of the Potts ADMM kernel that runs the labels side by side
// (cmf_potts_rows.cuh): which layouts it takes, its tensor maps, and the
// dispatch to the storage type's translation unit.
#include <climits>

#include "cmf_potts_rows.cuh"

namespace cmf {

cudaError_t potts_rows_step_f32(const PottsProblem& P, const PottsStateV& b, bool aniso,
                                const AdmmCoef& K, float cu_in, int iters,
                                const PottsRowsMaps& M, int* err, cudaStream_t st);
cudaError_t potts_rows_tile_step_f32(const PottsProblem& P, const PottsStateV& b, bool aniso,
                                     const AdmmCoef& K, float cu_in, int iters,
                                     const PottsRowsMaps& M, int fused, int* err,
                                     cudaStream_t st);
cudaError_t potts_rows_step_f16(const PottsProblem& P, const PottsStateV& b, bool aniso,
                                const AdmmCoef& K, float cu_in, int iters,
                                const PottsRowsMaps& M, int* err, cudaStream_t st);
cudaError_t potts_rows_tile_step_f16(const PottsProblem& P, const PottsStateV& b, bool aniso,
                                     const AdmmCoef& K, float cu_in, int iters,
                                     const PottsRowsMaps& M, int fused, int* err,
                                     cudaStream_t st);
cudaError_t potts_rows_step_bf16(const PottsProblem& P, const PottsStateV& b, bool aniso,
                                 const AdmmCoef& K, float cu_in, int iters,
                                 const PottsRowsMaps& M, int* err, cudaStream_t st);
cudaError_t potts_rows_tile_step_bf16(const PottsProblem& P, const PottsStateV& b, bool aniso,
                                      const AdmmCoef& K, float cu_in, int iters,
                                      const PottsRowsMaps& M, int fused, int* err,
                                      cudaStream_t st);

cudaError_t potts_cert_f32(const PottsProblem& P, const PottsRowsMaps& M, bool aniso, bool dr,
                           float tau, double* partials, const EvalTail& T, int* err,
                           cudaStream_t st);
cudaError_t potts_cert_f16(const PottsProblem& P, const PottsRowsMaps& M, bool aniso, bool dr,
                           float tau, double* partials, const EvalTail& T, int* err,
                           cudaStream_t st);
cudaError_t potts_cert_bf16(const PottsProblem& P, const PottsRowsMaps& M, bool aniso, bool dr,
                            float tau, double* partials, const EvalTail& T, int* err,
                            cudaStream_t st);

cudaError_t potts_dr_rows_f32(const PottsProblem& P, const PottsStateV& b, bool aniso,
                              const DrCoef& D, const PottsRowsMaps& M, int* err, cudaStream_t st);
cudaError_t potts_dr_rows_f16(const PottsProblem& P, const PottsStateV& b, bool aniso,
                              const DrCoef& D, const PottsRowsMaps& M, int* err, cudaStream_t st);
cudaError_t potts_dr_rows_bf16(const PottsProblem& P, const PottsStateV& b, bool aniso,
                               const DrCoef& D, const PottsRowsMaps& M, int* err, cudaStream_t st);

bool potts_rows_eligible(const PottsProblem& P, int storage, const AdmmCoef& K,
                         const PottsStateV& a, const PottsStateV& b) {
    return !(P.g.W % 2 && (K.ty || K.cp)) && potts_rows_layout(P, storage, a, b);
}

bool potts_rows_layout(const PottsProblem& P, int storage, const PottsStateV& a,
                       const PottsStateV& b) {
    const Grid& G = P.g;
    if (P.L > rows::kMaxLabels || cost_src(P) != kCostF32) return false;
    // the last pair of an odd width writes its first element alone, every
    // other one a pair at an even offset
    if (G.plane > (size_t)INT_MAX || G.plane * (size_t)P.L > (size_t)UINT_MAX) return false;
    const size_t es = dtype_size(storage);
    if ((G.pitch * es) % 16 || (G.pitch * 4) % 16) return false;
    auto al = [](const void* p) { return ((uintptr_t)p % 16) == 0; };
    if (!al(P.C) || (P.alpha.plane && !al(P.alpha.plane))) return false;
    for (const PottsStateV* s : {&a, &b})
        if (!al(s->u) || !al(s->qx) || !al(s->qy) || !al(s->p) || !al(s->ps)) return false;
    return true;
}

int potts_rows_fused(const PottsProblem& P, int storage, bool aniso) {
    return P.g.W % 2 ? potts_tma_auto_ty(storage, aniso, P.L) == 16 : 0;
}

cudaError_t potts_rows_maps(const PottsProblem& P, int storage, const PottsStateV& s,
                            PottsRowsMaps& m, const PottsRowsMaps* planes) {
    const Grid& G = P.g;
    const int es = (int)dtype_size(storage);
    const int cs = es == 4 ? rows::Seg<4>::cols : rows::Seg<2>::cols, c4 = rows::Seg<4>::cols;
    const struct {
        CUtensorMap* map;
        const void* base;
        int es, planes, box;
    } f[] = {{&m.qx, s.qx, es, P.L, cs}, {&m.qy, s.qy, es, P.L, cs}, {&m.p, s.p, es, P.L, cs},
              {&m.u, s.u, 4, P.L, c4},    {&m.ps, s.ps, 4, 1, c4},    {&m.C, P.C, 4, P.L, c4},
              {&m.al, P.alpha.plane, 4, 1, c4}};
    for (const auto& q : f) {
        if (planes && q.map == &m.C) {
            m.C = planes->C;
            m.al = planes->al;
            break;
        }
        if (!q.base) {  // constant alpha: its map is never read
            *q.map = m.ps;
            continue;
        }
        const cudaError_t e = encode_tma_3d(q.map, q.base, q.es, G.W, G.H, q.planes, G.pitch,
                                            q.box, 1, q.planes);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t potts_rows_step(int storage, const PottsProblem& P, const PottsStateV& b, bool aniso,
                            const AdmmCoef& K, float cu_in, int iters, const PottsRowsMaps& M,
                            int fused, int* err, cudaStream_t st) {
    if (P.g.W % 2) {
        switch (storage) {
            case CMF_F32:
                return potts_rows_tile_step_f32(P, b, aniso, K, cu_in, iters, M, fused, err, st);
            case CMF_F16:
                return potts_rows_tile_step_f16(P, b, aniso, K, cu_in, iters, M, fused, err, st);
            default:
                return potts_rows_tile_step_bf16(P, b, aniso, K, cu_in, iters, M, fused, err, st);
        }
    }
    switch (storage) {
        case CMF_F32: return potts_rows_step_f32(P, b, aniso, K, cu_in, iters, M, err, st);
        case CMF_F16: return potts_rows_step_f16(P, b, aniso, K, cu_in, iters, M, err, st);
        default: return potts_rows_step_bf16(P, b, aniso, K, cu_in, iters, M, err, st);
    }
}

cudaError_t potts_cert(int storage, const PottsProblem& P, const PottsRowsMaps& M, bool aniso,
                       bool dr, float tau, double* partials, const EvalTail& T, int* err,
                       cudaStream_t st) {
    switch (storage) {
        case CMF_F32: return potts_cert_f32(P, M, aniso, dr, tau, partials, T, err, st);
        case CMF_F16: return potts_cert_f16(P, M, aniso, dr, tau, partials, T, err, st);
        default: return potts_cert_bf16(P, M, aniso, dr, tau, partials, T, err, st);
    }
}

bool potts_dr_rows_takes(const PottsProblem& P, const DrCoef& D) {
    // one sweep, two columns per lane.  Against the strips faster at every size
    // measured, 128^2 to 2048^2 and L = 2 to 16 (L = 2, 1024^2 51 -> 28 us;
    // L = 4, 512^2 22.6 -> 16.5; L = 16, 2048^2 759 -> 520), with the same
    // results; more labels, more sweeps and odd widths stay where they were.
    return D.sweeps == 1 && P.g.W % 2 == 0;
}

cudaError_t potts_dr_rows_step(int storage, const PottsProblem& P, const PottsStateV& b,
                               bool aniso, const DrCoef& D, const PottsRowsMaps& M, int* err,
                               cudaStream_t st) {
    switch (storage) {
        case CMF_F32: return potts_dr_rows_f32(P, b, aniso, D, M, err, st);
        case CMF_F16: return potts_dr_rows_f16(P, b, aniso, D, M, err, st);
        default: return potts_dr_rows_bf16(P, b, aniso, D, M, err, st);
    }
}

}  // namespace cmf
