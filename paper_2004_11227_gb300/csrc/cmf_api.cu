// C-ABI layer of libcmf: argument validation, workspace layout, the
// iteration / certificate / solve drivers.  See include/cmf.h for the
// contract of every entry point.
#include <math.h>
#include <string.h>

#include <initializer_list>
#include <mutex>
#include <vector>

#include "cmf_kernels.cuh"
#include "cmf_tma.cuh"

using namespace cmf;

namespace {

constexpr size_t kAlign = 256;
inline size_t align_up(size_t x) { return (x + kAlign - 1) / kAlign * kAlign; }

// Workspace regions (offsets from the workspace base).
struct WsLayout {
    size_t phase;     // two state sets in phase_storage (two-phase Potts solves)
    size_t phase_set; // bytes of one of them
    size_t state;     // second state buffer set (ping-pong of the fused form)
    size_t state2;    // third set (binary fused form: routes two-iteration launches)
    size_t tmp;       // float planes used by the plain form
    size_t usum;      // two float planes of sum_i u_i (Potts rPDRQ by warp strips)
    size_t partials;  // 3 doubles per certificate block
    size_t scalars;   // 4 doubles
    size_t ctl;       // solve-loop control block (graph path)
    size_t hist;      // device history rows (graph path)
    size_t total;
};

size_t hist_rows_for(const cmf_params& p);

WsLayout ws_layout(int H, int W, int L, int pitch, const cmf_params& p, bool potts) {
    const size_t plane = (size_t)H * (size_t)pitch;
    const size_t es = dtype_size(p.storage);
    // one state set: u planes (float32), flow planes in the storage type, and
    // for Potts the float32 p_s plane; the Potts per-label planes are packed
    // [L][H][pitch]
    const size_t set = potts ? align_up(plane * 4 * L) + 3 * align_up(plane * es * L) +
                                   align_up(plane * 4)
                             : align_up(plane * 4) + 4 * align_up(plane * es);
    WsLayout w;
    size_t off = 0;
    w.phase = off;
    w.phase_set = 0;
    if (potts && p.phase_storage != 0) {
        const size_t ep = dtype_size(p.phase_storage);
        w.phase_set = align_up(plane * 4 * L) + 3 * align_up(plane * ep * L) + align_up(plane * 4);
        off += 2 * w.phase_set;
    }
    w.state = off;
    off += set;
    w.state2 = off;
    if (!potts && p.impl == CMF_FUSED) off += set;
    w.tmp = off;
    // plain forms: g and div q^{k+1} (per label for Potts); the fused kernels
    // keep everything on chip
    off += align_up(plane * 4 * (size_t)(p.impl == CMF_PLAIN ? (potts ? 2 * L : 2) : 0));
    w.usum = off;
    // fused Potts rPDRQ: each launch writes sum_i u_i of its output for the
    // next launch (ping-pong)
    if (potts && p.algo == CMF_RPDRQ && p.impl == CMF_FUSED) off += 2 * align_up(plane * 4);
    w.partials = off;
    {
        // one triple per certificate block: the certificate kernels' grid, or
        // the two-iteration launch that certifies its result
        const size_t nb = (size_t)eval_blocks(H, W);
        const size_t nc = (!potts && p.impl == CMF_FUSED) ? (size_t)binary_cert_max_blocks() : 0;
        off += align_up(sizeof(double) * 3 * (nb > nc ? nb : nc));
    }
    w.scalars = off;
    off += align_up(sizeof(double) * 4);
    w.ctl = off;
    off += align_up(64);
    w.hist = off;
    off += align_up(sizeof(double) * 5 * hist_rows_for(p));
    w.total = off;
    return w;
}

bool aligned(const void* ptr, size_t a) { return ((uintptr_t)ptr % a) == 0; }

cmf_status check_params(const cmf_params* p, int L) {
    if (!p) return CMF_EINVAL;
    if (p->algo < CMF_PADMM || p->algo > CMF_CP) return CMF_EINVAL;
    if (p->storage < CMF_F32 || p->storage > CMF_BF16) return CMF_EINVAL;
    if (p->impl != CMF_FUSED && p->impl != CMF_PLAIN) return CMF_EINVAL;
    if (p->sweeps < 1 || (p->impl == CMF_FUSED && p->sweeps > 4) || p->sweeps > 64)
        return CMF_EINVAL;
    if (!(p->c > 0) || !(p->a > 0) || !(p->a1 > 0) || !(p->a2 >= 0)) return CMF_EINVAL;
    if (!(p->rho > 0) || !(p->rho < 2)) return CMF_EINVAL;
    if (!(p->r > 0) || !(p->sigma > 0) || !(p->tau > 0)) return CMF_EINVAL;
    if (p->max_iter < 0 || p->check_every < 1 || !(p->tol_gap >= 0)) return CMF_EINVAL;
    if (p->variant != 0 && p->variant != 1 && p->variant != 2 && p->variant != 4 &&
        p->variant != 8 && p->variant != 16 && p->variant != 32)
        return CMF_EINVAL;
    if (p->costs < 0 || p->costs > 2) return CMF_EINVAL;
    if (p->tune_step != 0 && p->tune_step != 1) return CMF_EINVAL;
    // two-phase Potts solves: a 16-bit first phase, the caller's buffers float32
    if (p->phase_storage < 0 || p->phase_storage > CMF_BF16) return CMF_EINVAL;
    if (p->phase_storage != 0 &&
        (p->storage != CMF_F32 || !(p->phase_gap > p->tol_gap) || p->rho_schedule_len != 0 ||
         p->warm_start != 0))
        return CMF_EINVAL;
    // relaxation schedule {rho_k}: non-decreasing in (0, 2) (Thm 1, Thm 2),
    // continued by rho, for the two relaxed algorithms only
    if (p->rho_schedule_len < 0) return CMF_EINVAL;
    if (p->rho_schedule_len > 0) {
        if (!p->rho_schedule) return CMF_EINVAL;
        if (p->algo != CMF_RPADMM_EB && p->algo != CMF_RPDRQ) return CMF_EINVAL;
        double prev = 0.0;
        for (int k = 0; k < p->rho_schedule_len; ++k) {
            const double r = p->rho_schedule[k];
            if (!(r > 0) || !(r < 2) || !(r >= prev)) return CMF_EINVAL;
            prev = r;
        }
        if (!(prev <= p->rho)) return CMF_EINVAL;
    }
    (void)L;
    return CMF_OK;
}

cmf_status check_grid(int H, int W, int pitch) {
    if (H < 1 || W < 1 || pitch < W) return CMF_EINVAL;
    if ((double)H * (double)pitch > 4.0e12) return CMF_EINVAL;
    return CMF_OK;
}

Alpha make_alpha(const float* d_alpha, float alpha0) { return Alpha{d_alpha, alpha0}; }

Grid make_grid(int H, int W, int pitch) {
    return Grid{H, W, pitch, (size_t)H * (size_t)pitch};
}

// The Potts problem as the kernels see it.  costs == 1: d_C holds the image
// plane followed by the L levels; costs == 2: d_C holds L float16 planes.
PottsProblem potts_problem(const float* C, int L, const float* alpha, float alpha0, int H,
                           int W, int pitch, int costs) {
    PottsProblem P{C, L, make_alpha(alpha, alpha0), make_grid(H, W, pitch), nullptr, nullptr};
    if (costs == 1) P.lev = C + (size_t)H * (size_t)pitch;
    if (costs == 2) P.C16 = reinterpret_cast<const __half*>(C);
    return P;
}

StepConfig make_step(const cmf_params& p, int L, bool potts) {
    StepConfig s;
    s.dr = p.algo == CMF_RPDRQ;
    s.aniso = p.aniso != 0;
    s.plain = p.impl == CMF_PLAIN;
    s.ac = make_admm_coef(p, L);
    s.dc = make_dr_coef(p, L, potts);
    return s;
}

// Coefficients of iteration k (counted from the start of the call): the
// scheduled rho_k where the schedule covers k, else the call's own.
StepConfig step_at(const StepConfig& base, const cmf_params& p, int L, bool potts, int k) {
    if (k >= p.rho_schedule_len) return base;
    cmf_params q = p;
    q.rho = p.rho_schedule[k];
    return make_step(q, L, potts);
}

// ---- binary ---------------------------------------------------------------

BinStateV ws_binary_state(char* ws, size_t off, const Grid& G, int storage) {
    const size_t plane = G.plane;
    const size_t es = dtype_size(storage);
    char* base = ws + off;
    BinStateV s;
    s.u = (float*)base;
    base += align_up(plane * 4);
    void** f[4] = {&s.qx, &s.qy, &s.ps, &s.pt};
    for (int i = 0; i < 4; ++i) {
        *f[i] = base;
        base += align_up(plane * es);
    }
    return s;
}

cudaError_t copy_plane(void* dst, const void* src, const Grid& G, size_t es, cudaStream_t st) {
    if (dst == src) return cudaSuccess;
    return cudaMemcpy2DAsync(dst, G.pitch * es, src, G.pitch * es, G.W * es, G.H,
                             cudaMemcpyDeviceToDevice, st);
}

cudaError_t copy_binary(const BinStateV& dst, const BinStateV& src, const Grid& G, int storage,
                        cudaStream_t st) {
    const size_t es = dtype_size(storage);
    cudaError_t e;
    if ((e = copy_plane(dst.u, src.u, G, 4, st)) != cudaSuccess) return e;
    if ((e = copy_plane(dst.qx, src.qx, G, es, st)) != cudaSuccess) return e;
    if ((e = copy_plane(dst.qy, src.qy, G, es, st)) != cudaSuccess) return e;
    if ((e = copy_plane(dst.ps, src.ps, G, es, st)) != cudaSuccess) return e;
    return copy_plane(dst.pt, src.pt, G, es, st);
}

struct BinaryCall {
    BinProblem P;
    BinStateV user, ws, ws2;  // buffer sets 0, 1, 2 (set 2: fused form only)
    WsLayout w;
    char* wsbase;
    StepConfig cfg;
    cmf_params prm;         // the call's parameters (rho schedule)
    int storage;
    bool tma;               // fused ADMM through the persistent TMA kernel
    bool strip;             // fused ADMM by warp strips
    bool pairs;             // warp strips, two ADMM iterations per launch
    bool alone;             // chain: iterations that run alone run by strips or TMA tiles
    bool chain;             // chains of warps, up to four ADMM iterations per launch
    bool dr_rows;           // rPDRQ on shared TMA rows
    // tensor maps of the buffer sets (chain, dr_rows), encoded by binary_maps
    // where a launch first reads a set
    mutable BinChainMaps cmaps[3];
    mutable int mapped = 0;  // the sets encoded, a bit each
    int cert_blocks;        // partial triples the workspace holds
    // tensor maps of the user / workspace state sets (tma); with chain encoded by
    // one_iteration where a launch first reads a set
    mutable BinTmaMaps maps[2];
    mutable int tma_mapped = 0;  // the sets encoded, a bit each
    int* err;               // sticky device error word
};

cmf_status binary_prepare(const float* Cs, const float* Ct, const float* alpha, float alpha0,
                          int H, int W, int pitch, const cmf_params* p, float* u, void* qx,
                          void* qy, void* ps, void* pt, void* ws, size_t ws_bytes,
                          BinaryCall& call) {
    cmf_status s;
    if ((s = check_params(p, 2)) != CMF_OK) return s;
    if (p->costs != 0) return CMF_EINVAL;  // binary costs are planes
    if (p->phase_storage != 0) return CMF_EINVAL;  // two-phase solves: Potts only
    if ((s = check_grid(H, W, pitch)) != CMF_OK) return s;
    if (!Cs || !Ct || !u || !qx || !qy || !ps || !pt || !ws) return CMF_EINVAL;
    if (!alpha && !(alpha0 >= 0.0f && isfinite(alpha0))) return CMF_EINVAL;
    const size_t es = dtype_size(p->storage);
    if (!aligned(u, 4) || !aligned(Cs, 4) || !aligned(Ct, 4) || (alpha && !aligned(alpha, 4)))
        return CMF_EINVAL;
    if (!aligned(qx, es) || !aligned(qy, es) || !aligned(ps, es) || !aligned(pt, es))
        return CMF_EINVAL;
    if (!aligned(ws, kAlign)) return CMF_EINVAL;
    call.w = ws_layout(H, W, 2, pitch, *p, false);
    if (ws_bytes < call.w.total) return CMF_ENOMEM;
    call.P = BinProblem{Cs, Ct, make_alpha(alpha, alpha0), make_grid(H, W, pitch)};
    call.user = BinStateV{u, qx, qy, ps, pt};
    call.wsbase = (char*)ws;
    call.ws = ws_binary_state(call.wsbase, call.w.state, call.P.g, p->storage);
    call.ws2 = ws_binary_state(call.wsbase, call.w.state2, call.P.g, p->storage);
    call.cfg = make_step(*p, 2, false);
    call.prm = *p;
    call.storage = p->storage;
    call.err = &((SolveCtl*)(call.wsbase + call.w.ctl))->err;
    call.tma = false;
    call.strip = false;
    call.pairs = false;
    call.chain = false;
    call.dr_rows = false;
    // automatic choice: chains of warps (against pairs of iterations by warp
    // strips 8.25 -> 5.73 us per iteration at 1024^2, 87 -> 52 us at 4096^2;
    // odd widths, against tiles, 16 -> 7.2 us at 901 x 1407; the same results)
    if (!call.cfg.plain && !call.cfg.dr &&
        (p->variant == 0 || (p->variant == 4 && W % 2 == 0)) &&
        binary_chain_eligible(call.P, p->storage, call.user, call.ws, call.ws2) &&
        tma_available()) {
        call.chain = true;
        // The iterations that run alone (a rho schedule's, a remainder) keep the
        // kernels that made one a launch, with the same results, where a chain of
        // one warp is slower: warp strips at even widths up to 1024^2 (512^2 8.6
        // -> 6.5 us, 1024^2 12.7 -> 12.6; 1448^2 18.8 against 21.4) and with
        // 16-bit flows everywhere (1024^2 13.8 -> 10.7 us, 4096^2 107 -> 101), TMA
        // tiles at odd ones up to that size (512 x 513 8.6 -> 6.6 us, 1024 x 1025
        // equal; 1448 x 1447 20.9 against 29.3).
        const bool small = (size_t)H * (size_t)W <= (size_t)1 << 20;
        call.strip = W % 2 == 0 && binary_strip_eligible(call.P.g, p->storage, Cs, Ct, alpha,
                                                         call.user, call.ws);
        call.alone = call.strip && (small || es == 2);
        if (W % 2) {
            call.tma = call.alone = small && binary_tma_eligible(call.P.g, p->storage, call.user) &&
                                    binary_tma_eligible(call.P.g, p->storage, call.ws);
        }
        const int nb = eval_blocks(H, W), nc = binary_cert_max_blocks();
        call.cert_blocks = nb > nc ? nb : nc;
        return CMF_OK;
    }
    // rPDRQ, one sweep: strips on shared TMA rows (against the one-warp strips
    // faster at every size measured, 64^2 12.4 -> 6.2 us to 4096^2 174 -> 145 us
    // per iteration, with the same results)
    if (!call.cfg.plain && call.cfg.dr && p->variant == 0 &&
        binary_dr_rows_eligible(call.P, p->storage, call.cfg.dc, call.user, call.ws) &&
        tma_available()) {
        call.dr_rows = true;
        return CMF_OK;
    }
    // else warp strips where the layout allows them, two ADMM iterations per
    // launch (1.5x faster per iteration than one at 1024^2, 1.9x at 4096^2);
    // rPDRQ: the pipelined red-black sweeps
    if (!call.cfg.plain && (p->variant == 2 || p->variant == 4 || p->variant == 0)) {
        const bool ok =
            binary_strip_eligible(call.P.g, p->storage, Cs, Ct, alpha, call.user, call.ws);
        if (!ok && p->variant != 0)
            return CMF_EINVAL;  // warp strips requested but the layout does not allow them
        if (ok) {
            call.strip = true;
            call.pairs = p->variant != 2 && !call.cfg.dr;
            return CMF_OK;
        }
    }
    const int ty = p->variant >= 8 ? p->variant : 16;
    // automatic choice: the persistent TMA kernel wins on grids that fit the
    // L2 cache, the shared-memory tile kernel on larger ones (measured)
    const bool auto_tma = p->variant == 0 && (size_t)H * (size_t)W <= ((size_t)1 << 21);
    if (!call.cfg.dr && !call.cfg.plain && (p->variant >= 8 || auto_tma) &&
        binary_tma_eligible(call.P.g, p->storage, call.user) &&
        binary_tma_eligible(call.P.g, p->storage, call.ws)) {
        call.tma = binary_tma_maps(call.P.g, p->storage, call.user, ty, call.maps[0]) ==
                       cudaSuccess &&
                   binary_tma_maps(call.P.g, p->storage, call.ws, ty, call.maps[1]) ==
                       cudaSuccess;
    }
    if (!call.tma && !call.cfg.dr && !call.cfg.plain && p->variant >= 8)
        return CMF_EINVAL;  // TMA tiles requested but the layout does not allow them
    return CMF_OK;
}

const BinStateV& bset(const BinaryCall& c, int i) {
    return i == 0 ? c.user : (i == 1 ? c.ws : c.ws2);
}

// The tensor maps of buffer set i.  All three sets' (24 driver calls, 3.5 us of a
// 50 us certificate call at 64^2) are seldom read: certificates and replayed graphs
// read none, one iteration reads the caller's.
cudaError_t binary_maps(const BinaryCall& c, int i) {
    if (c.mapped >> i & 1) return cudaSuccess;
    const BinChainMaps* planes = nullptr;  // of a set already encoded
    for (int k = 0; k < 3; ++k)
        if (c.mapped >> k & 1) planes = &c.cmaps[k];
    const cudaError_t e =
        c.chain ? binary_chain_maps(c.P, c.storage, bset(c, i), c.cmaps[i], planes)
                : binary_dr_rows_maps(c.P, c.storage, bset(c, i), c.cmaps[i], planes);
    if (e == cudaSuccess) c.mapped |= 1 << i;
    return e;
}

// Whether the chain path leaves a lone iteration from set src into set dst to the
// kernels that make one a launch: where binary_prepare chose one, among the first
// two sets, and (iter0: its index among the call's unscheduled iterations) not
// the second of a pair with 16-bit flows, whose roundings are the pair's.
bool runs_alone(const BinaryCall& c, int src, int dst, int iter0) {
    if (src > 1 || dst > 1 || !c.alone) return false;
    return !(c.strip && c.storage != CMF_F32 && (iter0 & 1));
}

// That iteration (AdmmCoef: the scheduled one where a schedule covers it).
cudaError_t one_iteration(const BinaryCall& c, int src, int dst, const StepConfig& cfg,
                          cudaStream_t st) {
    if (c.strip)
        return binary_strip_step(c.storage, c.P, bset(c, src), bset(c, dst), cfg.aniso, cfg.ac,
                                 st);
    if (!(c.tma_mapped >> src & 1)) {
        const cudaError_t e =
            binary_tma_maps(c.P.g, c.storage, bset(c, src), 16, c.maps[src]);
        if (e != cudaSuccess) return e;
        c.tma_mapped |= 1 << src;
    }
    return binary_admm_tma_step(c.storage, c.P, bset(c, dst), cfg.aniso, cfg.ac, c.maps[src],
                                c.err, st);
}

// Run n iterations starting from `cur` (0 = user buffers, 1 = workspace,
// 2 = the workspace's third set, used by the two-iteration launches);
// returns the index of the buffer set holding the result.  k0 is the index of
// the first of them within the call (for the rho schedule).  cert != nullptr:
// also certify the result with that tail (in the last two-iteration launch
// when there is one, else with the certificate kernel).  dry: launch
// nothing, only follow the buffer sets.
cudaError_t binary_run(const BinaryCall& c, int n, int& cur, cudaStream_t st, int k0 = 0,
                       const EvalTail* cert = nullptr, bool dry = false) {
    float* tmp = (float*)(c.wsbase + c.w.tmp);
    double* partials = (double*)(c.wsbase + c.w.partials);
    bool certified = false;
    // Two-iteration launches after the scheduled iterations (one single
    // launch for an odd remainder).  With three buffer sets a run of at least
    // two launches ends in the set it started from: start -> x -> y -> x ...
    // -> start, x and y the other two sets; a lone launch goes to the
    // caller's set, or from it to the workspace.
    int i = 0;
    // A call of three or four iterations: pairs by warp strips up to 1448^2, which
    // need no tensor maps and no longer chains (64^2 29.9 -> 28.5 us, 1024^2 49.2
    // -> 45.6 a call; 2048^2 106 against 93; the same results).
    const bool pairs = c.pairs || (c.chain && c.strip && !cert && n >= 3 && n <= 4 &&
                                   c.prm.rho_schedule_len <= k0 &&
                                   (size_t)c.P.g.H * (size_t)c.P.g.W <= (size_t)1 << 21);
    if (c.chain && !pairs) {
        // one iteration per launch while the rho schedule lasts, then launches
        // of up to four iterations, at least two of them; the last one carries
        // the certificates
        const int sched = c.prm.rho_schedule_len > k0 ? c.prm.rho_schedule_len - k0 : 0;
        const int first = sched < n ? sched : n;
        const bool may_cert = cert && binary_chain_certifies(c.P.g, c.cert_blocks);
        const int rest = n - first, most = binary_chain_max_iters(false);
        int nl = rest < 2 ? rest : (rest + most - 1) / most;  // launches of the rest
        if (nl == 1 && rest > 1) nl = 2;
        if (may_cert && rest > 0 && rest / nl > binary_chain_max_iters(true)) ++nl;
        int start = cur;
        for (int j = 0; j < first + nl; ++j) {
            const int m = j - first;  // m >= 0: a launch of the rest
            if (m <= 0) start = cur;
            const int x = start == 0 ? 1 : 0, y = start == 2 ? 1 : 2;
            const int T = m < 0 ? 1 : rest / nl + (m < rest % nl ? 1 : 0);
            const int dst = m < 0 || nl == 1 ? (cur == 0 ? 1 : 0)
                                             : (m == nl - 1 ? start : (m % 2 == 0 ? x : y));
            certified = may_cert && j == first + nl - 1;
            if (!dry) {
                const StepConfig cfg = m < 0 ? step_at(c.cfg, c.prm, 2, false, k0 + j) : c.cfg;
                const bool alone = T == 1 && !certified && runs_alone(c, cur, dst, i);
                cudaError_t e =
                    alone ? one_iteration(c, cur, dst, cfg, st) : binary_maps(c, cur);
                if (e == cudaSuccess && !alone)
                    e = binary_chain_step(c.storage, c.P, bset(c, dst), cfg.aniso, cfg.ac, T, i,
                                          c.cmaps[cur], partials, c.cert_blocks,
                                          certified ? cert : nullptr, c.err, st);
                if (e != cudaSuccess) return e;
            }
            if (m >= 0) i += T;
            cur = dst;
        }
        i = n;
    }
    if (pairs) {
        const int sched = c.prm.rho_schedule_len > k0 ? c.prm.rho_schedule_len - k0 : 0;
        const int first = sched < n ? sched : n;
        for (; i < first; ++i) {
            const StepConfig cfg = step_at(c.cfg, c.prm, 2, false, k0 + i);
            const int dst = cur == 0 ? 1 : 0;
            if (!dry) {
                cudaError_t e = binary_strip_step(c.storage, c.P, bset(c, cur), bset(c, dst),
                                                  cfg.aniso, cfg.ac, st);
                if (e != cudaSuccess) return e;
            }
            cur = dst;
        }
        const int npairs = (n - first) / 2, nsingle = (n - first) % 2;
        const int nl = npairs + nsingle;
        const int start = cur;
        const int x = start == 0 ? 1 : 0, y = start == 2 ? 1 : 2;
        for (int j = 0; j < nl; ++j) {
            const int dst = nl == 1 ? (start == 0 ? 1 : 0)
                                    : (j == nl - 1 ? start : (j % 2 == 0 ? x : y));
            // the last pair launch carries the certificates when no single follows it
            const bool cj = cert && j == npairs - 1 && nsingle == 0;
            if (!dry) {
                const BinStateV& a = bset(c, cur);
                const BinStateV& b = bset(c, dst);
                cudaError_t e =
                    j < npairs ? binary_strip2_step(c.storage, c.P, a, b, c.cfg.aniso, c.cfg.ac,
                                                    st, cj ? cert : nullptr, partials)
                               : binary_strip_step(c.storage, c.P, a, b, c.cfg.aniso, c.cfg.ac,
                                                   st);
                if (e != cudaSuccess) return e;
            }
            certified = certified || cj;
            cur = dst;
        }
        i = n;
    }
    for (; i < n; ++i) {
        const StepConfig cfg = step_at(c.cfg, c.prm, 2, false, k0 + i);
        if (cfg.plain) {
            if (!dry) {
                cudaError_t e = binary_step(c.storage, c.P, c.user, c.user, cfg, tmp, st);
                if (e != cudaSuccess) return e;
            }
            cur = 0;
        } else if (c.dr_rows) {
            if (!dry) {
                cudaError_t e = binary_maps(c, cur);
                if (e == cudaSuccess)
                    e = binary_dr_rows_step(c.storage, c.P, cur == 0 ? c.ws : c.user, cfg.aniso,
                                            cfg.dc, c.cmaps[cur], c.err, st);
                if (e != cudaSuccess) return e;
            }
            cur ^= 1;
        } else if (c.strip) {
            const BinStateV& a = cur == 0 ? c.user : c.ws;
            const BinStateV& b = cur == 0 ? c.ws : c.user;
            if (!dry) {
                cudaError_t e =
                    cfg.dr ? binary_dr_strip_step(c.storage, c.P, a, b, cfg.aniso, cfg.dc, st)
                           : binary_strip_step(c.storage, c.P, a, b, cfg.aniso, cfg.ac, st);
                if (e != cudaSuccess) return e;
            }
            cur ^= 1;
        } else if (c.tma) {
            const BinStateV& b = cur == 0 ? c.ws : c.user;
            if (!dry) {
                cudaError_t e = binary_admm_tma_step(c.storage, c.P, b, cfg.aniso, cfg.ac,
                                                     c.maps[cur], c.err, st);
                if (e != cudaSuccess) return e;
            }
            cur ^= 1;
        } else {
            const BinStateV& a = cur == 0 ? c.user : c.ws;
            const BinStateV& b = cur == 0 ? c.ws : c.user;
            if (!dry) {
                cudaError_t e = binary_step(c.storage, c.P, a, b, cfg, tmp, st);
                if (e != cudaSuccess) return e;
            }
            cur ^= 1;
        }
    }
    if (cert && !certified && !dry)
        return binary_eval(c.storage, c.P, bset(c, cur), c.cfg.aniso, c.cfg.dr, c.cfg.dc.tau,
                           partials, st, *cert);
    return cudaSuccess;
}

// The certificate launch has reduced its partials into the scalars (its last
// block); read them and the error word.
cmf_status finish_eval(char* wsbase, const WsLayout& w, double* h_out, cudaStream_t st) {
    double* scal = (double*)(wsbase + w.scalars);
    double h[3];
    CMF_CUDA_TRY(cudaMemcpyAsync(h, scal, sizeof(h), cudaMemcpyDeviceToHost, st));
    int* err = &((SolveCtl*)(wsbase + w.ctl))->err;
    int herr = 0;
    CMF_CUDA_TRY(cudaMemcpyAsync(&herr, err, sizeof(int), cudaMemcpyDeviceToHost, st));
    CMF_CUDA_TRY(cudaStreamSynchronize(st));
    if (herr == kErrWaitTimeout) {
        CMF_CUDA_TRY(cudaMemsetAsync(err, 0, sizeof(int), st));
        return CMF_ETIMEOUT;
    }
    const double E = h[0], D = h[1];
    h_out[0] = E;
    h_out[1] = D;
    h_out[2] = (E - D) / (fabs(E) > 1e-30 ? fabs(E) : 1e-30);
    h_out[3] = sqrt(h[2] > 0 ? h[2] : 0.0);
    return CMF_OK;
}

// The certificate launch with its own reduction (no stop decision).
EvalTail reduce_tail(char* wsbase, const WsLayout& w) {
    EvalTail T;
    T.ctl = (SolveCtl*)(wsbase + w.ctl);
    T.scal = (double*)(wsbase + w.scalars);
    return T;
}

cmf_status binary_eval_state(const BinaryCall& c, const BinStateV& s, double* h_out,
                             cudaStream_t st) {
    const EvalTail T = reduce_tail(c.wsbase, c.w);
    CMF_CUDA_TRY(cudaMemsetAsync(&T.ctl->arrive, 0, sizeof(unsigned), st));
    CMF_CUDA_TRY(binary_eval(c.storage, c.P, s, c.cfg.aniso, c.cfg.dr, c.cfg.dc.tau,
                             (double*)(c.wsbase + c.w.partials), st, T));
    return finish_eval(c.wsbase, c.w, h_out, st);
}

// ---- Potts ----------------------------------------------------------------

PottsStateV ws_potts_state(char* ws, size_t off, const Grid& G, int L, int storage) {
    const size_t plane = G.plane;
    const size_t es = dtype_size(storage);
    char* base = ws + off;
    PottsStateV s;
    s.u = (float*)base;
    base += align_up(plane * 4 * L);
    s.qx = base;
    base += align_up(plane * es * L);
    s.qy = base;
    base += align_up(plane * es * L);
    s.p = base;
    base += align_up(plane * es * L);
    s.ps = (float*)base;
    return s;
}

cudaError_t copy_potts(const PottsStateV& dst, const PottsStateV& src, const Grid& G, int L,
                       int storage, cudaStream_t st) {
    const size_t es = dtype_size(storage);
    cudaError_t e;
    for (int i = 0; i < L; ++i) {
        const size_t o4 = G.plane * 4 * i, oe = G.plane * es * i;
        if ((e = copy_plane((char*)dst.u + o4, (char*)src.u + o4, G, 4, st)) != cudaSuccess)
            return e;
        if ((e = copy_plane((char*)dst.qx + oe, (char*)src.qx + oe, G, es, st)) != cudaSuccess)
            return e;
        if ((e = copy_plane((char*)dst.qy + oe, (char*)src.qy + oe, G, es, st)) != cudaSuccess)
            return e;
        if ((e = copy_plane((char*)dst.p + oe, (char*)src.p + oe, G, es, st)) != cudaSuccess)
            return e;
    }
    return copy_plane(dst.ps, src.ps, G, 4, st);  // p_s: float32
}

struct PottsCall {
    PottsProblem P;
    PottsStateV user, ws;
    WsLayout w;
    char* wsbase;
    StepConfig cfg;
    cmf_params prm;              // the call's parameters (rho schedule)
    int storage;
    bool tma;                    // fused ADMM through TMA-staged tiles
    bool strip;                  // fused ADMM by warp strips
    bool rows;                   // fused ADMM, labels side by side, up to two iterations a launch
    bool cert;                   // certificates with the labels side by side
    bool dr_rows;                // rPDRQ with the labels side by side
    // tensor maps of the user / workspace state sets (tma); with rows encoded where
    // a launch first reads a set
    mutable PottsTmaMaps maps[2];
    mutable int tma_mapped = 0;  // the sets encoded, a bit each
    int tma_rows;                // rows of a tile
    // tensor maps of the two sets (rows, dr_rows, cert), encoded by row_maps
    // where a launch first reads a set
    mutable PottsRowsMaps rmaps[2];
    mutable int mapped = 0;  // the sets encoded, a bit each
    int rfused;                  // potts_rows_fused
    int* err;                    // sticky device error word
};

// `layout`: the parameters the workspace was sized for (default *p); `set`:
// the second state set (default: the workspace's own, in p->storage).
cmf_status potts_prepare(const float* C, int L, const float* alpha, float alpha0, int H, int W,
                         int pitch, const cmf_params* p, float* u, void* qx, void* qy, void* pp,
                         void* ps, void* ws, size_t ws_bytes, PottsCall& call,
                         const cmf_params* layout = nullptr, const PottsStateV* set = nullptr) {
    cmf_status s;
    if (L < 2 || L > 64) return CMF_EINVAL;
    if ((s = check_params(p, L)) != CMF_OK) return s;
    if ((s = check_grid(H, W, pitch)) != CMF_OK) return s;
    if (!C || !u || !qx || !qy || !pp || !ps || !ws) return CMF_EINVAL;
    if (!alpha && !(alpha0 >= 0.0f && isfinite(alpha0))) return CMF_EINVAL;
    const size_t es = dtype_size(p->storage);
    if (!aligned(u, 4) || !aligned(C, p->costs == 2 ? 2 : 4) || (alpha && !aligned(alpha, 4)))
        return CMF_EINVAL;
    if (!aligned(qx, es) || !aligned(qy, es) || !aligned(pp, es) || !aligned(ps, 4))
        return CMF_EINVAL;
    if (!aligned(ws, kAlign)) return CMF_EINVAL;
    call.w = ws_layout(H, W, L, pitch, layout ? *layout : *p, true);
    if (ws_bytes < call.w.total) return CMF_ENOMEM;
    call.P = potts_problem(C, L, alpha, alpha0, H, W, pitch, p->costs);
    call.user = PottsStateV{u, qx, qy, pp, (float*)ps};
    call.wsbase = (char*)ws;
    call.ws = set ? *set : ws_potts_state(call.wsbase, call.w.state, call.P.g, L, p->storage);
    call.cfg = make_step(*p, L, true);
    call.prm = *p;
    call.storage = p->storage;
    call.err = &((SolveCtl*)(call.wsbase + call.w.ctl))->err;
    call.tma = false;
    call.strip = false;
    call.rows = false;
    call.dr_rows = false;
    // automatic choice: labels side by side (two iterations a launch; against
    // the strips 150 -> 61.5 us per iteration at 2048^2, L = 4 and 2293 -> 937 us
    // at 4096^2, L = 16, faster at every size measured from 128^2 and L = 2 on,
    // with the same results), else warp strips where the layout allows them,
    // else TMA tiles, else shared-memory tiles
    const bool free_choice = !call.cfg.plain && p->variant == 0;
    const bool dr_rows =
        free_choice && call.cfg.dr && potts_dr_rows_takes(call.P, call.cfg.dc);
    const bool rows =
        free_choice && !call.cfg.dr &&
        potts_rows_eligible(call.P, p->storage, call.cfg.ac, call.user, call.ws);
    const bool side =
        potts_rows_layout(call.P, p->storage, call.user, call.ws) && tma_available();
    // Certificates with the labels side by side, but for two labels in float32 at
    // even widths between 1024^2 and 1448^2, where the strips' take 2 us less (an
    // iteration and its check 69.7 -> 67.7 us and 115.7 -> 113.8; at 900^2 equal, at
    // 724^2 and 2048^2 the strips' take 9 and 7 us more, with 16-bit flows, rPDRQ or
    // more labels always more).
    const size_t px = (size_t)H * (size_t)W;
    call.cert = side && !(L == 2 && es == 4 && W % 2 == 0 && !call.cfg.dr &&
                          px >= (size_t)1 << 20 && px <= (size_t)1 << 21);
    if (dr_rows && side) {
        call.dr_rows = true;
        return CMF_OK;
    }
    if (rows && side) {
        call.rows = true;
        // lone iterations of two labels with 16-bit flows: strips, where two label
        // warps a block leave the rows short of warps (2048^2 69.5 -> 60.8 us,
        // 4096^2 247 -> 233; 1024^2 equal; three labels 76.8 against 85.5; the same
        // results)
        call.strip = L == 2 && es == 2 && px > (size_t)1 << 20 &&
                     potts_strip_eligible(call.P.g, p->storage, C, alpha, call.user, call.ws);
        // at odd widths, where a call is lone iterations throughout, TMA tiles up to
        // 2^20 pixels (1024 x 1023 27.3 -> 25.0 us; 2048 x 2047 89 against 101)
        if (L == 2 && es == 2 && W % 2 && px <= (size_t)1 << 20) {
            call.tma_rows = potts_tma_auto_ty(p->storage, p->aniso, L);
            call.tma = potts_tma_fits(p->storage, L, call.tma_rows) &&
                       potts_tma_eligible(call.P.g, p->storage, call.user) &&
                       potts_tma_eligible(call.P.g, p->storage, call.ws);
        }
        call.rfused = potts_rows_fused(call.P, p->storage, call.cfg.aniso);
        return CMF_OK;
    }
    if (!call.cfg.plain && (p->variant == 2 || p->variant == 4 || p->variant == 0)) {
        const bool ok = potts_strip_eligible(call.P.g, p->storage, C, alpha, call.user, call.ws);
        if (!ok && p->variant != 0)
            return CMF_EINVAL;  // warp strips requested but the layout does not allow them
        if (ok) {
            call.strip = true;
            return CMF_OK;
        }
    }
    const bool want_tma = !call.cfg.dr && !call.cfg.plain && p->variant != 1;
    const int ty = p->variant >= 8 ? p->variant
                                   : (want_tma ? potts_tma_auto_ty(p->storage, p->aniso, L) : 16);
    if (want_tma && potts_tma_fits(p->storage, L, ty) &&
        potts_tma_eligible(call.P.g, p->storage, call.user) &&
        potts_tma_eligible(call.P.g, p->storage, call.ws)) {
        call.tma = potts_tma_maps(call.P.g, L, p->storage, call.user, ty, call.maps[0]) ==
                       cudaSuccess &&
                   potts_tma_maps(call.P.g, L, p->storage, call.ws, ty, call.maps[1]) ==
                       cudaSuccess;
        call.tma_mapped = 3;
    }
    if (!call.tma && !call.cfg.dr && !call.cfg.plain && p->variant >= 8)
        return CMF_EINVAL;  // TMA tiles requested but the layout does not allow them
    return CMF_OK;
}

// The tensor maps of buffer set i (as binary_maps: most calls read one set's or
// none).
cudaError_t row_maps(const PottsCall& c, int i) {
    if (c.mapped >> i & 1) return cudaSuccess;
    const cudaError_t e = potts_rows_maps(c.P, c.storage, i == 0 ? c.user : c.ws, c.rmaps[i],
                                          c.mapped ? &c.rmaps[i ^ 1] : nullptr);
    if (e == cudaSuccess) c.mapped |= 1 << i;
    return e;
}

// The certificate launch for buffer set `set` (0 or 1): labels side by side
// where the layout allows it (a call, host part included: 2048^2, L = 16
// 619 -> 434 us, L = 4 195 -> 158 us; 721 x 1283, L = 8 199 -> 97 us; within a
// solve 1 to 10 us less per check from 8^2 to 512^2), else the strip or tile kernel.
cudaError_t potts_certify(const PottsCall& c, int set, cudaStream_t st, const EvalTail& T) {
    double* partials = (double*)(c.wsbase + c.w.partials);
    if (c.cert) {
        const cudaError_t e = row_maps(c, set);
        if (e != cudaSuccess) return e;
        return potts_cert(c.storage, c.P, c.rmaps[set], c.cfg.aniso, c.cfg.dr, c.cfg.dc.tau,
                          partials, T, c.err, st);
    }
    return potts_eval(c.storage, c.P, set == 0 ? c.user : c.ws, c.cfg.aniso, c.cfg.dr,
                      c.cfg.dc.tau, partials, st, T);
}

// As binary_run: n iterations from buffer set `cur` (0 or 1); cert: certify
// the result with that tail; dry: only follow the buffer sets.  home: with
// two iterations a launch, make the number of launches even where that costs
// one launch more (less than copying a state set back).
cudaError_t potts_run(const PottsCall& c, int n, int& cur, cudaStream_t st, int k0 = 0,
                      const EvalTail* cert = nullptr, bool dry = false, bool home = false) {
    // with two iterations a launch: single ones for the scheduled iterations and an
    // odd remainder
    const int sched = c.prm.rho_schedule_len > k0 ? c.prm.rho_schedule_len - k0 : 0;
    int singles = sched < n ? sched : n;
    singles += (n - singles) % 2;
    if (home && singles + 2 <= n && (singles + (n - singles) / 2) % 2) singles += 2;
    if (c.rows && n > 0 && !(c.tma && singles == n)) {
        float cu_in = 0.0f;  // the first launch reads u itself, later ones the w form
        for (int i = 0; i < n;) {
            const int it = i < singles ? 1 : 2;
            if (!dry) {
                const StepConfig cfg = step_at(c.cfg, c.prm, c.P.L, true, k0 + i);
                const bool alone = it == 1 && c.strip;
                cudaError_t e = alone ? potts_strip_step(c.storage, c.P, cur == 0 ? c.user : c.ws,
                                                         cur == 0 ? c.ws : c.user, cfg.aniso,
                                                         cfg.ac, cu_in, st)
                                      : row_maps(c, cur);
                if (e == cudaSuccess && !alone)
                    e = potts_rows_step(c.storage, c.P, cur == 0 ? c.ws : c.user, cfg.aniso,
                                        cfg.ac, cu_in, it, c.rmaps[cur], c.rfused, c.err, st);
                if (e != cudaSuccess) return e;
            }
            cu_in = c.cfg.ac.cu;
            cur ^= 1;
            i += it;
        }
        if (!dry) {
            cudaError_t e = potts_strip_finalize(c.storage, c.P, cur == 0 ? c.user : c.ws,
                                                 c.cfg.ac.cu, st);
            if (e != cudaSuccess) return e;
        }
        n = 0;
    }
    if (dry) {
        if (n > 0) cur = c.cfg.plain ? 0 : (n % 2 ? cur ^ 1 : cur);
        return cudaSuccess;
    }
    float* tmp = (float*)(c.wsbase + c.w.tmp);
    for (int i = 0; i < n; ++i) {
        const StepConfig cfg = step_at(c.cfg, c.prm, c.P.L, true, k0 + i);
        if (cfg.plain) {
            cudaError_t e = potts_step(c.storage, c.P, c.user, c.user, cfg, tmp, st);
            if (e != cudaSuccess) return e;
            cur = 0;
        } else if (c.dr_rows) {
            cudaError_t e = row_maps(c, cur);
            if (e == cudaSuccess)
                e = potts_dr_rows_step(c.storage, c.P, cur == 0 ? c.ws : c.user, cfg.aniso,
                                       cfg.dc, c.rmaps[cur], c.err, st);
            if (e != cudaSuccess) return e;
            cur ^= 1;
        } else if (c.strip && cfg.dr) {
            const PottsStateV& a = cur == 0 ? c.user : c.ws;
            const PottsStateV& b = cur == 0 ? c.ws : c.user;
            // sum_i u_i planes: the call's first launch sums u itself, later
            // ones read what the previous launch wrote
            float* U = (float*)(c.wsbase + c.w.usum);
            const size_t up = align_up((size_t)c.P.g.H * (size_t)c.P.g.pitch * 4) / 4;
            cudaError_t e = potts_dr_strip_step(c.storage, c.P, a, b, cfg.aniso, cfg.dc,
                                                i == 0 ? nullptr : U + cur * up,
                                                U + (cur ^ 1) * up, st);
            if (e != cudaSuccess) return e;
            cur ^= 1;
        } else if (c.strip) {
            const PottsStateV& a = cur == 0 ? c.user : c.ws;
            const PottsStateV& b = cur == 0 ? c.ws : c.user;
            // the first iteration reads u itself, later ones the w form (cu
            // does not depend on rho, so a schedule keeps it fixed)
            cudaError_t e = potts_strip_step(c.storage, c.P, a, b, cfg.aniso, cfg.ac,
                                             i == 0 ? 0.0f : cfg.ac.cu, st);
            if (e != cudaSuccess) return e;
            cur ^= 1;
            if (i == n - 1 &&
                (e = potts_strip_finalize(c.storage, c.P, b, cfg.ac.cu, st)) != cudaSuccess)
                return e;
        } else if (c.tma) {
            const PottsStateV& b = cur == 0 ? c.ws : c.user;
            cudaError_t e = cudaSuccess;
            if (!(c.tma_mapped >> cur & 1)) {
                e = potts_tma_maps(c.P.g, c.P.L, c.storage, cur == 0 ? c.user : c.ws, c.tma_rows,
                                   c.maps[cur]);
                if (e != cudaSuccess) return e;
                c.tma_mapped |= 1 << cur;
            }
            e = potts_admm_tma_step(c.storage, c.P, b, cfg.aniso, cfg.ac, c.maps[cur], c.err, st);
            if (e != cudaSuccess) return e;
            cur ^= 1;
        } else {
            const PottsStateV& a = cur == 0 ? c.user : c.ws;
            const PottsStateV& b = cur == 0 ? c.ws : c.user;
            cudaError_t e = potts_step(c.storage, c.P, a, b, cfg, tmp, st);
            if (e != cudaSuccess) return e;
            cur ^= 1;
        }
    }
    return cert ? potts_certify(c, cur, st, *cert) : cudaSuccess;
}

cmf_status potts_eval_state(const PottsCall& c, double* h_out, cudaStream_t st) {
    const EvalTail T = reduce_tail(c.wsbase, c.w);
    CMF_CUDA_TRY(cudaMemsetAsync(&T.ctl->arrive, 0, sizeof(unsigned), st));
    CMF_CUDA_TRY(potts_certify(c, 0, st, T));
    return finish_eval(c.wsbase, c.w, h_out, st);
}

// ---- device-driven solve loop (CUDA graph with a conditional WHILE node) ----

__global__ void k_solve_reset(SolveCtl* ctl, int it0) {
    ctl->it = it0;
    ctl->checks = 0;
    ctl->stop = 0;
    ctl->where = 0;
    ctl->arrive = 0;
    ctl->err = 0;  // an earlier phase's error was reported with its last certificates
}

// End of a two-chunk loop body: go on unless either half stopped.
__global__ void k_solve_loop_cond(const SolveCtl* ctl, cudaGraphConditionalHandle h) {
    cudaGraphSetConditional(h, ctl->stop == 0 ? 1u : 0u);
}

size_t hist_rows_for(const cmf_params& p) {
    const size_t r = (size_t)(p.max_iter / (p.check_every > 0 ? p.check_every : 1)) + 1;
    return r < 65536 ? r : 65536;  // later checks are decided but not recorded
}

// Whether the graph path can reproduce the host loop exactly: whole chunks
// only.  (A chunk that ends in the workspace buffers makes the loop body two
// chunks long, see solve_graph.)
bool graph_eligible(const cmf_params& p) {
    if (!p.use_graph || p.max_iter < p.check_every) return false;
    if (p.max_iter % p.check_every != 0) return false;
    return true;
}

// The error word at the start of a solve: the loop's reset kernel clears it,
// unless iterations run host-driven before it.
cudaError_t clear_error(const cmf_params& p, int* err, cudaStream_t st) {
    if (graph_eligible(p) && p.rho_schedule_len == 0) return cudaSuccess;
    return cudaMemsetAsync(err, 0, sizeof(int), st);
}

// Everything the kernels of a solve graph are built from: the device, the
// model, sizes, every device pointer, alpha0 and the parameters (their
// coefficients, the loop constants).  Calls with equal signatures can replay
// the same instantiated graph.  Zero-filled before use (padding included) and
// filled field by field, then compared bytewise.
struct SolveSig {
    int dev, model, L, H, W, pitch;
    float alpha0;
    const void* ptr[10];
    cmf_params p;  // rho schedule and warm start cleared: the graph does not depend on them
};

SolveSig make_sig(int model, int L, int H, int W, int pitch, float alpha0,
                  std::initializer_list<const void*> ptrs, const cmf_params& p) {
    SolveSig k;
    memset(&k, 0, sizeof(k));
    cudaGetDevice(&k.dev);
    k.model = model;
    k.L = L;
    k.H = H;
    k.W = W;
    k.pitch = pitch;
    k.alpha0 = alpha0;
    int i = 0;
    for (const void* q : ptrs)
        if (i < 10) k.ptr[i++] = q;
    // field by field: the caller's padding bytes (after `costs`, at the tail)
    // stay zero, so equal parameters always compare equal
    k.p.algo = p.algo;
    k.p.storage = p.storage;
    k.p.impl = p.impl;
    k.p.aniso = p.aniso;
    k.p.sweeps = p.sweeps;
    k.p.max_iter = p.max_iter;
    k.p.check_every = p.check_every;
    k.p.use_graph = p.use_graph;
    k.p.variant = p.variant;
    k.p.c = p.c;
    k.p.a = p.a;
    k.p.a1 = p.a1;
    k.p.a2 = p.a2;
    k.p.rho = p.rho;
    k.p.r = p.r;
    k.p.sigma = p.sigma;
    k.p.tau = p.tau;
    k.p.tol_gap = p.tol_gap;
    k.p.costs = p.costs;
    k.p.phase_storage = p.phase_storage;
    k.p.phase_gap = p.phase_gap;
    k.p.tune_step = p.tune_step;
    return k;
}

// Instantiated solve graphs, least recently used out.  Graph objects stay
// alive between calls (until evicted or cmf_release_graphs); an executable
// graph that is destroyed while in flight is freed when it completes.
constexpr size_t kGraphCache = 8;
struct GraphEntry {
    SolveSig sig;
    cudaGraph_t g;
    cudaGraphExec_t ge;
    unsigned long long used;
};
std::mutex g_graph_mu;
std::vector<GraphEntry>* g_graphs = new std::vector<GraphEntry>();  // never freed: no
                                                                     // CUDA calls at exit
unsigned long long g_graph_tick = 0;

cudaGraphExec_t graph_lookup(const SolveSig& k) {
    for (GraphEntry& e : *g_graphs)
        if (memcmp(&e.sig, &k, sizeof(k)) == 0) {
            e.used = ++g_graph_tick;
            return e.ge;
        }
    return nullptr;
}

void graph_insert(const SolveSig& k, cudaGraph_t g, cudaGraphExec_t ge) {
    if (g_graphs->size() >= kGraphCache) {
        size_t lru = 0;
        for (size_t i = 1; i < g_graphs->size(); ++i)
            if ((*g_graphs)[i].used < (*g_graphs)[lru].used) lru = i;
        cudaGraphExecDestroy((*g_graphs)[lru].ge);
        cudaGraphDestroy((*g_graphs)[lru].g);
        g_graphs->erase(g_graphs->begin() + lru);
    }
    g_graphs->push_back(GraphEntry{k, g, ge, ++g_graph_tick});
}

void graph_drop(cudaGraphExec_t ge) {
    for (size_t i = 0; i < g_graphs->size(); ++i)
        if ((*g_graphs)[i].ge == ge) {
            cudaGraphExecDestroy(ge);
            cudaGraphDestroy((*g_graphs)[i].g);
            g_graphs->erase(g_graphs->begin() + i);
            return;
        }
}

// The stall test of a two-phase solve's first phase (solve_decide): off when
// iters == 0; the window is the checks that cover `iters` iterations.
struct StallRule {
    int iters = 0;
    double factor = 0.0, near = 0.0;
    int checks(int check_every) const {
        return iters > 0 ? (iters + check_every - 1) / check_every : 0;
    }
};

// `chunk(stream, from)` launches check_every iterations starting in buffer
// set `from` (0 = the caller's, 1 = the workspace's) and returns the set they
// end in through `to`; `certify(stream, set)` launches the certificate kernel
// for a set into the partials.  A chunk that ends in the caller's buffers
// makes the loop body {chunk, certificates, decide}; one that ends in the
// workspace makes it two chunks, the second under a conditional IF node that
// the first half's decision sets, and a last kernel that sets the loop's
// condition (so a solve can stop after either half; `copy_back` then brings
// the state home).  The loop continues a solve that has already run it0
// iterations and recorded nh0 history rows on the host.  The graph is built
// and instantiated on the first call with signature `sig` and replayed after.
template <typename Chunk, typename EndOf, typename Copy>
cmf_status solve_graph(const cmf_params* p, const SolveSig& sig, char* wsbase, const WsLayout& w,
                       Chunk chunk, EndOf end_of, Copy copy_back, double* h_hist,
                       int hist_cap, int* h_iters, cudaStream_t st, int it0 = 0, int nh0 = 0,
                       const StallRule& sr = StallRule()) {
    SolveCtl* ctl = (SolveCtl*)(wsbase + w.ctl);
    double* dhist = (double*)(wsbase + w.hist);
    const int rows = (int)hist_rows_for(*p);
    // the certificate launch reduces its partials and takes the stop decision
    // in its last block: one node per check
    EvalTail T = reduce_tail(wsbase, w);
    T.decide = true;
    T.hist = dhist;
    T.hist_rows = rows;
    T.K = p->check_every;
    T.max_iter = p->max_iter;
    T.tol = p->tol_gap;
    T.stall = sr.checks(p->check_every);
    T.stall_f = sr.factor;
    T.stall_near = sr.near;
    k_solve_reset<<<1, 1, 0, st>>>(ctl, it0);
    CMF_CUDA_TRY(cudaGetLastError());

    std::lock_guard<std::mutex> lock(g_graph_mu);
    cudaGraphExec_t ge = graph_lookup(sig);
    if (!ge) {
        cudaStream_t cs = nullptr, cs2 = nullptr;
        cudaGraph_t g = nullptr;
        bool ok = false;
        do {
            if (cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking) != cudaSuccess) break;
            if (cudaStreamCreateWithFlags(&cs2, cudaStreamNonBlocking) != cudaSuccess) break;
            if (cudaGraphCreate(&g, 0) != cudaSuccess) break;
            cudaGraphConditionalHandle h;
            if (cudaGraphConditionalHandleCreate(&h, g, 1, cudaGraphCondAssignDefault) !=
                cudaSuccess)
                break;
            cudaGraphNodeParams np = {};
            np.type = cudaGraphNodeTypeConditional;
            np.conditional.handle = h;
            np.conditional.type = cudaGraphCondTypeWhile;
            np.conditional.size = 1;
            cudaGraphNode_t node;
            if (cudaGraphAddNode(&node, g, nullptr, nullptr, 0, &np) != cudaSuccess) break;
            cudaGraph_t body = np.conditional.phGraph_out[0];
            if (cudaStreamBeginCaptureToGraph(cs, body, nullptr, nullptr, 0,
                                              cudaStreamCaptureModeRelaxed) != cudaSuccess)
                break;
            // the set a chunk from the caller's buffers ends in decides the body
            const int mid = end_of(0);
            // the IF node's handle, only when there is a second half (a handle
            // without its node fails the instantiation)
            cudaError_t e = cudaSuccess;
            cudaGraphConditionalHandle h_if = 0;
            if (mid) e = cudaGraphConditionalHandleCreate(&h_if, body, 0, cudaGraphCondAssignDefault);
            if (e == cudaSuccess) {
                EvalTail T1 = T;
                T1.h = mid ? h_if : h;
                T1.set_h = mid ? 2 : 1;
                T1.where = mid;
                int got = 0;
                e = chunk(cs, 0, got, T1);  // iterations and their certificates
                if (e == cudaSuccess && got != mid) e = cudaErrorInvalidValue;
            }
            if (e == cudaSuccess && mid) {
                // second half: an IF node on the first half's decision
                cudaStreamCaptureStatus cst;
                const cudaGraphNode_t* deps = nullptr;
                const cudaGraphEdgeData* edges = nullptr;
                size_t ndeps = 0;
                cudaGraph_t cg = nullptr;
                e = cudaStreamGetCaptureInfo(cs, &cst, nullptr, &cg, &deps, &edges, &ndeps);
                cudaGraphNodeParams ip = {};
                ip.type = cudaGraphNodeTypeConditional;
                ip.conditional.handle = h_if;
                ip.conditional.type = cudaGraphCondTypeIf;
                ip.conditional.size = 1;
                cudaGraphNode_t ifnode;
                if (e == cudaSuccess)
                    e = cudaGraphAddNode(&ifnode, body, deps, edges, ndeps, &ip);
                if (e == cudaSuccess)
                    e = cudaStreamUpdateCaptureDependencies(cs, &ifnode, nullptr, 1,
                                                            cudaStreamSetCaptureDependencies);
                if (e == cudaSuccess)
                    e = cudaStreamBeginCaptureToGraph(cs2, ip.conditional.phGraph_out[0],
                                                      nullptr, nullptr, 0,
                                                      cudaStreamCaptureModeRelaxed);
                if (e == cudaSuccess) {
                    int end = mid;
                    EvalTail T2 = T;  // conditions left to k_solve_loop_cond
                    cudaError_t f = chunk(cs2, mid, end, T2);
                    if (f == cudaSuccess && end != 0) f = cudaErrorInvalidValue;
                    cudaGraph_t cap2 = nullptr;
                    cudaError_t f2 = cudaStreamEndCapture(cs2, &cap2);
                    e = f != cudaSuccess ? f : f2;
                }
                if (e == cudaSuccess) {
                    k_solve_loop_cond<<<1, 1, 0, cs>>>(ctl, h);
                    e = cudaGetLastError();
                }
            }
            cudaGraph_t captured = nullptr;
            cudaError_t e4 = cudaStreamEndCapture(cs, &captured);
            if (e != cudaSuccess || e4 != cudaSuccess) break;
            if (cudaGraphInstantiate(&ge, g, 0) != cudaSuccess) break;
            ok = true;
        } while (0);
        if (cs2) cudaStreamDestroy(cs2);
        if (cs) cudaStreamDestroy(cs);
        if (!ok) {
            if (ge) cudaGraphExecDestroy(ge);
            if (g) cudaGraphDestroy(g);
            return CMF_ECUDA;
        }
        graph_insert(sig, g, ge);
    }
    if (cudaGraphLaunch(ge, st) != cudaSuccess) {
        graph_drop(ge);
        return CMF_ECUDA;
    }
    // The control block and the first history rows follow one another in the
    // workspace: one copy brings both home (a copy and its synchronisation cost
    // about 10 us, a 64^2 solve 150), a second one only rows beyond them.
    const int room = hist_cap > nh0 ? hist_cap - nh0 : 0;
    const int want = h_hist ? (rows < room ? rows : room) : 0;
    constexpr int kFirstRows = 96;
    const int head = want < kFirstRows ? want : kFirstRows;
    const size_t row_bytes = 5 * sizeof(double), hist_at = w.hist - w.ctl;
    double buf[(256 + kFirstRows * 5 * sizeof(double)) / sizeof(double)];
    static_assert(sizeof(SolveCtl) <= 256, "the history follows the control block's 256 bytes");
    CMF_CUDA_TRY(cudaMemcpyAsync(buf, ctl, head > 0 ? hist_at + head * row_bytes : sizeof(SolveCtl),
                                 cudaMemcpyDeviceToHost, st));
    CMF_CUDA_TRY(cudaStreamSynchronize(st));
    SolveCtl hc;
    memcpy(&hc, buf, sizeof(hc));
    const int n = hc.checks < want ? hc.checks : want;
    if (n > 0)
        memcpy(h_hist + 5 * (size_t)nh0, (const char*)buf + hist_at,
               (n < head ? n : head) * row_bytes);
    if (n > head)
        CMF_CUDA_TRY(cudaMemcpy(h_hist + 5 * (size_t)(nh0 + head), dhist + 5 * (size_t)head,
                                (n - head) * row_bytes, cudaMemcpyDeviceToHost));
    if (h_iters) *h_iters = hc.it;
    if (hc.where != 0) {  // stopped after the first half of a two-chunk body
        CMF_CUDA_TRY(copy_back(hc.where));
        CMF_CUDA_TRY(cudaStreamSynchronize(st));
    }
    return hc.stop == 1 ? CMF_OK : (hc.stop == 3 ? CMF_ETIMEOUT : CMF_NOT_CONVERGED);
}

// Progress of a host-driven solve loop.
struct LoopState {
    int it = 0;    // iterations done
    int nh = 0;    // certificate checks done
    int cur = 0;   // buffer set holding the state (0 = caller's)
    bool converged = false;
};

// Host-driven chunks of check_every iterations, each with the certificates
// of its result, until convergence, max_iter, or it >= it_stop.
// `run_cert(n, cur, k0, out)` advances n iterations whose first is iteration
// k0 of the solve and writes the certificates (E, D, gap, res) to out.
template <typename RunCert>
cmf_status loop_chunks(const cmf_params* p, int it_stop, RunCert run_cert, double* h_hist,
                       int hist_cap, LoopState& ls, const StallRule& sr = StallRule()) {
    double out[4];
    const int stall = sr.checks(p->check_every);
    double gref = 0.0;  // the stall test, as solve_decide keeps it
    int nchk = 0;
    while (ls.it < p->max_iter && ls.it < it_stop) {
        const int k =
            p->check_every < p->max_iter - ls.it ? p->check_every : p->max_iter - ls.it;
        cmf_status s = run_cert(k, ls.cur, ls.it, out);
        if (s != CMF_OK) return s;
        ls.it += k;
        if (h_hist && ls.nh < hist_cap) {
            double* row = h_hist + 5 * (size_t)ls.nh;
            row[0] = ls.it;
            row[1] = out[0];
            row[2] = out[1];
            row[3] = out[2];
            row[4] = out[3];
        }
        ++ls.nh;
        bool stalled = false;
        if (stall > 0 && nchk % stall == 0) {
            stalled = nchk > 0 && out[2] < sr.near && out[2] > sr.factor * gref;
            gref = out[2];
        }
        ++nchk;
        if (out[2] <= p->tol_gap || stalled) {
            ls.converged = true;
            break;
        }
    }
    return CMF_OK;
}

template <typename Copy>
cmf_status finish_loop(const LoopState& ls, Copy copy_back, int* h_iters, cudaStream_t st) {
    if (ls.cur != 0) CMF_CUDA_TRY(copy_back(ls.cur));
    CMF_CUDA_TRY(cudaStreamSynchronize(st));
    if (h_iters) *h_iters = ls.it;
    return ls.converged ? CMF_OK : CMF_NOT_CONVERGED;
}

// The solve driver: the iterations a rho schedule covers run host-driven
// (their coefficients change from launch to launch, a graph's are fixed), the
// rest in the device-driven graph where it applies, else host-driven.
// `chunk(stream, from, to, tail)` captures one graph chunk with its
// certificates, `end_of(from)` tells the set a chunk ends in.
// it0, nh0: iterations and history rows an earlier phase of the same solve
// has already done (the loop continues their count; max_iter is the total).
template <typename RunCert, typename Copy, typename Chunk, typename EndOf>
cmf_status solve_driver(const cmf_params* p, const SolveSig& sig, char* wsbase, const WsLayout& w,
                        RunCert run_cert, Copy copy_back, Chunk chunk, EndOf end_of,
                        double* h_hist, int hist_cap, int* h_iters, cudaStream_t st,
                        int it0 = 0, int nh0 = 0, const StallRule& sr = StallRule()) {
    LoopState ls;
    ls.it = it0;
    ls.nh = nh0;
    if (!graph_eligible(*p)) {
        cmf_status s = loop_chunks(p, p->max_iter, run_cert, h_hist, hist_cap, ls, sr);
        if (s != CMF_OK) return s;
        return finish_loop(ls, copy_back, h_iters, st);
    }
    if (p->rho_schedule_len > 0) {
        cmf_status s = loop_chunks(p, p->rho_schedule_len, run_cert, h_hist, hist_cap, ls);
        if (s != CMF_OK) return s;
        if (ls.cur != 0) CMF_CUDA_TRY(copy_back(ls.cur));  // the graph starts from set 0
        ls.cur = 0;
        if (ls.converged || ls.it >= p->max_iter) return finish_loop(ls, copy_back, h_iters, st);
    }
    return solve_graph(p, sig, wsbase, w, chunk, end_of, copy_back, h_hist, hist_cap,
                       h_iters, st, ls.it, ls.nh, sr);
}

}  // namespace

// ===========================================================================
// Public entry points
// ===========================================================================
extern "C" {

cmf_status cmf_default_params(int algo, int L, cmf_params* p) {
    if (!p || algo < CMF_PADMM || algo > CMF_CP || L < 2) return CMF_EINVAL;
    memset(p, 0, sizeof(*p));
    p->algo = algo;
    p->storage = CMF_F32;
    p->impl = CMF_FUSED;
    p->aniso = 0;
    p->sweeps = 1;
    p->max_iter = 10000;
    p->check_every = 10;
    p->warm_start = 0;
    p->use_graph = 1;
    p->c = 0.3;
    p->a = 8.0;
    p->a1 = 2.0;
    p->a2 = 2.0 * L;
    p->rho = 1.9;
    p->r = 1.618;
    p->sigma = L == 2 ? 0.2 : 5.0;
    p->tau = L == 2 ? 1.0 : 0.4;
    if (algo == CMF_CP) {  // ALG1 (Sec. 4): sigma = 0.4, tau = 1 / (||K*K|| bound x sigma)
        p->sigma = 0.4;
        p->tau = 1.0 / ((L == 2 ? 10.0 : 9.0 + L) * 0.4);
    }
    p->tol_gap = 1e-4;
    return CMF_OK;
}

const char* cmf_status_str(cmf_status s) {
    switch (s) {
        case CMF_OK: return "ok";
        case CMF_EINVAL: return "invalid argument";
        case CMF_ENOMEM: return "workspace too small";
        case CMF_ECUDA: return "CUDA error";
        case CMF_ETIMEOUT: return "device wait timed out";
        case CMF_NOT_CONVERGED: return "not converged (max_iter reached)";
    }
    return "unknown status";
}

size_t cmf_workspace_bytes(int H, int W, int L, int pitch, const cmf_params* p) {
    if (!p || check_grid(H, W, pitch) != CMF_OK || L < 2 || L > 64) return 0;
    const size_t potts = ws_layout(H, W, L, pitch, *p, true).total;
    if (L > 2) return potts;
    const size_t binary = ws_layout(H, W, 2, pitch, *p, false).total;
    return binary > potts ? binary : potts;  // L = 2 serves both models
}

cmf_status cmf_init_binary(const float* d_Cs, const float* d_Ct, int H, int W, int pitch,
                           const cmf_params* p, float* d_u, void* d_qx, void* d_qy, void* d_ps,
                           void* d_pt, void* stream) {
    cmf_status s;
    if ((s = check_params(p, 2)) != CMF_OK) return s;
    if ((s = check_grid(H, W, pitch)) != CMF_OK) return s;
    if (!d_Cs || !d_Ct || !d_u || !d_qx || !d_qy || !d_ps || !d_pt) return CMF_EINVAL;
    BinProblem P{d_Cs, d_Ct, make_alpha(nullptr, 0.f), make_grid(H, W, pitch)};
    BinStateV st{d_u, d_qx, d_qy, d_ps, d_pt};
    CMF_CUDA_TRY(binary_init(p->storage, P, st, p->algo == CMF_RPDRQ, (float)p->tau,
                             (cudaStream_t)stream));
    return CMF_OK;
}

cmf_status cmf_iterate_binary(const float* d_Cs, const float* d_Ct, const float* d_alpha,
                              float alpha0, int H, int W, int pitch, const cmf_params* p,
                              int n_iter, float* d_u, void* d_qx, void* d_qy, void* d_ps,
                              void* d_pt, void* d_ws, size_t ws_bytes, void* stream) {
    BinaryCall c;
    cmf_status s = binary_prepare(d_Cs, d_Ct, d_alpha, alpha0, H, W, pitch, p, d_u, d_qx, d_qy,
                                  d_ps, d_pt, d_ws, ws_bytes, c);
    if (s != CMF_OK) return s;
    if (n_iter < 0) return CMF_EINVAL;
    cudaStream_t st = (cudaStream_t)stream;
    CMF_CUDA_TRY(cudaMemsetAsync(&((SolveCtl*)(c.wsbase + c.w.ctl))->err, 0, sizeof(int), st));
    int cur = 0;
    CMF_CUDA_TRY(binary_run(c, n_iter, cur, st));
    if (cur != 0) CMF_CUDA_TRY(copy_binary(c.user, bset(c, cur), c.P.g, c.storage, st));
    return CMF_OK;
}

cmf_status cmf_eval_binary(const float* d_Cs, const float* d_Ct, const float* d_alpha,
                           float alpha0, int H, int W, int pitch, const cmf_params* p,
                           const float* d_u, const void* d_qx, const void* d_qy,
                           const void* d_ps, const void* d_pt, double* h_out, void* d_ws,
                           size_t ws_bytes, void* stream) {
    if (!h_out) return CMF_EINVAL;
    BinaryCall c;
    cmf_status s = binary_prepare(d_Cs, d_Ct, d_alpha, alpha0, H, W, pitch, p, (float*)d_u,
                                  (void*)d_qx, (void*)d_qy, (void*)d_ps, (void*)d_pt, d_ws,
                                  ws_bytes, c);
    if (s != CMF_OK) return s;
    return binary_eval_state(c, c.user, h_out, (cudaStream_t)stream);
}

cmf_status cmf_solve_binary(const float* d_Cs, const float* d_Ct, const float* d_alpha,
                            float alpha0, int H, int W, int pitch, const cmf_params* p,
                            float* d_u, void* d_qx, void* d_qy, void* d_ps, void* d_pt,
                            double* h_hist, int hist_cap, int* h_iters, void* d_ws,
                            size_t ws_bytes, void* stream) {
    BinaryCall c;
    cmf_status s = binary_prepare(d_Cs, d_Ct, d_alpha, alpha0, H, W, pitch, p, d_u, d_qx, d_qy,
                                  d_ps, d_pt, d_ws, ws_bytes, c);
    if (s != CMF_OK) return s;
    if (hist_cap < 0) return CMF_EINVAL;
    cudaStream_t st = (cudaStream_t)stream;
    CMF_CUDA_TRY(clear_error(*p, c.err, st));
    if (!p->warm_start)
        CMF_CUDA_TRY(binary_init(c.storage, c.P, c.user, c.cfg.dr, c.cfg.dc.tau, st));
    const SolveSig sig = make_sig(0, 2, H, W, pitch, alpha0,
                                  {d_Cs, d_Ct, d_alpha, d_u, d_qx, d_qy, d_ps, d_pt, d_ws},
                                  *p);
    return solve_driver(
        p, sig, c.wsbase, c.w,
        [&](int n, int& cur, int k0, double* out) -> cmf_status {
            const EvalTail T = reduce_tail(c.wsbase, c.w);
            CMF_CUDA_TRY(cudaMemsetAsync(&T.ctl->arrive, 0, sizeof(unsigned), st));
            CMF_CUDA_TRY(binary_run(c, n, cur, st, k0, &T));
            return finish_eval(c.wsbase, c.w, out, st);
        },
        [&](int from) { return copy_binary(c.user, bset(c, from), c.P.g, c.storage, st); },
        [&](cudaStream_t s, int from, int& to, const EvalTail& T) {  // after the schedule
            to = from;
            return binary_run(c, p->check_every, to, s, p->rho_schedule_len, &T);
        },
        [&](int from) {
            int to = from;
            binary_run(c, p->check_every, to, nullptr, p->rho_schedule_len, nullptr, true);
            return to;
        },
        h_hist, hist_cap, h_iters, st);
}

cmf_status cmf_release_graphs(void) {
    std::lock_guard<std::mutex> lock(g_graph_mu);
    for (GraphEntry& e : *g_graphs) {
        cudaGraphExecDestroy(e.ge);
        cudaGraphDestroy(e.g);
    }
    g_graphs->clear();
    return CMF_OK;
}

cmf_status cmf_init_potts(const float* d_C, int L, int H, int W, int pitch, const cmf_params* p,
                          float* d_u, void* d_qx, void* d_qy, void* d_p, void* d_ps,
                          void* stream) {
    cmf_status s;
    if (L < 2 || L > 64) return CMF_EINVAL;
    if ((s = check_params(p, L)) != CMF_OK) return s;
    if ((s = check_grid(H, W, pitch)) != CMF_OK) return s;
    if (!d_C || !d_u || !d_qx || !d_qy || !d_p || !d_ps) return CMF_EINVAL;
    if (!aligned(d_C, p->costs == 2 ? 2 : 4)) return CMF_EINVAL;
    const PottsProblem P = potts_problem(d_C, L, nullptr, 0.f, H, W, pitch, p->costs);
    PottsStateV st{d_u, d_qx, d_qy, d_p, (float*)d_ps};
    CMF_CUDA_TRY(potts_init(p->storage, P, st, p->algo == CMF_RPDRQ, (float)p->tau,
                            (cudaStream_t)stream));
    return CMF_OK;
}

cmf_status cmf_iterate_potts(const float* d_C, int L, const float* d_alpha, float alpha0, int H,
                             int W, int pitch, const cmf_params* p, int n_iter, float* d_u,
                             void* d_qx, void* d_qy, void* d_p, void* d_ps, void* d_ws,
                             size_t ws_bytes, void* stream) {
    PottsCall c;
    cmf_status s = potts_prepare(d_C, L, d_alpha, alpha0, H, W, pitch, p, d_u, d_qx, d_qy, d_p,
                                 d_ps, d_ws, ws_bytes, c);
    if (s != CMF_OK) return s;
    if (n_iter < 0) return CMF_EINVAL;
    cudaStream_t st = (cudaStream_t)stream;
    CMF_CUDA_TRY(cudaMemsetAsync(c.err, 0, sizeof(int), st));
    int cur = 0;
    CMF_CUDA_TRY(potts_run(c, n_iter, cur, st, 0, nullptr, false, true));
    if (cur != 0) CMF_CUDA_TRY(copy_potts(c.user, c.ws, c.P.g, L, c.storage, st));
    return CMF_OK;
}

cmf_status cmf_eval_potts(const float* d_C, int L, const float* d_alpha, float alpha0, int H,
                          int W, int pitch, const cmf_params* p, const float* d_u,
                          const void* d_qx, const void* d_qy, const void* d_p, const void* d_ps,
                          double* h_out, void* d_ws, size_t ws_bytes, void* stream) {
    if (!h_out) return CMF_EINVAL;
    PottsCall c;
    cmf_status s = potts_prepare(d_C, L, d_alpha, alpha0, H, W, pitch, p, (float*)d_u,
                                 (void*)d_qx, (void*)d_qy, (void*)d_p, (void*)d_ps, d_ws,
                                 ws_bytes, c);
    if (s != CMF_OK) return s;
    return potts_eval_state(c, h_out, (cudaStream_t)stream);
}

// The first phase of a two-phase solve also ends when its certified gap,
// below kPhaseStallNear x phase_gap, has not fallen to kPhaseStallFactor
// times its value kPhaseStallIters iterations earlier (tested once per such
// window): the 16-bit storage's rounding floor of this instance is near (it
// rises with the step size c), and float32 storage continues from there.
constexpr int kPhaseStallIters = 200;
constexpr double kPhaseStallFactor = 0.7;
constexpr double kPhaseStallNear = 10.0;

cmf_status cmf_solve_potts(const float* d_C, int L, const float* d_alpha, float alpha0, int H,
                           int W, int pitch, const cmf_params* p, float* d_u, void* d_qx,
                           void* d_qy, void* d_p, void* d_ps, double* h_hist, int hist_cap,
                           int* h_iters, void* d_ws, size_t ws_bytes, void* stream) {
    PottsCall c;
    cmf_status s = potts_prepare(d_C, L, d_alpha, alpha0, H, W, pitch, p, d_u, d_qx, d_qy, d_p,
                                 d_ps, d_ws, ws_bytes, c);
    if (s != CMF_OK) return s;
    if (hist_cap < 0) return CMF_EINVAL;
    cudaStream_t st = (cudaStream_t)stream;
    CMF_CUDA_TRY(clear_error(*p, c.err, st));
    int it0 = 0, nh0 = 0;
    if (p->phase_storage != 0) {
        // phase one: the same solve in 16-bit flow storage, in the
        // workspace's two phase sets, to the switch gap
        cmf_params q = *p;
        q.storage = p->phase_storage;
        q.tol_gap = p->phase_gap;
        q.phase_storage = 0;
        q.phase_gap = 0.0;
        const Grid G = make_grid(H, W, pitch);
        const PottsStateV A = ws_potts_state((char*)d_ws, c.w.phase, G, L, q.storage);
        const PottsStateV B =
            ws_potts_state((char*)d_ws, c.w.phase + c.w.phase_set, G, L, q.storage);
        PottsCall c1;
        s = potts_prepare(d_C, L, d_alpha, alpha0, H, W, pitch, &q, A.u, A.qx, A.qy, A.p, A.ps,
                          d_ws, ws_bytes, c1, p, &B);
        if (s != CMF_OK) return s;
        CMF_CUDA_TRY(potts_init(c1.storage, c1.P, c1.user, c1.cfg.dr, c1.cfg.dc.tau, st));
        const SolveSig sig1 = make_sig(2, L, H, W, pitch, alpha0, {d_C, d_alpha, d_ws}, q);
        int it1 = 0;
        s = solve_driver(
            &q, sig1, c1.wsbase, c1.w,
            [&](int n, int& cur, int k0, double* out) -> cmf_status {
                const EvalTail T = reduce_tail(c1.wsbase, c1.w);
                CMF_CUDA_TRY(cudaMemsetAsync(&T.ctl->arrive, 0, sizeof(unsigned), st));
                CMF_CUDA_TRY(potts_run(c1, n, cur, st, k0, &T));
                return finish_eval(c1.wsbase, c1.w, out, st);
            },
            [&](int) { return copy_potts(c1.user, c1.ws, c1.P.g, L, c1.storage, st); },
            [&](cudaStream_t s2, int from, int& to, const EvalTail& T) {
                to = from;
                return potts_run(c1, q.check_every, to, s2, 0, &T);
            },
            [&](int from) {
                int to = from;
                potts_run(c1, q.check_every, to, nullptr, 0, nullptr, true);
                return to;
            },
            h_hist, hist_cap, &it1, st, 0, 0, StallRule{kPhaseStallIters, kPhaseStallFactor,
                                                        kPhaseStallNear * q.tol_gap});
        if (s != CMF_OK && s != CMF_NOT_CONVERGED) return s;
        // the switch: the 16-bit state written exactly into the caller's
        // float32 buffers; phase two continues from it
        CMF_CUDA_TRY(potts_widen(q.storage, G, L, A, c.user, st));
        it0 = it1;
        nh0 = it1 / p->check_every;
        if (it0 >= p->max_iter) {
            CMF_CUDA_TRY(cudaStreamSynchronize(st));
            if (h_iters) *h_iters = it0;
            return CMF_NOT_CONVERGED;
        }
    } else if (!p->warm_start) {
        CMF_CUDA_TRY(potts_init(c.storage, c.P, c.user, c.cfg.dr, c.cfg.dc.tau, st));
    }
    const SolveSig sig = make_sig(1, L, H, W, pitch, alpha0,
                                  {d_C, d_alpha, d_u, d_qx, d_qy, d_p, d_ps, d_ws}, *p);
    return solve_driver(
        p, sig, c.wsbase, c.w,
        [&](int n, int& cur, int k0, double* out) -> cmf_status {
            const EvalTail T = reduce_tail(c.wsbase, c.w);
            CMF_CUDA_TRY(cudaMemsetAsync(&T.ctl->arrive, 0, sizeof(unsigned), st));
            CMF_CUDA_TRY(potts_run(c, n, cur, st, k0, &T));
            return finish_eval(c.wsbase, c.w, out, st);
        },
        [&](int) { return copy_potts(c.user, c.ws, c.P.g, L, c.storage, st); },
        [&](cudaStream_t s, int from, int& to, const EvalTail& T) {  // after the schedule
            to = from;
            return potts_run(c, p->check_every, to, s, p->rho_schedule_len, &T);
        },
        [&](int from) {
            int to = from;
            potts_run(c, p->check_every, to, nullptr, p->rho_schedule_len, nullptr, true);
            return to;
        },
        h_hist, hist_cap, h_iters, st, it0, nh0);
}

}  // extern "C"

// ===========================================================================
// Autotuner: time to the gap for each candidate launch configuration
// ===========================================================================
namespace {

// Candidate list for a parameter set: kernel variants of the fused ADMM path
// and sRBGS sweep counts of the fused rPDRQ path.  Binary problems run the chains
// of warps under variant 4 at even widths, under variant 0 alone at odd ones.
std::vector<cmf_params> tune_candidates(const cmf_params& p, bool binary, int W) {
    std::vector<cmf_params> out;
    const bool fused = p.impl == CMF_FUSED;
    const bool dr = p.algo == CMF_RPDRQ;
    std::vector<int> variants = {p.variant};
    std::vector<int> sweeps = {p.sweeps};
    if (fused && !dr) variants = binary && W % 2 == 0 ? std::vector<int>{1, 2, 4, 8, 16, 32}
                                                      : std::vector<int>{0, 1, 2, 8, 16, 32};
    if (fused && dr) sweeps = {1, 2, 3};
    for (int v : variants)
        for (int s : sweeps) {
            cmf_params q = p;
            q.variant = v;
            q.sweeps = s;
            q.warm_start = 0;
            out.push_back(q);
        }
    // the ADMM step size (tune_step): larger c with the given variant
    const bool admm = p.algo == CMF_PADMM || p.algo == CMF_RPADMM_FG ||
                      p.algo == CMF_RPADMM_EB || p.algo == CMF_TY;
    if (p.tune_step == 1 && admm)
        for (double f : {2.0, 4.0, 8.0}) {
            cmf_params q = p;
            q.c = p.c * f;
            q.warm_start = 0;
            out.push_back(q);
        }
    // two-phase solves (tune_step): each step size also with the switch left
    // to the first phase's stall test alone (phase_gap 1.5 tol_gap)
    const double stall_only = 1.5 * p.tol_gap;
    if (p.tune_step == 1 && admm && p.phase_storage != 0 && stall_only < p.phase_gap)
        for (double f : {1.0, 2.0, 4.0, 8.0}) {
            cmf_params q = p;
            q.c = p.c * f;
            q.phase_gap = stall_only;
            q.warm_start = 0;
            out.push_back(q);
        }
    return out;
}

template <typename Solve>
cmf_status tune_loop(const cmf_params* p, bool binary, int W, Solve solve, cmf_params* best,
                     double* h_best_ms, cudaStream_t st) {
    if (!p || !best) return CMF_EINVAL;
    cudaEvent_t e0, e1;
    CMF_CUDA_TRY(cudaEventCreate(&e0));
    CMF_CUDA_TRY(cudaEventCreate(&e1));
    double best_ms = 1e300;
    bool found = false;
    cmf_status last = CMF_EINVAL;
    for (const cmf_params& q : tune_candidates(*p, binary, W)) {
        cmf_status s = solve(q);  // warm-up (and validity check)
        last = s;
        if (s != CMF_OK) continue;
        double ms_min = 1e300;
        for (int rep = 0; rep < 2; ++rep) {
            cudaEventRecord(e0, st);
            s = solve(q);
            cudaEventRecord(e1, st);
            cudaEventSynchronize(e1);
            float ms = 0.f;
            cudaEventElapsedTime(&ms, e0, e1);
            if (s == CMF_OK && ms < ms_min) ms_min = ms;
        }
        if (ms_min < best_ms) {
            best_ms = ms_min;
            *best = q;
            found = true;
        }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (!found) return last == CMF_OK ? CMF_NOT_CONVERGED : last;
    if (h_best_ms) *h_best_ms = best_ms;
    return CMF_OK;
}

}  // namespace

extern "C" cmf_status cmf_autotune_binary(const float* d_Cs, const float* d_Ct,
                                          const float* d_alpha, float alpha0, int H, int W,
                                          int pitch, const cmf_params* p, float* d_u,
                                          void* d_qx, void* d_qy, void* d_ps, void* d_pt,
                                          void* d_ws, size_t ws_bytes, cmf_params* best,
                                          double* h_best_ms, void* stream) {
    return tune_loop(
        p, true, W,
        [&](const cmf_params& q) {
            return cmf_solve_binary(d_Cs, d_Ct, d_alpha, alpha0, H, W, pitch, &q, d_u, d_qx,
                                    d_qy, d_ps, d_pt, nullptr, 0, nullptr, d_ws, ws_bytes,
                                    stream);
        },
        best, h_best_ms, (cudaStream_t)stream);
}

extern "C" cmf_status cmf_autotune_potts(const float* d_C, int L, const float* d_alpha,
                                         float alpha0, int H, int W, int pitch,
                                         const cmf_params* p, float* d_u, void* d_qx,
                                         void* d_qy, void* d_p, void* d_ps, void* d_ws,
                                         size_t ws_bytes, cmf_params* best, double* h_best_ms,
                                         void* stream) {
    return tune_loop(
        p, false, W,
        [&](const cmf_params& q) {
            return cmf_solve_potts(d_C, L, d_alpha, alpha0, H, W, pitch, &q, d_u, d_qx, d_qy,
                                   d_p, d_ps, nullptr, 0, nullptr, d_ws, ws_bytes, stream);
        },
        best, h_best_ms, (cudaStream_t)stream);
}
