// Potts certificates with the labels side by side (Eq. relaxed-potts, Eq.
// potts-mf): primal energy at the simplex projection of u, dual value of the
// re-projected flows, squared conservation residual.
//
// Work unit: one block, a strip of 64 columns (two adjacent columns per lane,
// 60 owned) and a band of rows, streamed top-down.  Warp l < L sums label l's
// terms of the energy and the residual and puts C_l + div P_alpha(y_l) of each
// pixel into shared memory; theta warps (one per four labels, rows in turn)
// find the simplex thresholds of the coming rows from the u rows in shared
// memory; the last warp keeps the next rows of every plane in flight with TMA
// (elements outside the grid read as zero) and sums the minima over the
// labels.  mbarriers couple them: full (a row has arrived), TH (its thresholds
// are there), SF (every label is done with a step).  Step k handles row
// rf + k; a label reads row k + 1 of the state, row k's costs, p_s and alpha.
//   - row k + kRing is issued when every label has done step k: its state slot
//     was read in step k - 1, its cost slot in step k, and its threshold slot
//     with the state (row 0's before the first step, see cmf_rows_order.cuh);
//   - a candidate slot is rewritten kRing steps on, after its writer has had a
//     row that was issued after the sum over that slot.
//
// What bounds it.  The strip kernel walked the labels one after another,
// re-read u for the thresholds and p_s and alpha per label, and issued 180-220
// thread instructions per label-pixel at 60% of the issue slots (583 us at
// 2048^2, L = 16, float16; odd widths: tiles).  Here each plane is read once
// (1.40 GB of DRAM reads for 1.38 GB) and the thresholds come from shared
// memory: 137 thread instructions per label-pixel (two correctly rounded
// square roots, two projections and two double-float sums per pair are most of
// them), 61% of the issue slots, DRAM at 45%.  Measured at 2048^2, float32: L = 16
// 390 us (ncu), a call 619 -> 434 us; L = 4 a call 195 -> 158 us.
#pragma once

#include "cmf_potts_rows.cuh"

namespace cmf {
namespace cert {

template <int LC, int ES>
struct Layout {
    static constexpr int fs = rows::up128(LC * rows::Seg<ES>::cols * ES);
    static constexpr int f4 = rows::up128(LC * rows::Seg<4>::cols * 4);
    static constexpr int f1 = rows::up128(rows::Seg<4>::cols * 4);
    static constexpr int state = 3 * fs + f4;  // q_x, q_y, p, u
    static constexpr int aux = f4 + 2 * f1;    // C, p_s, alpha
    static constexpr int sh = LC * 256;        // candidates of a row
    static constexpr int o_aux = kRing * state;
    static constexpr int o_sh = o_aux + kRing * aux;
    static constexpr int o_th = o_sh + kRing * sh;
    static constexpr int o_us = o_th + kRing * 256;
    static constexpr int o_bar = o_us + kRing * 256;
    static constexpr int bytes = o_bar + 3 * 8 * kRing + 128;
};

}  // namespace cert

template <typename S, bool ANISO, bool DR, int LC>
__global__ void __launch_bounds__(32 * (LC + cert::theta_warps(LC) + 1),
                                  LC == 4 ? 3 : (LC == 8 ? 2 : 1))
    k_potts_cert(const __grid_constant__ PottsRowsMaps M, PottsProblem P, float tau, int R,
                 int nstrips, double* partials, EvalTail tail, int* err) {
    using namespace rows;
    using cert::kRing;
    using PS = Pair<S>;
    constexpr int ES = sizeof(S), NT = cert::theta_warps(LC);
    using Y = cert::Layout<LC, ES>;
    extern __shared__ __align__(128) unsigned char dsm_raw[];
    const Grid G = P.g;
    const int L = P.L;
    unsigned char* const dsm = dsm_raw + ((128u - (smem_u32(dsm_raw) & 127u)) & 127u);
    uint64_t* const bar = reinterpret_cast<uint64_t*>(dsm + Y::o_bar);
    const uint32_t b_full = smem_u32(bar), b_th = b_full + 8 * kRing, b_sf = b_th + 8 * kRing;
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const unsigned full_mask = 0xffffffffu;

    const int r0 = (blockIdx.x / nstrips) * R;
    const int r1 = min(r0 + R, G.H);
    const int cfirst = (int)(blockIdx.x % nstrips) * 60 - 2;
    const int c = cfirst + 2 * lane;
    const bool own = lane >= 1 && lane <= 30 && c < G.W;
    const bool pair = c + 1 < G.W;  // else the last column of an odd width alone
    const int off4 = cfirst & (Seg<4>::align - 1), offs = cfirst & (Seg<ES>::align - 1);
    const int rf = r0 - 1, ke = r1 - 1 - rf, il = r1 - rf;  // last step, last row

    if (threadIdx.x == 0) {
        for (int i = 0; i < kRing; ++i) {
            mbar_init(bar + i, 1);
            mbar_init(bar + kRing + i, 1);
            mbar_init(bar + 2 * kRing + i, L);
        }
        fence_mbar_init();
    }
    const bool has_al = P.alpha.plane != nullptr;
    if (!has_al)  // constant alpha: every row's slot holds it
        for (int i = threadIdx.x; i < kRing * Seg<4>::cols; i += blockDim.x) {
            const int r = i / Seg<4>::cols;
            reinterpret_cast<float*>(dsm + Y::o_aux + r * Y::aux + Y::f4 +
                                     Y::f1)[i - r * Seg<4>::cols] = P.alpha.value;
        }
    __syncthreads();
    bool ok = true;
    DF accE = {0.f, 0.f}, accD = {0.f, 0.f}, accR = {0.f, 0.f};
    auto slot = [](int i) { return i & (kRing - 1); };
    auto phase = [](int i) { return (uint32_t)(i / kRing) & 1u; };
    auto f2 = [](const unsigned char* q) { return *reinterpret_cast<const float2*>(q); };

    if (wib < L) {
        // ---- label warps ---------------------------------------------------
        const float mxe = (c >= 0 && c < G.W - 1) ? 1.f : 0.f;
        const float mxo = (c + 1 >= 0 && c + 1 < G.W - 1) ? 1.f : 0.f;
        const unsigned char* const st_s = dsm + wib * Seg<ES>::cols * ES + ES * (offs + 2 * lane);
        const unsigned char* const st_u =
            dsm + 3 * Y::fs + wib * Seg<4>::cols * 4 + 4 * (off4 + 2 * lane);
        const unsigned char* const ax = dsm + Y::o_aux + 4 * (off4 + 2 * lane);
        const unsigned char* const axc = ax + wib * Seg<4>::cols * 4;
        const unsigned char* const th = dsm + Y::o_th + lane * 8;
        const unsigned char* const us = dsm + Y::o_us + lane * 8;
        unsigned char* const sh = dsm + Y::o_sh + wib * 256 + lane * 8;
        auto sp = [](const unsigned char* q) {
            return *reinterpret_cast<const typename PS::T*>(q);
        };
        auto load_row = [&](int i, Row<S>& x) {
            const unsigned char* q = st_s + slot(i) * Y::state;
            x.qx = sp(q);
            x.qy = sp(q + Y::fs);
            x.p = sp(q + 2 * Y::fs);
            x.u = f2(st_u + slot(i) * Y::state);
        };
        auto left_of = [&](float v) { return __shfl_up_sync(full_mask, v, 1); };
        auto right_of = [&](float v) { return __shfl_down_sync(full_mask, v, 1); };
        auto div_of = [&](float2 qx, float left, float2 qy, float wy, float2 up) {
            return make_float2(fmaf(wy, qy.x, fmaf(mxe, qx.x, -left)) - up.x,
                               fmaf(wy, qy.y, fmaf(mxo, qx.y, -qx.x)) - up.y);
        };
        Row<S> x0, x1;
        float2 th0 = make_float2(0.f, 0.f), fy_up = th0, py_up = th0;
        ok = mbar_wait(b_full, 0);
        if (cert::thresholds_from(0) == 0) ok = ok && mbar_wait(b_th, 0);
        if (ok) load_row(0, x1);
#pragma unroll 1
        for (int k = 0; ok && k <= ke; ++k) {
            ok = mbar_wait(b_full + 8 * slot(k + 1), phase(k + 1)) &&
                 mbar_wait(b_th + 8 * slot(k + 1), phase(k + 1));
            if (!ok) break;
            const int t = rf + k;
            x0 = x1;
            load_row(k + 1, x1);
            const float2 th1 = f2(th + slot(k + 1) * 256);
            const unsigned char* const a = ax + slot(k) * Y::aux;
            const float2 al = f2(a + Y::f4 + Y::f1), cl = f2(axc + slot(k) * Y::aux);
            float2 fs = f2(a + Y::f4), fp = PS::f2(x0.p);
            const float wy = (unsigned)t < (unsigned)(G.H - 1) ? 1.f : 0.f;
            // flows y of row t
            float2 fx = PS::f2(x0.qx), fy = PS::f2(x0.qy);
            if (DR) {
                const float u_r = right_of(x0.u.x), ty = tau * wy;
                fx.x -= tau * mxe * (x0.u.y - x0.u.x);
                fx.y -= tau * mxo * (u_r - x0.u.y);
                fy.x -= ty * (x1.u.x - x0.u.x);
                fy.y -= ty * (x1.u.y - x0.u.y);
                const float2 sum = f2(us + slot(k) * 256);
                fp.x += tau * x0.u.x;
                fp.y += tau * x0.u.y;
                fs.x -= tau * sum.x;
                fs.y -= tau * sum.y;
            }
            float2 px = fx, py = fy;
            project1<ANISO, false>(px.x, py.x, al.x);
            project1<ANISO, false>(px.y, py.y, al.y);
            const float2 d = div_of(fx, left_of(fx.y), fy, wy, fy_up);
            const float2 dp = div_of(px, left_of(px.y), py, wy, py_up);
            // primal terms at ub = max(u - theta, 0)
            const float2 ub = make_float2(fmaxf(x0.u.x - th0.x, 0.f), fmaxf(x0.u.y - th0.y, 0.f));
            const float2 ud = make_float2(fmaxf(x1.u.x - th1.x, 0.f), fmaxf(x1.u.y - th1.y, 0.f));
            const float ubr = right_of(ub.x);
            *reinterpret_cast<float2*>(sh + slot(k) * Y::sh) =
                make_float2(cl.x + dp.x, cl.y + dp.y);
            if (own && k > 0) {
                const float gxe = mxe * (ub.y - ub.x), gxo = mxo * (ubr - ub.y);
                const float gye = wy * (ud.x - ub.x), gyo = wy * (ud.y - ub.y);
                const float tve = ANISO ? fabsf(gxe) + fabsf(gye) : sqrtf(gxe * gxe + gye * gye);
                const float tvo = ANISO ? fabsf(gxo) + fabsf(gyo) : sqrtf(gxo * gxo + gyo * gyo);
                const float re = d.x - fs.x + fp.x, ro = d.y - fs.y + fp.y;
                float e = ub.x * cl.x + al.x * tve, r2 = re * re;
                if (pair) {
                    e += ub.y * cl.y + al.y * tvo;
                    r2 += ro * ro;
                }
                df_add(accE, e);
                df_add(accR, r2);
            }
            fy_up = fy;
            py_up = py;
            th0 = th1;
            __syncwarp();
            if (lane == 0) mbar_arrive(b_sf + 8 * slot(k));
        }
    } else if (wib < L + NT) {
        // ---- theta warps: Michelot's iteration -----------------------------
        // theta = (sum_active - 1) / n_active, active = the entries above theta
        // (the thresholds never decrease, so each pass sums and counts that set
        // afresh); stop when the counts no longer change
        for (int i = wib - L; i <= il; i += NT) {
            ok = mbar_wait(b_full + 8 * slot(i), phase(i));
            if (!ok) break;
            const unsigned char* const u0 =
                dsm + slot(i) * Y::state + 3 * Y::fs + 4 * (off4 + 2 * lane);
            float2 u[LC];
            float2 sum = make_float2(0.f, 0.f);
#pragma unroll
            for (int l = 0; l < LC; ++l)
                if (l < L) {
                    u[l] = f2(u0 + l * Seg<4>::cols * 4);
                    sum.x += u[l].x;
                    sum.y += u[l].y;
                }
            int nx = L, ny = L;
            float2 t = make_float2((sum.x - 1.f) / (float)nx, (sum.y - 1.f) / (float)ny);
            for (int it = 0; it < L; ++it) {
                float ax = 0.f, ay = 0.f;
                int mx = 0, my = 0;
#pragma unroll
                for (int l = 0; l < LC; ++l)
                    if (l < L) {
                        if (u[l].x > t.x) {
                            ax += u[l].x;
                            ++mx;
                        }
                        if (u[l].y > t.y) {
                            ay += u[l].y;
                            ++my;
                        }
                    }
                const bool cx = mx != nx && mx > 0, cy = my != ny && my > 0;
                if (!__any_sync(full_mask, cx || cy)) break;
                if (cx) {
                    nx = mx;
                    t.x = (ax - 1.f) / (float)nx;
                }
                if (cy) {
                    ny = my;
                    t.y = (ay - 1.f) / (float)ny;
                }
            }
            reinterpret_cast<float2*>(dsm + Y::o_th + slot(i) * 256)[lane] = t;
            if (DR) reinterpret_cast<float2*>(dsm + Y::o_us + slot(i) * 256)[lane] = sum;
            __syncwarp();
            if (lane == 0) mbar_arrive(b_th + 8 * slot(i));
        }
    } else {
        // ---- last warp: input rows, minima over the labels ------------------
        const uint32_t tx = (uint32_t)L * (3u * Seg<ES>::cols * ES + 2u * Seg<4>::cols * 4u) +
                            (has_al ? 2u : 1u) * Seg<4>::cols * 4u;
        const int x4 = cfirst - off4, xs = cfirst - offs;
        // one map a lane (q_x, q_y, p, u, p_s, C, alpha): its box, its slot's offset
        const int nmaps = has_al ? 7 : 6;
        const CUtensorMap* const map = &M.qx + (lane < nmaps ? lane : 0);
        const int mx = lane < 3 ? xs : x4;
        const int moff = lane < 4 ? lane * Y::fs
                                  : Y::o_aux + (lane == 5 ? 0 : Y::f4 + (lane == 6 ? Y::f1 : 0));
        auto issue = [&](int i) {
            if (i > il) return;
            uint64_t* fb = bar + slot(i);
            if (lane == 0) mbar_arrive_expect_tx(fb, tx);
            __syncwarp();
            unsigned char* d = dsm + moff + (lane < 4 ? slot(i) * Y::state : slot(i) * Y::aux);
            if (lane < nmaps) tma_load_3d(d, map, fb, mx, rf + i, 0);
        };
        for (int i = 0; i < kRing; ++i) issue(i);
        int k = 0;
        for (; k <= ke; ++k) {
            ok = mbar_wait(b_sf + 8 * slot(k), phase(k));
            if (!ok) break;
            const unsigned char* q = dsm + Y::o_sh + slot(k) * Y::sh + lane * 8;
            float2 m = f2(q);
            for (int l = 1; l < L; ++l) {
                const float2 v = f2(q + l * 256);
                m.x = fminf(m.x, v.x);
                m.y = fminf(m.y, v.y);
            }
            if (own && k > 0) df_add(accD, pair ? m.x + m.y : m.x);
            __syncwarp();
            issue(k + kRing);
        }
        if (!ok && lane == 0)  // let the copies in flight land (each wait bounded)
            for (int i = max(0, min(k + kRing, il + 1) - kRing); i < min(k + kRing, il + 1); ++i)
                mbar_wait(b_full + 8 * slot(i), phase(i));
    }
    if (!ok && lane == 0) atomicExch(err, kErrWaitTimeout);
    block_reduce3_store_df(accE, accD, accR, partials + 3 * (size_t)blockIdx.x);
    eval_tail(tail, partials, gridDim.x);
}

// ---- host side -------------------------------------------------------------

template <typename S, bool ANISO, bool DR, int LC>
static cudaError_t launch_potts_cert(const PottsProblem& P, const PottsRowsMaps& M, float tau,
                                     double* partials, const EvalTail& T, int* err,
                                     cudaStream_t st) {
    auto kern = k_potts_cert<S, ANISO, DR, LC>;
    constexpr size_t dyn = cert::Layout<LC, (int)sizeof(S)>::bytes;
    static std::atomic<long long> limit[kMaxDevices];
    cudaError_t e = raise_dyn_smem(limit, kern, dyn);
    if (e != cudaSuccess) return e;
    static std::atomic<long long> memo[LC + 1][kMaxDevices];  // blocks resident per label count
    const int threads = 32 * (P.L + cert::theta_warps(LC) + 1);
    long long resident = 0;
    e = per_device(
        memo[P.L],
        [&](int dev, long long& v) -> cudaError_t {
            int sms = 0, blocks = 0;
            cudaError_t e2 = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
            if (e2 != cudaSuccess) return e2;
            e2 = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, kern, threads, dyn);
            if (e2 != cudaSuccess) return e2;
            v = (long long)sms * (blocks > 0 ? blocks : 1);
            return cudaSuccess;
        },
        resident);
    if (e != cudaSuccess) return e;
    const Grid& G = P.g;
    const int nstrips = (G.W + 59) / 60;
    // band height: whole rounds of resident blocks, each costing its rows and
    // the pipeline's fill; at most eval_blocks(H, W) blocks, the partials'
    // count (60-column strips are fewer than 32-column tiles)
    const long long most = eval_blocks(G.H, G.W) / nstrips;
    long long best = -1;
    int R = G.H;
    for (int rounds = 1; rounds <= 8; ++rounds) {
        long long bands = rounds * resident / nstrips;
        bands = bands > most ? most : bands;
        bands = bands < 1 ? 1 : (bands > G.H ? G.H : bands);
        const int r = (int)((G.H + bands - 1) / bands);
        const long long items = (long long)nstrips * ((G.H + r - 1) / r);
        const long long cost = (items + resident - 1) / resident * (r + 6);
        if (best < 0 || cost < best) {
            best = cost;
            R = r;
        }
    }
    const int nitems = nstrips * ((G.H + R - 1) / R);
    kern<<<nitems, threads, dyn, st>>>(M, P, tau, R, nstrips, partials, T, err);
    return cudaGetLastError();
}

template <typename S>
static cudaError_t potts_cert_s(const PottsProblem& P, const PottsRowsMaps& M, bool aniso, bool dr,
                                float tau, double* partials, const EvalTail& T, int* err,
                                cudaStream_t st) {
#define CMF_CERT_LC(AN, D, LC) launch_potts_cert<S, AN, D, LC>(P, M, tau, partials, T, err, st)
#define CMF_CERT(AN, D)                       \
    (P.L <= 4 ? CMF_CERT_LC(AN, D, 4)         \
              : (P.L <= 8 ? CMF_CERT_LC(AN, D, 8) : CMF_CERT_LC(AN, D, rows::kMaxLabels)))
    if (dr) return aniso ? CMF_CERT(true, true) : CMF_CERT(false, true);
    return aniso ? CMF_CERT(true, false) : CMF_CERT(false, false);
#undef CMF_CERT
#undef CMF_CERT_LC
}

}  // namespace cmf
