// Potts rPDRQ iteration with the labels side by side (Eq. pdrq:4labels, one
// symmetric red-black sweep), even widths.
//
// Work unit: one block, a strip of 64 columns (two adjacent columns per lane,
// 56 owned) and a band of rows, streamed top-down.  Warp l < L runs label l:
// at step k row m enters (u^k and b), the three half-sweeps run on rows m-1,
// m-2 and m-3, and row t = m-4 is finished (flow steps and reflections), as in
// the strip kernel.  A service warp keeps the next rows in flight with TMA
// (elements outside the grid read as zero), sums u^k over the labels for the
// rows about to enter (b needs it), and sums the finished u for the reflection
// of pbar_s; so no plane of label sums is kept between launches.  mbarriers
// couple them: full (a row has arrived), UR (its label sum is there), SF (every
// label is done with a step).
//   - row k + 1 + kRing is issued when every label has done step k: its state
//     slot was read in step k at the latest, its C / p_s / alpha slot held row
//     k - 3, whose last readers are step k and the service warp just before;
//   - the label sum of row k + kLead is given when step k's finished u has been
//     summed; a finished-u slot is rewritten kSh steps on, by a warp that has
//     waited for row k + kSh + 1's sum.
//
// What bounds it.  The one-label strip kernel reads alpha, p_s and the plane of
// label sums again for every label and the reflected flows a second time four
// rows on, and its dependent loads leave the issue slots idle; here every plane
// is read once, ahead of use, and a flow stays in registers from its row's
// entry to its row's end.  At 2048^2, L = 4, float32 an iteration cannot do
// without 638 MB (94 us at the copy bandwidth).  What is left is each row's
// chain of shuffles, three quotients per pixel pair and the projection, hence
// as many label warps per SM as the registers hold: short rings, so that four
// blocks of 5 warps or two of 9 share an SM (rings of eight rows: 133 us, and
// 105 at L = 8, 1024^2), and the label sums three rows ahead (two: 121 us).
// Measured per iteration (CUDA events), one-label strips before: 2048^2 L = 4
// float32 209 -> 115 us; 1024^2 L = 16 227 -> 133; 1024^2 L = 8 118 -> 66;
// 512^2 L = 4 22.6 -> 16.5; 128^2 L = 16 56 -> 12.4 (there a block is one
// strip, and its labels no longer follow one another).  Same results bit for bit.
#pragma once

#include "cmf_potts_rows.cuh"

namespace cmf {
namespace dr_rows {

constexpr int kRing = 4;  // state rows (and label sums) in shared memory
constexpr int kAux = 8;   // C, p_s, alpha rows
constexpr int kSh = 4;    // finished-u rows
constexpr int kLead = 3;  // label sums are given this many rows ahead
static_assert(kLead <= kSh + 1, "a finished-u row is summed before its slot is rewritten");

template <int LC, int ES>
struct Layout {
    static constexpr int fs = rows::up128(LC * rows::Seg<ES>::cols * ES);
    static constexpr int f4 = rows::up128(LC * rows::Seg<4>::cols * 4);
    static constexpr int f1 = rows::up128(rows::Seg<4>::cols * 4);
    static constexpr int state = 3 * fs + f4;  // q_x, q_y, p, u
    static constexpr int aux = f4 + 2 * f1;    // C, p_s, alpha
    static constexpr int sh = LC * 256;
    static constexpr int o_aux = kRing * state;
    static constexpr int o_sh = o_aux + kAux * aux;
    static constexpr int o_us = o_sh + kSh * sh;
    static constexpr int o_bar = o_us + kRing * 256;
    static constexpr int bytes = o_bar + 8 * (2 * kRing + 4) + 128;
    static_assert(bytes <= 232448, "shared memory of a block");
};

}  // namespace dr_rows

template <typename S, bool ANISO, int LC>
__global__ void __launch_bounds__(32 * (LC + 1), LC == 4 ? 4 : (LC == 8 ? 2 : 1))
    k_potts_dr_rows(const __grid_constant__ PottsRowsMaps M, PottsProblem P, PottsState<S> s1,
                    DrCoef D, int R, int nstrips, int* err) {
    using namespace dr_rows;
    using rows::mbar_arrive;
    using rows::mbar_wait;
    using rows::Seg;
    using strip::project_sel;
    using strip::Pair;
    using PS = Pair<S>;
    constexpr int ES = sizeof(S);
    using Y = Layout<LC, ES>;
    extern __shared__ __align__(128) unsigned char dsm_raw[];
    const Grid G = P.g;
    const int L = P.L;
    unsigned char* const dsm = dsm_raw + ((128u - (smem_u32(dsm_raw) & 127u)) & 127u);
    uint64_t* const bar = reinterpret_cast<uint64_t*>(dsm + Y::o_bar);
    const uint32_t b_full = smem_u32(bar), b_ur = b_full + 8 * kRing, b_sf = b_ur + 8 * kRing;
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const unsigned full_mask = 0xffffffffu;

    const int r0 = (blockIdx.x / nstrips) * R;  // even: a step's colours are constants
    const int r1 = min(r0 + R, G.H);
    const int cfirst = (int)(blockIdx.x % nstrips) * 56 - 4;
    const int c = cfirst + 2 * lane;
    const bool colin = c >= 0 && c < G.W;  // W is even: both columns of the pair
    const bool own = colin && lane >= 2 && lane <= 29;
    const int offs = cfirst & (Seg<ES>::align - 1);  // float32 segments start at cfirst
    // input row i is row rf + i; step k takes in row m = rf + 1 + k and finishes
    // row m - 4
    const int rf = r0 - 4, il = r1 + 3 - rf, ke = il - 1;

    if (threadIdx.x == 0) {
        for (int i = 0; i < 2 * kRing; ++i) mbar_init(bar + i, 1);
        for (int i = 0; i < 4; ++i) mbar_init(bar + 2 * kRing + i, L);
        fence_mbar_init();
    }
    const bool has_al = P.alpha.plane != nullptr;
    if (!has_al)  // constant alpha: every row's slot holds it
        for (int i = threadIdx.x; i < kAux * Seg<4>::cols; i += blockDim.x) {
            const int r = i / Seg<4>::cols;
            reinterpret_cast<float*>(dsm + Y::o_aux + r * Y::aux + Y::f4 +
                                     Y::f1)[i - r * Seg<4>::cols] = P.alpha.value;
        }
    __syncthreads();
    bool ok = true;
    auto f2 = [](const unsigned char* q) { return *reinterpret_cast<const float2*>(q); };

    if (wib == L) {
        // ---- service warp --------------------------------------------------
        const uint32_t tx = (uint32_t)L * (3u * Seg<ES>::cols * ES + 2u * Seg<4>::cols * 4u) +
                            (has_al ? 2u : 1u) * Seg<4>::cols * 4u;
        const int xs = cfirst - offs;
        // one map a lane (q_x, q_y, p, u, p_s, C, alpha): its box, its slot's
        // offset (one lane for all: 2048^2, L = 4 117 us, 1024^2, L = 8 70)
        const int nmaps = has_al ? 7 : 6;
        const CUtensorMap* const map = &M.qx + (lane < nmaps ? lane : 0);
        const int mx = lane < 3 ? xs : cfirst;
        const int moff = lane < 4 ? lane * Y::fs
                                  : Y::o_aux + (lane == 5 ? 0 : Y::f4 + (lane == 6 ? Y::f1 : 0));
        auto issue = [&](int i) {
            if (i > il) return;
            uint64_t* fb = bar + (i & (kRing - 1));
            if (lane == 0) mbar_arrive_expect_tx(fb, tx);
            __syncwarp();
            unsigned char* d =
                dsm + moff + (lane < 4 ? (i & (kRing - 1)) * Y::state : (i & (kAux - 1)) * Y::aux);
            if (lane < nmaps) tma_load_3d(d, map, fb, mx, rf + i, 0);
        };
        // sum over the labels, in label order, of float2s `stride` bytes apart
        auto label_sum = [&](const unsigned char* q, int stride) {
            float2 v[LC];
#pragma unroll
            for (int l = 0; l < LC; ++l)
                if (l < L) v[l] = f2(q + l * stride);
            float2 a = make_float2(0.f, 0.f);
#pragma unroll
            for (int l = 0; l < LC; ++l)
                if (l < L) {
                    a.x += v[l].x;
                    a.y += v[l].y;
                }
            return a;
        };
        auto give_sum = [&](int i) {  // U of input row i
            if (i > il) return true;
            if (!mbar_wait(b_full + 8 * (i & (kRing - 1)), (i / kRing) & 1)) return false;
            const float2 a = label_sum(
                dsm + (i & (kRing - 1)) * Y::state + 3 * Y::fs + 8 * lane, Seg<4>::cols * 4);
            reinterpret_cast<float2*>(dsm + Y::o_us + (i & (kRing - 1)) * 256)[lane] = a;
            __syncwarp();
            if (lane == 0) mbar_arrive(b_ur + 8 * (i & (kRing - 1)));
            return true;
        };
        for (int i = 0; i < kRing; ++i) issue(i);
        int k = 0;
        for (int i = 0; i < kLead && ok; ++i) ok = give_sum(i);
        for (; ok && k <= ke; ++k) {
            ok = mbar_wait(b_sf + 8 * (k & 3), (k >> 2) & 1);
            if (!ok) break;
            const int t = rf + k - 3;  // finished in step k
            if (t >= r0) {
                const float2 us = label_sum(dsm + Y::o_sh + (k & (kSh - 1)) * Y::sh + 8 * lane, 256);
                if (own) {
                    const float2 pbs =
                        f2(dsm + Y::o_aux + ((k - 3) & (kAux - 1)) * Y::aux + Y::f4 + 8 * lane);
                    const float ps1x = pbs.x - D.tau * us.x, ps1y = pbs.y - D.tau * us.y;
                    Pair<float>::st(
                        s1.ps + t * G.pitch + c,
                        pbs.x + D.rho * ((2.f * ps1x - pbs.x + D.tau) - ps1x),
                        pbs.y + D.rho * ((2.f * ps1y - pbs.y + D.tau) - ps1y));
                }
            }
            __syncwarp();
            if (k == 0) issue(kRing);  // row 0's slot, read before step 0
            issue(k + 1 + kRing);
            ok = give_sum(k + kLead);
        }
        if (!ok && lane == 0) {
            // a wait ran out: report it and let the copies in flight land
            // before the block's shared memory goes
            atomicExch(err, kErrWaitTimeout);
            const int n = min(k + 2 + kRing, il + 1);
            for (int i = max(0, n - kRing); i < n; ++i)
                mbar_wait(b_full + 8 * (i & (kRing - 1)), (i / kRing) & 1);
        }
        return;
    }

    // ---- label warps -------------------------------------------------------
    const int l = wib;
    const float stL = D.sigma * D.tau * (float)L, st_ = D.sigma * D.tau;
    const float mxo = c + 1 < G.W - 1 ? 1.f : 0.f;
    const float ncx_e = (c > 0 ? 1.f : 0.f) + (c < G.W - 1 ? 1.f : 0.f);
    const float ncx_o = 1.f + mxo;
    const unsigned char* const st_s = dsm + l * Seg<ES>::cols * ES + ES * (offs + 2 * lane);
    const unsigned char* const st_u = dsm + 3 * Y::fs + l * Seg<4>::cols * 4 + 8 * lane;
    const unsigned char* const ax = dsm + Y::o_aux + 8 * lane;
    const unsigned char* const axc = ax + l * Seg<4>::cols * 4;
    const unsigned char* const usr = dsm + Y::o_us + 8 * lane;
    unsigned char* const sh = dsm + Y::o_sh + l * 256 + 8 * lane;
    auto sp = [](const unsigned char* q) {
        return *reinterpret_cast<const typename PS::T*>(q);
    };
    uint32_t o = (uint32_t)l * (uint32_t)G.plane + (uint32_t)((rf - 3) * G.pitch + c);
    // rings over rows m, m-1, ...: row m at position U
    float2 V[8], B[8];
    typename PS::T qx[8], qy[8], pp[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        V[i] = B[i] = make_float2(0.f, 0.f);
        qx[i] = qy[i] = pp[i] = PS::zero();
    }
    ok = mbar_wait(b_full, 0);
    if (ok) qy[7] = sp(st_s + Y::fs);
    // one step, k = 8 n + U
    auto body = [&](auto uc, int k) -> bool {
        constexpr int U = decltype(uc)::value;
        constexpr int I = (U + 1) & (kRing - 1);  // ring slot of input row k + 1
        constexpr uint32_t ph = ((U + 1) / kRing) & 1;
        const int m = rf + 1 + k;
        if (!mbar_wait(b_full + 8 * I, ph)) return false;
        if (!mbar_wait(b_ur + 8 * I, ph)) return false;
        // aux row of input row k + 1 + d
        auto aux = [&](int d) { return ((U + 1 + d) & (kAux - 1)) * Y::aux; };
        {  // row m enters: u^k and b
            const unsigned char* q = st_s + I * Y::state;
            qx[U] = sp(q);
            qy[U] = sp(q + Y::fs);
            pp[U] = sp(q + 2 * Y::fs);
            const float2 in_u = f2(st_u + I * Y::state), UU = f2(usr + I * 256);
            const float2 in_ps = f2(ax + aux(0) + Y::f4);
            const float2 x = PS::f2(qx[U]), y = PS::f2(qy[U]), p = PS::f2(pp[U]);
            const float2 qu = PS::f2(qy[(U + 7) & 7]);
            const float left = __shfl_up_sync(full_mask, x.y, 1);
            const float wy = m < G.H - 1 ? 1.f : 0.f;
            float2 b;
            b.x = -D.sigma * (x.x - left + wy * y.x - qu.x + p.x - in_ps.x) +
                  (stL * in_u.x - st_ * UU.x);
            b.y = -D.sigma * (mxo * x.y - x.x + wy * y.y - qu.y + p.y - in_ps.y) +
                  (stL * in_u.y - st_ * UU.y);
            B[U] = b;  // not used outside the grid
            V[U] = in_u;
        }
        // half-sweeps on rows m-1 (red), m-2 (black), m-3 (red); m has the
        // parity of k + 1
#pragma unroll
        for (int s = 0; s < 3; ++s) {
            const int j = m - 1 - s;
            constexpr int kOdd = (U + 1) & 1;
            const bool j_odd = ((kOdd + 1 + s) & 1) != 0;
            const bool act_e = !j_odd == ((s & 1) == 0);
            const float2 cur = V[(U + 7 - s) & 7], up = V[(U + 6 - s) & 7], dn = V[(U + 8 - s) & 7];
            const float2 bj = B[(U + 7 - s) & 7];
            const float ncy = (j > 0 ? 1.f : 0.f) + (j < G.H - 1 ? 1.f : 0.f);
            const bool in = colin && j >= 0 && j < G.H;
            if (act_e) {
                const float left = __shfl_up_sync(full_mask, cur.y, 1);
                const float v = __fdividef(bj.x * D.inv_st + (left + cur.y + up.x + dn.x),
                                           D.kappa + ncx_e + ncy);
                V[(U + 7 - s) & 7].x = in ? v : cur.x;
            } else {
                const float right = __shfl_down_sync(full_mask, cur.x, 1);
                const float v = __fdividef(bj.y * D.inv_st + (cur.x + right + up.y + dn.y),
                                           D.kappa + ncx_o + ncy);
                V[(U + 7 - s) & 7].y = in ? v : cur.y;
            }
        }
        // row t = m - 4 is final: flow steps and reflections
        const int t = m - 4;
        constexpr int F = (U + 4) & 7;
        const float2 un = V[F], ud = V[(U + 5) & 7];
        const float u_right = __shfl_down_sync(full_mask, un.x, 1);
        *reinterpret_cast<float2*>(sh + (U & (kSh - 1)) * Y::sh) = un;
        const float2 al = f2(ax + aux(-4) + Y::f4 + Y::f1), cl = f2(axc + aux(-4));
        __syncwarp();
        if (lane == 0) mbar_arrive(b_sf + 8 * (U & 3));
        if (t >= r0 && own) {
            const float wy = t < G.H - 1 ? 1.f : 0.f;
            const float gx[2] = {un.y - un.x, mxo * (u_right - un.y)};
            const float gy[2] = {wy * (ud.x - un.x), wy * (ud.y - un.y)};
            const float2 x = PS::f2(qx[F]), y = PS::f2(qy[F]), p = PS::f2(pp[F]);
            const float qbx[2] = {x.x, x.y}, qby[2] = {y.x, y.y}, pb[2] = {p.x, p.y};
            const float cc[2] = {cl.x, cl.y}, a[2] = {al.x, al.y}, u[2] = {un.x, un.y};
            float oqx[2], oqy[2], op[2];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const float q1 = qbx[e] - D.tau * gx[e], q2 = qby[e] - D.tau * gy[e];
                float tx = 2.f * q1 - qbx[e], ty = 2.f * q2 - qby[e];
                project_sel<ANISO>(tx, ty, a[e]);
                oqx[e] = qbx[e] + D.rho * (tx - q1);
                oqy[e] = qby[e] + D.rho * (ty - q2);
                const float p1 = pb[e] + D.tau * u[e];
                op[e] = pb[e] + D.rho * (fminf(2.f * p1 - pb[e], cc[e]) - p1);
            }
            Pair<float>::st(s1.u + o, un.x, un.y);
            PS::st(s1.qx + o, oqx[0], oqx[1]);
            PS::st(s1.qy + o, oqy[0], oqy[1]);
            PS::st(s1.p + o, op[0], op[1]);
        }
        o += G.pitch;
        return true;
    };
    if (ok) {
#pragma unroll 1
        for (int k = 0; k <= ke; k += 8) {
#define CMF_STEP(U)                                                                      \
    if (k + U > ke || !(ok = body(std::integral_constant<int, U>(), k + U))) break
            CMF_STEP(0);
            CMF_STEP(1);
            CMF_STEP(2);
            CMF_STEP(3);
            CMF_STEP(4);
            CMF_STEP(5);
            CMF_STEP(6);
            CMF_STEP(7);
#undef CMF_STEP
        }
    }
    if (!ok && lane == 0) atomicExch(err, kErrWaitTimeout);
}

// ---- host side -------------------------------------------------------------

template <typename S, bool ANISO, int LC>
static cudaError_t launch_potts_dr_rows(const PottsProblem& P, const PottsState<S>& b,
                                        const DrCoef& D, const PottsRowsMaps& M, int* err,
                                        cudaStream_t st) {
    auto kern = k_potts_dr_rows<S, ANISO, LC>;
    constexpr size_t dyn = dr_rows::Layout<LC, (int)sizeof(S)>::bytes;
    static std::atomic<long long> limit[kMaxDevices];
    cudaError_t e = raise_dyn_smem(limit, kern, dyn);
    if (e != cudaSuccess) return e;
    static std::atomic<long long> memo[LC + 1][kMaxDevices];  // blocks resident per label count
    const int threads = 32 * (P.L + 1);
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
    const int nstrips = (G.W + 55) / 56;
    // band height (even): whole rounds of resident blocks, each costing its
    // rows and the seven that fill the pipeline
    long long best = -1;
    int R = G.H + (G.H & 1);
    for (int rounds = 1; rounds <= 8; ++rounds) {
        long long bands = rounds * resident / nstrips;
        bands = bands < 1 ? 1 : (bands > G.H ? G.H : bands);
        int r = (int)((G.H + bands - 1) / bands);
        r += r & 1;
        const long long items = (long long)nstrips * ((G.H + r - 1) / r);
        const long long cost = (items + resident - 1) / resident * (r + 9);
        if (best < 0 || cost < best) {
            best = cost;
            R = r;
        }
    }
    const int nitems = nstrips * ((G.H + R - 1) / R);
    kern<<<nitems, threads, dyn, st>>>(M, P, b, D, R, nstrips, err);
    return cudaGetLastError();
}

template <typename S>
static cudaError_t potts_dr_rows_s(const PottsProblem& P, const PottsStateV& b, bool aniso,
                                   const DrCoef& D, const PottsRowsMaps& M, int* err,
                                   cudaStream_t st) {
    const PottsState<S> B = b.as<S>();
#define CMF_DR(AN)                                                                         \
    (P.L <= 4 ? launch_potts_dr_rows<S, AN, 4>(P, B, D, M, err, st)                        \
              : (P.L <= 8 ? launch_potts_dr_rows<S, AN, 8>(P, B, D, M, err, st)            \
                          : launch_potts_dr_rows<S, AN, rows::kMaxLabels>(P, B, D, M, err, st)))
    return aniso ? CMF_DR(true) : CMF_DR(false);
#undef CMF_DR
}

}  // namespace cmf
