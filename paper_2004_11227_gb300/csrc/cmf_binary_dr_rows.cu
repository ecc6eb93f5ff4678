// Binary rPDRQ iteration (Eq. iteration:quadratic:seg, one symmetric red-black
// sweep) on rows brought ahead by TMA, even widths.
//
// Work unit: one block, kWarps adjacent strips of 64 columns (two adjacent
// columns per lane, 56 owned) and a band of rows, streamed top-down.  At step k
// row m enters (u^k and b), the three half-sweeps run on rows m-1, m-2 and m-3,
// and row m-4 is finished (flow steps and reflections) from the flows kept in
// registers since their row entered.  A service warp keeps the next rows of the
// whole block's width in flight with TMA (elements outside the grid read as
// zero): row k + 1 + kRing is issued when every warp has done step k, whose last
// reads were of row k + 1's state slot and of row k - 3's cost / alpha slot.
// Otherwise the warps share nothing: each strip carries its own halo.  A warp at
// step k + 4 has waited for row k + 5, issued after step k was seen done, so four
// barriers tell the steps apart.
//
// What bounds it.  The one-warp strip kernel waited for loads issued a row ahead
// and read the flows a second time four rows on.  At 4096^2, float32, an
// iteration cannot do without 872 MB (128 us at the copy bandwidth); smaller
// grids live in L2, where a step takes 0.4 us however few warps there are.  Four
// strips share a ring because a ring a warp, with a quarter of the width per box,
// kept the copy engine busy (1024^2: 16.5 us), and eight lanes issue the boxes of
// a row because one lane took 0.45 us a step for them.  Halo rows come without
// costs and alpha (512^2: 8.6 -> 8.3 us).  Half-sweeps spaced two rows apart,
// which do not wait for one another, were slower (0.5 us a step, three more
// steps a band).  Measured per iteration (CUDA events), one-warp strips before:
// 4096^2 float32 174 -> 145 us, float16 132 -> 108 us; 2048^2 48 -> 39 us; 1024^2
// 16.5 -> 12.4 us (float16 14.3); 256^2 12.4 -> 6.2 us.  Same results bit for bit.
#include <limits.h>

#include <type_traits>

#include "cmf_potts_rows.cuh"

namespace cmf {
namespace bdr {

constexpr int kRing = 4;   // state rows in shared memory
constexpr int kAux = 8;    // cost and alpha rows
constexpr int kWarps = 4;  // strips per block
constexpr int kOut = 56;   // owned columns of a strip
constexpr int kFill = 9;   // steps beyond a band's rows

// Columns of a staged row: the strips' and what aligning its start to 16 bytes
// can put in front.
template <int ES>
struct Seg {
    static constexpr int align = 16 / ES;
    static constexpr int cols = kWarps * kOut + 8 + (ES == 4 ? 0 : 8);
};

template <int ES>
struct Layout {
    static constexpr int fs = rows::up128(Seg<ES>::cols * ES);
    static constexpr int f4 = rows::up128(Seg<4>::cols * 4);
    static constexpr int state = 4 * fs + f4;  // q_x, q_y, p_s, p_t, u
    static constexpr int aux = 3 * f4;         // C_s, C_t, alpha
    static constexpr int o_aux = kRing * state;
    static constexpr int o_bar = o_aux + kAux * aux;
    static constexpr int bytes = o_bar + 8 * (kRing + 4) + 128;
};

template <typename S, bool ANISO>
__global__ void __launch_bounds__(32 * (kWarps + 1), 3)
    k_binary_dr_rows(const __grid_constant__ BinChainMaps M, BinProblem P, BinState<S> s1,
                     DrCoef D, int R, int nstrips, int* err) {
    using rows::mbar_arrive;
    using rows::mbar_wait;
    using PS = strip::Pair<S>;
    using PF = strip::Pair<float>;
    using SP = typename PS::T;
    constexpr int ES = sizeof(S);
    using Y = Layout<ES>;
    extern __shared__ __align__(128) unsigned char bdr_raw[];
    const Grid G = P.g;
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    unsigned char* const sm = bdr_raw + ((128u - (smem_u32(bdr_raw) & 127u)) & 127u);
    uint64_t* const bar = reinterpret_cast<uint64_t*>(sm + Y::o_bar);
    const uint32_t b_full = smem_u32(bar), b_sf = b_full + 8 * kRing;
    const unsigned full_mask = 0xffffffffu;

    const int r0 = (int)(blockIdx.x / nstrips) * R;  // even: a step's colours are constants
    const int r1 = min(r0 + R, G.H);
    const int cfirst = (int)(blockIdx.x % nstrips) * (kWarps * kOut) - 4;
    const int c = cfirst + kOut * wib + 2 * lane;
    const bool colin = c >= 0 && c < G.W;  // W is even: both columns of the pair
    const bool own = colin && lane >= 2 && lane <= 29;
    const int offs = cfirst & (Seg<ES>::align - 1);  // float32 segments start at cfirst
    // input row i is row rf + i; step k takes in row m = rf + 1 + k and finishes
    // row m - 4
    const int rf = r0 - 4, il = r1 + 3 - rf, ke = il - 1;
    const bool has_al = P.alpha.plane != nullptr;

    if (threadIdx.x == 0) {
        for (int i = 0; i < kRing; ++i) mbar_init(bar + i, 1);
        for (int i = 0; i < 4; ++i) mbar_init(bar + kRing + i, kWarps);
        fence_mbar_init();
    }
    if (!has_al)  // constant alpha: every row's slot holds it
        for (int i = threadIdx.x; i < kAux * Seg<4>::cols; i += blockDim.x) {
            const int r = i / Seg<4>::cols;
            reinterpret_cast<float*>(sm + Y::o_aux + r * Y::aux + 2 * Y::f4)[i - r * Seg<4>::cols] =
                P.alpha.value;
        }
    __syncthreads();

    if (wib == kWarps) {
        // ---- service warp: one box a lane --------------------------------------
        const uint32_t tx = 4u * Seg<ES>::cols * ES + Seg<4>::cols * 4u;
        const uint32_t tx_aux = (has_al ? 3u : 2u) * Seg<4>::cols * 4u;
        const CUtensorMap* const map = &M.qx + (lane < 8 ? lane : 0);
        const int x = lane < 4 ? cfirst - offs : cfirst;
        auto issue = [&](int i) {
            if (i > il) return;
            uint64_t* fb = bar + (i & (kRing - 1));
            const int y = rf + i;
            const bool owned = y >= r0 && y < r1;  // costs and alpha: no halo
            if (lane == 0) mbar_arrive_expect_tx(fb, owned ? tx + tx_aux : tx);
            __syncwarp();
            unsigned char* d = lane < 5 ? sm + (i & (kRing - 1)) * Y::state + lane * Y::fs
                                        : sm + Y::o_aux + (i & (kAux - 1)) * Y::aux +
                                              (lane - 5) * Y::f4;
            if (lane < (owned ? (has_al ? 8 : 7) : 5)) tma_load_3d(d, map, fb, x, y, 0);
        };
        for (int i = 0; i < kRing; ++i) issue(i);
        bool ok = true;
        for (int k = 0; k <= ke; ++k) {
            ok = mbar_wait(b_sf + 8 * (k & 3), (k >> 2) & 1);
            if (!ok) break;
            if (k == 0) issue(kRing);  // row 0's slot, read before step 0
            issue(k + 1 + kRing);
        }
        if (!ok && lane == 0) {
            // a wait ran out: report it and let the copies in flight (at most a
            // ring of rows) land before the shared memory goes
            atomicExch(err, kErrWaitTimeout);
            for (int i = 0; i < kRing; ++i) {
                mbar_wait(b_full + 8 * i, 0);
                mbar_wait(b_full + 8 * i, 1);
            }
        }
        return;
    }

    // ---- strips ----------------------------------------------------------------
    const float mxo = c + 1 < G.W - 1 ? 1.f : 0.f;
    const float ncx_e = (c > 0 ? 1.f : 0.f) + (c < G.W - 1 ? 1.f : 0.f);
    const float ncx_o = 1.f + mxo;
    const unsigned char* const st_s = sm + ES * (offs + kOut * wib + 2 * lane);
    const unsigned char* const st_u = sm + 4 * Y::fs + 4 * kOut * wib + 8 * lane;
    const unsigned char* const ax = sm + Y::o_aux + 4 * kOut * wib + 8 * lane;
    auto sp = [](const unsigned char* q) { return *reinterpret_cast<const SP*>(q); };
    auto f2 = [](const unsigned char* q) { return *reinterpret_cast<const float2*>(q); };
    int o = (rf - 3) * G.pitch + c;
    // rings over rows m, m-1, ...: row m at position U
    float2 V[8], B[8];
    SP qx[8], qy[8], ps[8], pt[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        V[i] = B[i] = make_float2(0.f, 0.f);
        qx[i] = qy[i] = ps[i] = pt[i] = PS::zero();
    }
    bool ok = mbar_wait(b_full, 0);
    if (ok) qy[7] = sp(st_s + Y::fs);
    // one step, k = 8 n + U
    auto body = [&](auto uc, int k) -> bool {
        constexpr int U = decltype(uc)::value;
        constexpr int I = (U + 1) & (kRing - 1);  // ring slot of input row k + 1
        constexpr uint32_t ph = ((U + 1) / kRing) & 1;
        const int m = rf + 1 + k;
        if (!mbar_wait(b_full + 8 * I, ph)) return false;
        {  // row m enters: u^k and b
            const unsigned char* q = st_s + I * Y::state;
            qx[U] = sp(q);
            qy[U] = sp(q + Y::fs);
            ps[U] = sp(q + 2 * Y::fs);
            pt[U] = sp(q + 3 * Y::fs);
            V[U] = f2(st_u + I * Y::state);
            const float2 x = PS::f2(qx[U]), y = PS::f2(qy[U]), qu = PS::f2(qy[(U + 7) & 7]);
            const float2 s = PS::f2(ps[U]), t = PS::f2(pt[U]);
            const float left = __shfl_up_sync(full_mask, x.y, 1);
            const float wy = m < G.H - 1 ? 1.f : 0.f;
            B[U].x = -D.sigma * (x.x - left + wy * y.x - qu.x + t.x - s.x);
            B[U].y = -D.sigma * (mxo * x.y - x.x + wy * y.y - qu.y + t.y - s.y);
        }
        // half-sweeps on rows m-1 (red), m-2 (black), m-3 (red); m has the
        // parity of k + 1
#pragma unroll
        for (int s = 0; s < 3; ++s) {
            const int j = m - 1 - s;
            const bool j_odd = ((U + s) & 1) != 0;
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
        const unsigned char* a = ax + ((U - 3) & (kAux - 1)) * Y::aux;
        const float2 cs = f2(a), ct = f2(a + Y::f4), al = f2(a + 2 * Y::f4);
        __syncwarp();
        if (lane == 0) mbar_arrive(b_sf + 8 * (U & 3));
        if (t >= r0 && own) {
            const float wy = t < G.H - 1 ? 1.f : 0.f;
            const float gx_e = un.y - un.x, gx_o = mxo * (u_right - un.y);
            const float gy_e = wy * (ud.x - un.x), gy_o = wy * (ud.y - un.y);
            const float2 fx = PS::f2(qx[F]), fy = PS::f2(qy[F]);
            const float2 fs = PS::f2(ps[F]), ft = PS::f2(pt[F]);
            float qx_e, qy_e, ps_e, pt_e, qx_o, qy_o, ps_o, pt_o;
            binary_dr_flows<S, ANISO>(D, un.x, gx_e, gy_e, fx.x, fy.x, fs.x, ft.x, al.x, cs.x,
                                      ct.x, qx_e, qy_e, ps_e, pt_e);
            // the strips' results add the odd columns' squares the other way round
            // (float32)
            binary_dr_flows<S, ANISO, ES == 4>(D, un.y, gx_o, gy_o, fx.y, fy.y, fs.y, ft.y, al.y,
                                               cs.y, ct.y, qx_o, qy_o, ps_o, pt_o);
            PF::st(s1.u + o, un.x, un.y);
            PS::st(s1.qx + o, qx_e, qx_o);
            PS::st(s1.qy + o, qy_e, qy_o);
            PS::st(s1.ps + o, ps_e, ps_o);
            PS::st(s1.pt + o, pt_e, pt_o);
        }
        o += G.pitch;
        return true;
    };
    if (ok) {
#pragma unroll 1
        for (int k = 0; k <= ke; k += 8) {
#define CMF_STEP(U) \
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

template <typename S, bool ANISO>
static cudaError_t launch(const BinProblem& P, const BinState<S>& b, const DrCoef& D,
                          const BinChainMaps& M, int* err, cudaStream_t st) {
    auto kern = k_binary_dr_rows<S, ANISO>;
    constexpr int threads = 32 * (kWarps + 1);
    constexpr size_t dyn = Layout<(int)sizeof(S)>::bytes;
    static std::atomic<long long> limit[kMaxDevices], memo[kMaxDevices];
    cudaError_t e = raise_dyn_smem(limit, kern, dyn);
    if (e != cudaSuccess) return e;
    long long resident = 0;
    e = per_device(
        memo,
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
    const int nstrips = (G.W + kWarps * kOut - 1) / (kWarps * kOut);
    // band height (even): whole rounds of resident blocks, each costing its rows
    // and the steps that fill the pipeline
    long long best = -1;
    int R = G.H + (G.H & 1);
    for (int rounds = 1; rounds <= 8; ++rounds) {
        long long bands = rounds * resident / nstrips;
        bands = bands < 1 ? 1 : (bands > G.H ? G.H : bands);
        int r = (int)((G.H + bands - 1) / bands);
        r += r & 1;
        const long long items = (long long)nstrips * ((G.H + r - 1) / r);
        const long long cost = (items + resident - 1) / resident * (r + kFill);
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
static cudaError_t step(const BinProblem& P, const BinStateV& b, bool aniso, const DrCoef& D,
                        const BinChainMaps& M, int* err, cudaStream_t st) {
    const BinState<S> B = b.as<S>();
    return aniso ? launch<S, true>(P, B, D, M, err, st) : launch<S, false>(P, B, D, M, err, st);
}

}  // namespace bdr

bool binary_dr_rows_eligible(const BinProblem& P, int storage, const DrCoef& D,
                             const BinStateV& a, const BinStateV& b) {
    // one sweep, two columns per lane
    return D.sweeps == 1 && P.g.W % 2 == 0 &&
           (size_t)P.g.H * (size_t)P.g.pitch <= (size_t)INT_MAX &&
           binary_chain_eligible(P, storage, a, b, b);
}

cudaError_t binary_dr_rows_maps(const BinProblem& P, int storage, const BinStateV& s,
                                BinChainMaps& m, const BinChainMaps* planes) {
    const int es = (int)dtype_size(storage);
    return binary_row_maps(P, storage, s, es == 4 ? bdr::Seg<4>::cols : bdr::Seg<2>::cols,
                           bdr::Seg<4>::cols, m, planes);
}

cudaError_t binary_dr_rows_step(int storage, const BinProblem& P, const BinStateV& b, bool aniso,
                                const DrCoef& D, const BinChainMaps& M, int* err,
                                cudaStream_t st) {
    switch (storage) {
        case CMF_F32: return bdr::step<float>(P, b, aniso, D, M, err, st);
        case CMF_F16: return bdr::step<__half>(P, b, aniso, D, M, err, st);
        default: return bdr::step<__nv_bfloat16>(P, b, aniso, D, M, err, st);
    }
}

}  // namespace cmf
