// Binary ADMM, up to four iterations per launch by a chain of warps (Eq.
// rpADMMII, Eq. rpADMMI, pADMM-TY, ALG1), with the certificates of the result
// as one more link.
//
// Work unit: one block, a strip of 128 columns (four adjacent columns per
// lane) and a band of rows, streamed top-down.  Warp t < T makes iteration
// k+t+1: at step s it takes row r+1 of its input (row r it has), forms g of
// that row, and makes row r = r0 - T + s - 2 t, which the next warp of the
// chain reads one step later.  Warp 0's input rows, and every row's C_s, C_t
// and alpha, come by TMA (elements outside the grid read as zero); the rows
// between two warps pass through shared memory, two slots each, in the storage
// type as a store and a load would round them; the last warp writes the
// result.  With CERT two further warps sum the certificates of the rows the
// last one makes (one the energy, one the dual value and the residual: either
// is about an iteration's work).  A producer warp keeps kIn rows in flight and waits for each row
// before the step that reads it, so the one block barrier per step is all the
// other warps wait on:
//   - a slot between two warps is written in one step, read in the next and
//     rewritten in the one after;
//   - an input slot is refilled after the barrier behind the step that read
//     it; a C_s / C_t / alpha slot (a ring of 16 rows) after the last warp of
//     the chain has used it (kIn + 2 T < 18, with CERT 16).
// Each iteration needs one more column and row on every side and the first
// one two to the left and above: T + 1 columns of the strip's left end and T
// of its right end are halo (with CERT one more on the right).
//
// What bounds it.  The two-iteration strip kernel keeps both stages of two
// columns in 119 registers, 16 warps per SM, and issues 124-158 thread
// instructions per pixel and iteration (60% of the issue slots); odd widths
// ran one iteration per launch on tiles.  A chain holds one iteration per
// warp, so four columns a lane fit 96 registers (one address, predicate and
// shuffle for four pixels; float32 spills 4 to 8 bytes, with the certificates
// up to 60), and the state passes through DRAM once per four iterations (at
// 4096^2 that floor is 32 us per iteration).  At 1024^2 that is 111 thread
// instructions with the bands' halo rows, 59% of the issue slots; the rest is
// the barrier (2.0 to 2.2 stalls per issue) and the dependent chain of a row.  Two
// columns a lane, one or two rows per barrier, took 1.2 to 1.4 times the
// instructions.  Small grids are bound by the
// chain's fill (three steps per iteration) and the launch.  Measured per
// iteration (CUDA events, float32; before: two iterations per launch by strips,
// odd widths tiles): 4096^2 87.2 -> 52.2 us, 2048^2 23.8 -> 15.0 us, 1024^2
// 8.25 -> 5.73 us, 64^2 3.6 -> 2.1 us, 901 x 1407 15.9 -> 7.2 us, 2001^2
// 56.5 -> 16.0 us; float16 4096^2 85.2 -> 56.0 us.
#pragma once

#include <climits>
#include <type_traits>

#include "cmf_kernels.cuh"
#include "cmf_strip.cuh"
#include "cmf_tma.cuh"

namespace cmf {
namespace chain {

using strip::Pair;

constexpr int kMaxIters = 4, kMaxCert = 3;  // iterations per launch, and with certificates
constexpr int kAux = 16;      // C_s / C_t / alpha rows in shared memory
constexpr int kIn = 4;        // input rows in flight
constexpr int kCols = 128;    // columns of a strip

template <int ES>
struct Seg {  // columns of a staged row segment: the strip and its aligned start
    static constexpr int align = 16 / ES;
    static constexpr int cols = kCols + (ES == 4 ? 0 : 8);
    static constexpr int row = cols * ES;                     // bytes
    static constexpr int slot = (row + 127) / 128 * 128;
};

// Byte offsets from a 128-byte aligned base.
template <int ES>
struct Layout {
    static constexpr int fs = Seg<ES>::slot, f4 = Seg<4>::slot;
    static constexpr int in = 4 * fs + f4;     // q_x, q_y, p_s, p_t, u of a row
    static constexpr int aux = 3 * f4;         // C_s, C_t, alpha of a row
    static constexpr int ms = kCols * ES;
    static constexpr int mid = 4 * ms + f4;    // a row between two warps
    static constexpr int o_in = kAux * aux;
    static constexpr int o_mid = o_in + kIn * in;
    __host__ __device__ static int o_bar(int links) { return o_mid + links * 2 * mid; }
    __host__ __device__ static int bytes(int links) { return o_bar(links) + 8 * kIn + 128; }
};

// Halo columns on the left and right, in whole lanes.
__host__ __device__ constexpr int left_cols(int T) { return (T + 4) / 4 * 4; }
__host__ __device__ constexpr int right_cols(int T, bool cert) {
    return (T + (cert ? 4 : 3)) / 4 * 4;
}

// Four adjacent elements of a plane in float32 and in the storage type.
struct F4 {
    float v[4];
};
template <typename S>
struct Quad {  // 16-bit flows: two stored pairs
    using PS = Pair<S>;
    struct alignas(8) T {
        typename PS::T a, b;
    };
    static __device__ __forceinline__ T ld(const unsigned char* q) {
        return *reinterpret_cast<const T*>(q);
    }
    static __device__ __forceinline__ F4 f4(T t) {
        const float2 a = PS::f2(t.a), b = PS::f2(t.b);
        return F4{{a.x, a.y, b.x, b.y}};
    }
    static __device__ __forceinline__ T pk(const F4& f) {
        return T{PS::pk(f.v[0], f.v[1]), PS::pk(f.v[2], f.v[3])};
    }
};
template <>
struct Quad<float> {
    using T = float4;
    static __device__ __forceinline__ T ld(const unsigned char* q) {
        return *reinterpret_cast<const float4*>(q);
    }
    static __device__ __forceinline__ F4 f4(T t) { return F4{{t.x, t.y, t.z, t.w}}; }
    static __device__ __forceinline__ T pk(const F4& f) {
        return make_float4(f.v[0], f.v[1], f.v[2], f.v[3]);
    }
};

template <typename S>
struct Row {
    typename Quad<S>::T qx, qy, ps, pt;
    float4 u;
};

__device__ __forceinline__ float rsqrt_ftz(float x) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// P_alpha (Eq. projections) in the roundings of strip::project_sel; swap: the
// squares added the other way round.  The smallest normal number bounds the
// reciprocal root (where the squared norm is below it the scale is at most
// alpha / 1.1e-19, and the result stays within alpha).
template <bool ANISO>
__device__ __forceinline__ void project(float& x, float& y, float al, bool swap) {
    al = fmaxf(al, 0.f);
    if (ANISO) {
        x = fminf(fmaxf(x, -al), al);
        y = fminf(fmaxf(y, -al), al);
    } else {
        const float p = swap ? y : x, q = swap ? x : y;
        const float n2 = __fmaf_rn(p, p, __fmul_rn(q, q));
        const float t = __fmul_rn(al, rsqrt_ftz(fmaxf(n2, 1.17549435e-38f)));
        const float s = n2 > __fmul_rn(al, al) ? t : 1.f;
        x = __fmul_rn(x, s);
        y = __fmul_rn(y, s);
    }
}

}  // namespace chain

// SIMPLE: rpADMMII / rpADMMI / pADMMI; otherwise pADMM-TY or ALG1.  Every
// rounding is that of the strip kernels (EVEN: even widths) or of the tile
// kernels (odd widths), so the results of a problem do not depend on which of
// them ran it: the strip kernels add the squares of the projection the other
// way round at odd columns, and with 16-bit flows the second iteration of
// their pairs does at even ones too (iter0: the call's index of warp 0's
// iteration).
//
// One block: the band r0 .. r1-1 of the strip whose first staged column is
// cfirst (hl and hr: its halo columns), from the state of M into s1.
template <typename S, bool ANISO, bool SIMPLE, bool EVEN, bool CERT>
__device__ __forceinline__ void binary_chain_block(
    const BinChainMaps& M, const BinProblem& Pr, const BinState<S>& s1, const AdmmCoef& K,
    const int T, const int iter0, const int r0, const int r1, const int cfirst, const int hl,
    const int hr, DF& accE, DF& accD, DF& accR, int* err) {
    using namespace chain;
    using St = Store<S>;
    using QS = Quad<S>;
    using QF = Quad<float>;
    constexpr int ES = sizeof(S);
    using Y = Layout<ES>;
    extern __shared__ __align__(128) unsigned char dsm_raw[];
    const Grid G = Pr.g;
    unsigned char* const dsm = dsm_raw + ((128u - (smem_u32(dsm_raw) & 127u)) & 127u);
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const unsigned full_mask = 0xffffffffu;
    const int links = T - 1 + (CERT ? 1 : 0);  // handovers between warps

    const int c = cfirst + 4 * lane;
    const bool own = 4 * lane >= hl && 4 * lane < kCols - hr && c < G.W;
    const int offs = cfirst & (Seg<ES>::align - 1);  // float32 segments start at cfirst
    // steps -2 .. se; input row i is row rx + i, read by warp 0 at step i - 2
    const int rows = r1 - r0, rx = r0 - T - 1;
    const int se = rows + 3 * T - (CERT ? 1 : 3);
    const int il = rows + 2 * T + (CERT ? 1 : 0);  // last input row
    uint64_t* const bar = reinterpret_cast<uint64_t*>(dsm + Y::o_bar(links));
    const bool has_al = Pr.alpha.plane != nullptr;

    if (threadIdx.x == 0) {
        for (int i = 0; i < kIn; ++i) mbar_init(bar + i, 1);
        fence_mbar_init();
    }
    if (!has_al)  // constant alpha: every slot holds it
        for (int i = threadIdx.x; i < kAux * kCols; i += blockDim.x)
            reinterpret_cast<float*>(dsm + i / kCols * Y::aux + 2 * Y::f4)[i % kCols] =
                Pr.alpha.value;
    __syncthreads();

    if (wib == T + (CERT ? 2 : 0)) {
        // ---- producer ------------------------------------------------------
        const uint32_t tx = 4u * Seg<ES>::row + (has_al ? 4u : 3u) * Seg<4>::row;
        const int xs = cfirst - offs;
        auto issue = [&](int i) {
            if (i > il || lane != 0) return;
            unsigned char* d = dsm + Y::o_in + (i & (kIn - 1)) * Y::in;
            unsigned char* a = dsm + (i & (kAux - 1)) * Y::aux;
            uint64_t* b = bar + (i & (kIn - 1));
            mbar_arrive_expect_tx(b, tx);
            tma_load_3d(d, &M.qx, b, xs, rx + i, 0);
            tma_load_3d(d + Y::fs, &M.qy, b, xs, rx + i, 0);
            tma_load_3d(d + 2 * Y::fs, &M.ps, b, xs, rx + i, 0);
            tma_load_3d(d + 3 * Y::fs, &M.pt, b, xs, rx + i, 0);
            tma_load_3d(d + 4 * Y::fs, &M.u, b, cfirst, rx + i, 0);
            tma_load_3d(a, &M.Cs, b, cfirst, rx + i, 0);
            tma_load_3d(a + Y::f4, &M.Ct, b, cfirst, rx + i, 0);
            if (has_al) tma_load_3d(a + 2 * Y::f4, &M.al, b, cfirst, rx + i, 0);
        };
        for (int i = 0; i < kIn; ++i) issue(i);
        bool ok = true;
        for (int s = -2; s <= se; ++s) {
            // row s + 2 is there when the step begins; after a wait that ran
            // out the steps go on without waiting (the state is then undefined)
            const int i = s + 2;
            if (i <= il && ok &&
                !mbar_wait_bounded(bar + (i & (kIn - 1)), (i / kIn) & 1, kWaitLimitCycles)) {
                ok = false;
                if (lane == 0) atomicExch(err, kErrWaitTimeout);
            }
            __syncthreads();
            if (i > 0 && ok) issue(i - 1 + kIn);  // row i - 1 was read in the step before
        }
        // after a timeout: let the copies in flight land (each wait bounded)
        if (!ok)
            for (int i = 0; i < kIn; ++i) {
                mbar_wait_bounded(bar + i, 0, kWaitLimitCycles);
                mbar_wait_bounded(bar + i, 1, kWaitLimitCycles);
            }
    } else {
        const int t = min(wib, T);  // place in the chain
        // 0/1 weights of the x differences (0 left of the grid, at the last
        // column and right of it); only a strip's edges have zeros
        float mx[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) mx[i] = (c + i >= 0 && c + i < G.W - 1) ? 1.f : 0.f;
        const unsigned char* const in_s = dsm + Y::o_in + ES * (offs + 4 * lane);
        const unsigned char* const in_u = dsm + Y::o_in + 4 * Y::fs + 16 * lane;
        unsigned char* const mid = dsm + Y::o_mid + lane * 4 * ES;
        const unsigned char* const rd = mid + (t - 1) * 2 * Y::mid;
        unsigned char* const wr = mid + t * 2 * Y::mid;
        const int mu = 4 * Y::ms + lane * (16 - 4 * ES);  // u of a row between two warps
        // the strip's last lane with columns of an odd or ragged width
        const bool ragged = cfirst + kCols > G.W && (G.W & 3);

        auto row_w = [&](int r) { return (unsigned)r < (unsigned)(G.H - 1) ? 1.f : 0.f; };
        auto left_of = [&](float v) { return __shfl_up_sync(full_mask, v, 1); };
        auto right_of = [&](float v) { return __shfl_down_sync(full_mask, v, 1); };
        // divergence of a row's flows, given q_y above
        auto div_of = [&](const F4& qx, const F4& qy, float wy, const F4& up) {
            const float left = left_of(qx.v[3]);
            F4 d;
#pragma unroll
            for (int i = 0; i < 4; ++i)
                d.v[i] = __fsub_rn(fmaf(wy, qy.v[i],
                                        fmaf(mx[i], qx.v[i], i ? -qx.v[i ? i - 1 : 0] : -left)),
                                   up.v[i]);
            return d;
        };
        uint32_t slot = 0;                        // warp 0's input slot
        uint32_t arow = (uint32_t)(-1 - 2 * t) & (kAux - 1);  // aux slot of row r
        const unsigned char* const ax = dsm + 16 * lane;
        // a row of this warp's input: TMA rows for warp 0, else the row the
        // warp before made in the last step (slot par)
        auto load = [&](int par, Row<S>& x) {
            if (t == 0) {
                const unsigned char* q = in_s + slot * Y::in;
                x.qx = QS::ld(q);
                x.qy = QS::ld(q + Y::fs);
                x.ps = QS::ld(q + 2 * Y::fs);
                x.pt = QS::ld(q + 3 * Y::fs);
                x.u = QF::ld(in_u + slot * Y::in);
            } else {
                const unsigned char* q = rd + par * Y::mid;
                x.qx = QS::ld(q);
                x.qy = QS::ld(q + Y::ms);
                x.ps = QS::ld(q + 2 * Y::ms);
                x.pt = QS::ld(q + 3 * Y::ms);
                x.u = QF::ld(q + mu);
            }
        };
        const F4 zero = {{0.f, 0.f, 0.f, 0.f}};
        Row<S> x[2];  // rows r and r + 1
        x[0].qx = x[0].qy = x[0].ps = x[0].pt = QS::pk(zero);
        x[0].u = QF::pk(zero);
        x[1] = x[0];
        int r = r0 - T - 2 - 2 * t;

        if (!CERT || t < T) {
            // ---- an iteration ----------------------------------------------
            F4 g[2] = {zero, zero}, qn_up = zero;
            float wy0 = 0.f;
            const bool last = t == T - 1;
            const bool swap_even = EVEN && ES == 2 && ((iter0 + t) & 1);
            const int sa = 3 * t - 2, sz = rows + 2 * T - 2 + t + (CERT ? 1 : 0);
            uint32_t o = (uint32_t)(r * G.pitch + c);
            auto body = [&](auto uc, int s) {
                constexpr int A = decltype(uc)::value, B = A ^ 1;
                __syncthreads();
                if (s >= sa && s <= sz) {
                    load(B, x[B]);
                    const unsigned char* a = ax + arow * Y::aux;
                    const F4 al = QF::f4(QF::ld(a + 2 * Y::f4));
                    // g = div q + p_t - p_s - u / c of row r + 1
                    const float wy1 = row_w(r + 1);
                    {
                        const F4 ps = QS::f4(x[B].ps), pt = QS::f4(x[B].pt), u = QF::f4(x[B].u);
                        g[B] = div_of(QS::f4(x[B].qx), QS::f4(x[B].qy), wy1, QS::f4(x[A].qy));
#pragma unroll
                        for (int i = 0; i < 4; ++i)
                            g[B].v[i] = fmaf(u.v[i], -K.inv_c,
                                             __fsub_rn(__fadd_rn(g[B].v[i], pt.v[i]), ps.v[i]));
                    }
                    // q^{k+1} of row r
                    Row<S> y;
                    {
                        F4 tx = QS::f4(x[A].qx), ty = QS::f4(x[A].qy);
                        const float my = wy0 * K.inv_a, gr = right_of(g[A].v[0]);
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            const float gx = (i < 3 ? g[A].v[i < 3 ? i + 1 : 3] : gr) - g[A].v[i];
                            const float gy = g[B].v[i] - g[A].v[i];
                            if (!SIMPLE && !EVEN) {
                                tx.v[i] = __fadd_rn(tx.v[i], __fmul_rn(gx, mx[i] * K.inv_a));
                                ty.v[i] = __fadd_rn(ty.v[i], __fmul_rn(gy, my));
                            } else {
                                tx.v[i] = fmaf(gx, mx[i] * K.inv_a, tx.v[i]);
                                ty.v[i] = fmaf(gy, my, ty.v[i]);
                            }
                            project<ANISO>(tx.v[i], ty.v[i], al.v[i], i & 1 ? EVEN : swap_even);
                        }
                        y.qx = QS::pk(tx);
                        y.qy = QS::pk(ty);
                    }
                    // its divergence, then p_s, p_t, u
                    {
                        const F4 ty = QS::f4(y.qy);
                        const F4 d = div_of(QS::f4(y.qx), ty, wy0, qn_up);
                        qn_up = ty;
                        const F4 ps = QS::f4(x[A].ps), pt = QS::f4(x[A].pt), u = QF::f4(x[A].u);
                        const F4 cs = QF::f4(QF::ld(a)), ct = QF::f4(QF::ld(a + Y::f4));
                        F4 sn, tn, un;
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            if (SIMPLE) {
                                const float rd = __fmul_rn(K.rho_p, d.v[i]);
                                const float e = __fsub_rn(pt.v[i], ps.v[i]);
                                tn.v[i] = St::rt(fminf(fmaf(K.inv_a1, fmaf(u.v[i], K.inv_c, -rd),
                                                            fmaf(-K.rho_a1, e, pt.v[i])),
                                                       ct.v[i]));
                                sn.v[i] = St::rt(
                                    fminf(fmaf(K.inv_a1,
                                               __fadd_rn(fmaf(-u.v[i], K.inv_c, rd), K.inv_c),
                                               fmaf(K.rho_a1, e, ps.v[i])),
                                          cs.v[i]));
                                const float h = fmaf(-K.omr, e, __fsub_rn(tn.v[i], sn.v[i]));
                                un.v[i] = __fsub_rn(u.v[i], __fmul_rn(K.cu, __fadd_rn(h, rd)));
                            } else {
                                binary_pu<S>(K, g[A].v[i], d.v[i], ps.v[i], pt.v[i], u.v[i],
                                             cs.v[i], ct.v[i], sn.v[i], tn.v[i], un.v[i]);
                            }
                        }
                        y.ps = QS::pk(sn);
                        y.pt = QS::pk(tn);
                        y.u = QF::pk(un);
                    }
                    if (CERT || !last) {
                        unsigned char* q = wr + A * Y::mid;
                        *reinterpret_cast<typename QS::T*>(q) = y.qx;
                        *reinterpret_cast<typename QS::T*>(q + Y::ms) = y.qy;
                        *reinterpret_cast<typename QS::T*>(q + 2 * Y::ms) = y.ps;
                        *reinterpret_cast<typename QS::T*>(q + 3 * Y::ms) = y.pt;
                        *reinterpret_cast<float4*>(q + mu) = y.u;
                    }
                    if (last && own && r >= r0 && r < r1) {
                        if (!ragged || c + 3 < G.W) {
                            *reinterpret_cast<typename QS::T*>(s1.qx + o) = y.qx;
                            *reinterpret_cast<typename QS::T*>(s1.qy + o) = y.qy;
                            *reinterpret_cast<typename QS::T*>(s1.ps + o) = y.ps;
                            *reinterpret_cast<typename QS::T*>(s1.pt + o) = y.pt;
                            *reinterpret_cast<float4*>(s1.u + o) = y.u;
                        } else {  // the last columns one by one
                            const F4 tx = QS::f4(y.qx), ty = QS::f4(y.qy), sn = QS::f4(y.ps),
                                     tn = QS::f4(y.pt), un = QF::f4(y.u);
#pragma unroll
                            for (int i = 0; i < 3; ++i)
                                if (c + i < G.W) {
                                    St::st(s1.qx + o + i, tx.v[i]);
                                    St::st(s1.qy + o + i, ty.v[i]);
                                    St::st(s1.ps + o + i, sn.v[i]);
                                    St::st(s1.pt + o + i, tn.v[i]);
                                    s1.u[o + i] = un.v[i];
                                }
                        }
                    }
                    wy0 = wy1;
                }
                o += G.pitch;
                ++r;
                arow = (arow + 1) & (kAux - 1);
                slot = (slot + 1) & (kIn - 1);
            };
#pragma unroll 1
            for (int s = -2; s <= se; s += 2) {
                body(std::integral_constant<int, 0>(), s);
                if (s + 1 > se) break;
                body(std::integral_constant<int, 1>(), s + 1);
            }
        } else {
            // ---- certificates of the rows the last iteration makes ---------
            const int sa = 3 * T - 2;
            if (wib == T) {
                // primal energy E at clip(u, 0, 1)
                const unsigned char* const ru = rd + mu;
                F4 un = zero;
#pragma unroll 1
                for (int s = -2; s <= se; ++s) {
                    __syncthreads();
                    if (s >= sa) {
                        F4 ub = un;
                        un = QF::f4(QF::ld(ru + ((s & 1) ^ 1) * Y::mid));
#pragma unroll
                        for (int i = 0; i < 4; ++i) un.v[i] = __saturatef(un.v[i]);
                        const float ubr = right_of(ub.v[0]);
                        if (own && r >= r0 && r < r1) {
                            const unsigned char* a = ax + arow * Y::aux;
                            const F4 cs = QF::f4(QF::ld(a)), ct = QF::f4(QF::ld(a + Y::f4)),
                                     al = QF::f4(QF::ld(a + 2 * Y::f4));
                            const float wy = row_w(r);
#pragma unroll
                            for (int h = 0; h < 4; h += 2) {  // a pair's terms together
                                float e = 0.f, tv = 0.f;
#pragma unroll
                                for (int i = h; i < h + 2; ++i) {
                                    if (c + i >= G.W) continue;
                                    const float gx =
                                        mx[i] *
                                        ((i < 3 ? ub.v[i < 3 ? i + 1 : 3] : ubr) - ub.v[i]);
                                    const float gy = wy * (un.v[i] - ub.v[i]);
                                    tv += al.v[i] * (ANISO ? fabsf(gx) + fabsf(gy)
                                                           : sqrtf(gx * gx + gy * gy));
                                    e += (1.f - ub.v[i]) * cs.v[i] + ub.v[i] * ct.v[i];
                                }
                                df_add(accE, tv);
                                df_add(accE, e);
                            }
                        }
                    }
                    ++r;
                    arow = (arow + 1) & (kAux - 1);
                }
            } else {
                // dual value D of the re-projected flows, squared residual
                F4 py_up = zero, qn_up = zero;  // q_y of the row above, projected and as it is
#pragma unroll 1
                for (int s = -2; s <= se; ++s) {
                    __syncthreads();
                    if (s > sa) {
                        // row r: the slot the last iteration wrote two steps ago
                        // is being rewritten, so the row was kept
                        const unsigned char* a = ax + arow * Y::aux;
                        const F4 al = QF::f4(QF::ld(a + 2 * Y::f4));
                        const float wy = row_w(r);
                        const F4 qx = QS::f4(x[0].qx), qy = QS::f4(x[0].qy);
                        F4 px = qx, py = qy;
#pragma unroll
                        for (int i = 0; i < 4; ++i)
                            project<ANISO>(px.v[i], py.v[i], al.v[i], EVEN && (i & 1));
                        const F4 d = div_of(qx, qy, wy, qn_up), dp = div_of(px, py, wy, py_up);
                        if (own && r >= r0 && r < r1) {
                            const F4 ps = QS::f4(x[0].ps), pt = QS::f4(x[0].pt);
                            const F4 cs = QF::f4(QF::ld(a)), ct = QF::f4(QF::ld(a + Y::f4));
#pragma unroll
                            for (int h = 0; h < 4; h += 2) {
                                float r2 = 0.f, m = 0.f;
#pragma unroll
                                for (int i = h; i < h + 2; ++i) {
                                    if (c + i >= G.W) continue;
                                    const float res = d.v[i] - ps.v[i] + pt.v[i];
                                    r2 += res * res;
                                    m += fminf(cs.v[i], ct.v[i] + dp.v[i]);
                                }
                                df_add(accR, r2);
                                df_add(accD, m);
                            }
                        }
                        py_up = py;
                        qn_up = qy;
                    }
                    if (s >= sa) load((s & 1) ^ 1, x[0]);
                    ++r;
                    arow = (arow + 1) & (kAux - 1);
                }
            }
        }
    }
}

// One launch of the single-problem solver.
template <typename S, bool ANISO, bool SIMPLE, bool EVEN, bool CERT>
__global__ void __launch_bounds__(32 * (CERT ? chain::kMaxCert + 3 : chain::kMaxIters + 1), CERT ? 3 : 4)
    k_binary_chain(const __grid_constant__ BinChainMaps M, BinProblem P, BinState<S> s1,
                   AdmmCoef K, int T, int iter0, int R, int nstrips, double* partials,
                   EvalTail tail, int* err) {
    const int hl = chain::left_cols(T), hr = chain::right_cols(T, CERT);
    const int r0 = (blockIdx.x / nstrips) * R;
    DF accE = {0.f, 0.f}, accD = {0.f, 0.f}, accR = {0.f, 0.f};
    binary_chain_block<S, ANISO, SIMPLE, EVEN, CERT>(
        M, P, s1, K, T, iter0, r0, min(r0 + R, P.g.H),
        (int)(blockIdx.x % nstrips) * (chain::kCols - hl - hr) - hl, hl, hr, accE, accD, accR,
        err);
    if (CERT) {
        block_reduce3_store_df(accE, accD, accR, partials + 3 * (size_t)blockIdx.x);
        eval_tail(tail, partials, gridDim.x);
    }
}

// ---- host side -------------------------------------------------------------

template <typename S, bool ANISO, bool SIMPLE, bool EVEN, bool CERT>
static cudaError_t launch_binary_chain(const BinProblem& P, const BinState<S>& b,
                                       const AdmmCoef& K, int T, int iter0, const BinChainMaps& M,
                                       double* partials, int max_blocks, const EvalTail& tail,
                                       int* err, cudaStream_t st) {
    auto kern = k_binary_chain<S, ANISO, SIMPLE, EVEN, CERT>;
    const int links = T - 1 + (CERT ? 1 : 0);
    const size_t dyn = chain::Layout<(int)sizeof(S)>::bytes(links);
    static std::atomic<long long> limit[kMaxDevices];
    cudaError_t e = raise_dyn_smem(limit, kern, dyn);
    if (e != cudaSuccess) return e;
    // blocks resident per device and chain length
    static std::atomic<long long> memo[chain::kMaxIters + 1][kMaxDevices];
    const int threads = 32 * (T + (CERT ? 3 : 1));
    long long resident = 0;
    e = per_device(
        memo[T],
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
    const int out = chain::kCols - chain::left_cols(T) - chain::right_cols(T, CERT);
    const int nstrips = (G.W + out - 1) / out;
    // band height: whole rounds of resident blocks, each costing its rows
    // plus the steps that fill and drain the chain
    long long best = -1;
    int R = G.H;
    for (int rounds = 1; rounds <= 8; ++rounds) {
        long long bands = rounds * resident / nstrips;
        if (CERT && bands > max_blocks / nstrips) bands = max_blocks / nstrips;
        bands = bands < 1 ? 1 : (bands > G.H ? G.H : bands);
        const int r = (int)((G.H + bands - 1) / bands);
        const long long items = (long long)nstrips * ((G.H + r - 1) / r);
        const long long cost = (items + resident - 1) / resident * (r + 3 * T + 2);
        if (best < 0 || cost < best) {
            best = cost;
            R = r;
        }
    }
    const int nitems = nstrips * ((G.H + R - 1) / R);
    kern<<<nitems, threads, dyn, st>>>(M, P, b, K, T, iter0, R, nstrips, partials, tail, err);
    return cudaGetLastError();
}

template <typename S, bool SIMPLE, bool EVEN>
static cudaError_t binary_chain_step_s(const BinProblem& P, const BinStateV& b, bool aniso,
                                       const AdmmCoef& K, int T, int iter0, const BinChainMaps& M,
                                       double* partials, int max_blocks, const EvalTail* cert,
                                       int* err, cudaStream_t st) {
    const BinState<S> B = b.as<S>();
    const EvalTail tail = cert ? *cert : EvalTail();
#define CMF_CHAIN(AN, CE)                                                                  \
    launch_binary_chain<S, AN, SIMPLE, EVEN, CE>(P, B, K, T, iter0, M, partials, max_blocks, tail, \
                                                 err, st)
    if (cert) return aniso ? CMF_CHAIN(true, true) : CMF_CHAIN(false, true);
    return aniso ? CMF_CHAIN(true, false) : CMF_CHAIN(false, false);
#undef CMF_CHAIN
}

}  // namespace cmf
