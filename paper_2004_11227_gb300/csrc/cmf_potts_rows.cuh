// Potts ADMM, one or two iterations per launch, labels side by side (Eq.
// multi:fg:4, the Eckstein-Bertsekas Potts equations after Thm 2, pADMM-TY,
// ALG1).
//
// Work unit: one block, a strip of 64 columns (two adjacent columns per lane)
// and a band of rows, streamed top-down.  Warp l < L runs label l; one or two
// service warps keep the next rows of every plane in flight with TMA (one box
// of L row segments per field and row; elements outside the grid read as
// zero) and sum the labels' shares of the p_s update.
//
// Stage A makes iteration k+1 of row j as the one-label strip kernel does and
// puts the label's share of the p_s update into shared memory; the service
// warp adds the L shares in label order and gives p_s^{k+1} of the row back.
// With T == 2, stage B makes iteration k+2 of row j-3 from A's rows j-3 and
// j-2, which by then have their p_s^{k+1}; iteration k+1 never reaches
// memory.  Warps are coupled by mbarriers only: labels arrive once per step
// (SF: shares full), wait for the p_s of the row two steps back (PR: p_s
// ready) and for their next input row (full).  No other barrier is needed:
//   - a state row's slot is free once every label has arrived for the row
//     above it (the labels have it in registers by then), a cost / p_s /
//     alpha slot three arrivals later (stage B's last read);
//   - a share slot is rewritten four rows on, after its writer has waited for
//     a p_s that the service warp gave after summing it (T == 2), or for an
//     input row issued after that (T == 1);
//   - a service warp that only brings rows waits for the labels' steps no longer
//     than it has rows to issue (cmf_rows_order.cuh);
//   - stage B's shares of row s-3 are complete when every label has arrived
//     for row s.
// The multipliers travel as w = u - cu p_s between launches, as in the
// one-label strip kernel.
//
// What bounds it.  The one-label strip kernel reads alpha and p_s again for
// every label and moves the state once per iteration (588 B per pixel and
// iteration at L = 16, float32: 1.45 ms at 4096^2 at the copy bandwidth; it
// took 2.29 ms); here alpha and p_s are read once and the state moves once per
// two iterations (half the bytes: 0.73 ms).  What is left is instruction
// issue and the latency of a row's chain of shuffles: 75 thread instructions
// per label-pixel and iteration (float16 flows 83, for the conversions), four
// label warps per scheduler (96 registers, 4 to 20 bytes of them spilled at two
// iterations), 59-61% of the issue slots, DRAM at 69% (float16 43%; 2048^2,
// L = 16).  Hence scalar
// arithmetic with the coefficients as constant operands (packed float32
// instructions spent what they saved on register moves), rings whose
// positions are constants (the row loop is unrolled by their length, eight),
// 32-bit output indexes, and stage B before stage A rather than interleaved
// (which spilled).  Measured per iteration (CUDA events), one-label strips
// (odd widths: TMA tiles) before: 4096^2 L = 16 float32 2293 -> 937 us,
// float16 1618 -> 964 us; 2048^2 L = 4 float32 150 -> 61.5 us; 512^2 L = 4
// 26.8 -> 8.4 us; 721 x 1283, L = 8 94 -> 28 us.
#pragma once

#include <type_traits>

#include "cmf_kernels.cuh"
#include "cmf_rows_order.cuh"
#include "cmf_strip.cuh"
#include "cmf_tma.cuh"

namespace cmf {
namespace rows {

using strip::Pair;

constexpr int kMaxLabels = 16;

// Columns of a staged row segment: 64 plus what aligning its start to 16
// bytes can put in front.
template <int ES>
struct Seg {
    static constexpr int align = 16 / ES;
    static constexpr int cols = 64 + (ES == 4 ? 4 : 8);
};

__host__ __device__ constexpr int up128(int b) { return (b + 127) / 128 * 128; }

// Shared memory of a block for up to LC labels (byte offsets from a 128-byte
// aligned base).  LC is a template parameter so that a warp reaches every
// field and slot with one register and constant offsets.
template <int LC, int ES, bool TILE>
struct Layout {
    static constexpr int fs = up128(LC * Seg<ES>::cols * ES);  // a flow field of a row
    static constexpr int f4 = up128(LC * Seg<4>::cols * 4);    // a float32 field of a row
    static constexpr int f1 = up128(Seg<4>::cols * 4);         // one plane of a row
    static constexpr int state = 3 * fs + f4;                  // q_x, q_y, p, u
    static constexpr int aux = f4 + 2 * f1;                    // C, p_s, alpha
    static constexpr int sh = LC * (TILE ? 512 : 256);         // shares of a row
    static constexpr int o_aux = kState * state;
    static constexpr int o_sha = o_aux + kAux * aux;
    static constexpr int o_shb = o_sha + kSh * sh;
    static constexpr int o_ps = o_shb + kSh * sh;
    static constexpr int o_bar = o_ps + kPs * 256;
    static constexpr int bytes = o_bar + 8 * (kAux + 4 + 4) + 128;  // + alignment of the base
};

__device__ __forceinline__ float2 add2(float2 a, float2 b) {
    return make_float2(__fadd_rn(a.x, b.x), __fadd_rn(a.y, b.y));
}
__device__ __forceinline__ float2 sub2(float2 a, float2 b) {
    return make_float2(__fsub_rn(a.x, b.x), __fsub_rn(a.y, b.y));
}
__device__ __forceinline__ float2 mul2(float2 a, float b) {
    return make_float2(__fmul_rn(a.x, b), __fmul_rn(a.y, b));
}
__device__ __forceinline__ float2 fma2(float2 a, float b, float2 c) {
    return make_float2(__fmaf_rn(a.x, b, c.x), __fmaf_rn(a.y, b, c.y));
}
__device__ __forceinline__ float rsqrt_ftz(float x) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// P_alpha (Eq. projections), the scale selected, in the roundings of
// strip::project_sel.  The smallest normal number bounds the reciprocal root:
// where the squared norm is below it (|q| < 1.1e-19) the scale is
// alpha / 1.1e-19 at most, and the result stays within alpha.  SWAP: the
// squares are added the other way round.
template <bool ANISO, bool SWAP>
__device__ __forceinline__ void project1(float& x, float& y, float al) {
    al = fmaxf(al, 0.f);
    if (ANISO) {
        x = fminf(fmaxf(x, -al), al);
        y = fminf(fmaxf(y, -al), al);
    } else {
        const float n2 = SWAP ? __fmaf_rn(y, y, __fmul_rn(x, x)) : __fmaf_rn(x, x, __fmul_rn(y, y));
        const float t = __fmul_rn(al, rsqrt_ftz(fmaxf(n2, 1.17549435e-38f)));
        const float s = n2 > __fmul_rn(al, al) ? t : 1.f;
        x = __fmul_rn(x, s);
        y = __fmul_rn(y, s);
    }
}

__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ __noinline__ inline bool mbar_wait_slow(uint32_t bar, uint32_t parity) {
    const long long t0 = clock64();
    while (!mbar_try(bar, parity))
        if (clock64() - t0 > kWaitLimitCycles) return false;
    return true;
}
// Wait for a barrier's phase, about one second at most.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity) {
    if (mbar_try(bar, parity)) return true;
    return mbar_wait_slow(bar, parity);
}

template <typename S>
struct Row {
    typename Pair<S>::T qx, qy, p;
    float2 u;  // u^k (stage A's input), v (its output), then u^{k+1}
};

}  // namespace rows

// SIMPLE: rpADMMII / rpADMMI / pADMMI; otherwise pADMM-TY or ALG1.  The
// roundings are those of the one-label strip kernel, or (TILE: odd widths) of
// the TMA tile kernel, which sums the two parts of the p_s update apart: a
// solve's p_s keeps a rounding difference of single iterations (its weakly
// determined directions hardly contract), so the results of a problem do not
// depend on which kernel ran it.  fused (TILE): products rounded into the sums.
//
// One block: the band r0 .. r1-1 of the strip whose first staged column is
// cfirst, from the state of M into s1.
template <typename S, bool ANISO, bool SIMPLE, int T, int LC, bool TILE>
__device__ __forceinline__ void potts_rows_block(const PottsRowsMaps& M, const PottsProblem& P,
                                                 const PottsState<S>& s1, const AdmmCoef& K,
                                                 const float cu_in, const int r0, const int r1,
                                                 const int cfirst, const int fused, int* err) {
    using namespace rows;
    using St = Store<S>;
    using PS = Pair<S>;
    constexpr int ES = sizeof(S);
    using Y = Layout<LC, ES, TILE>;
    constexpr int HL = T == 2 ? 2 : 1;  // halo lanes on each side
    extern __shared__ __align__(128) unsigned char dsm_raw[];
    const Grid G = P.g;
    const int L = P.L;
    unsigned char* const dsm = dsm_raw + ((128u - (smem_u32(dsm_raw) & 127u)) & 127u);
    uint64_t* const bar = reinterpret_cast<uint64_t*>(dsm + Y::o_bar);
    const uint32_t b_full = smem_u32(bar), b_sf = b_full + 8 * kAux, b_pr = b_sf + 8 * 4;
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const unsigned full_mask = 0xffffffffu;

    const int c = cfirst + 2 * lane;
    const bool own = lane >= HL && lane <= 31 - HL && c < G.W;
    const bool pair = c + 1 < G.W;  // else the last column of an odd width alone
    const int off4 = cfirst & (Seg<4>::align - 1), offs = cfirst & (Seg<ES>::align - 1);

    // rows read: rf .. rl; stage A runs on rows rf+1 .. rl-1 (its flows of the
    // first only serve the divergence of the next), stage B on r0-1 .. r1-1.
    // Step k handles row j = js + k in stage A and row j - 3 in stage B; input
    // row rf + i has index i.
    const int rf = r0 - 1 - T, rl = r1 + T - 1;
    const int js = rf + 1, ke = (T == 2 ? r1 + 2 : r1 - 1) - js, il = rl - rf;

    if (threadIdx.x == 0) {
        for (int i = 0; i < kAux; ++i) mbar_init(bar + i, 1);
        for (int i = 0; i < 4; ++i) {
            mbar_init(bar + kAux + i, L);
            mbar_init(bar + kAux + 4 + i, 1);
        }
        fence_mbar_init();
        // rows js-2 and js-1 have no stage-A p_s: their (unused) phases are over
        mbar_arrive(b_pr);
        mbar_arrive(b_pr + 8);
    }
    if (T == 2)  // and what stage B reads for them is finite
        for (int i = threadIdx.x; i < kPs * 32; i += blockDim.x)
            reinterpret_cast<float2*>(dsm + Y::o_ps)[i] = make_float2(0.f, 0.f);
    const bool has_al = P.alpha.plane != nullptr;
    if (!has_al)  // constant alpha: every row's slot holds it
        for (int i = threadIdx.x; i < kAux * Seg<4>::cols; i += blockDim.x) {
            const int r = i / Seg<4>::cols;
            reinterpret_cast<float*>(dsm + Y::o_aux + r * Y::aux + Y::f4 +
                                     Y::f1)[i - r * Seg<4>::cols] = P.alpha.value;
        }
    __syncthreads();
    bool ok = true;

    if (wib >= L) {
        // ---- service warps: the label sums; the input rows -------------------
        constexpr bool two = service_warps(T, LC) == 2;
        if (wib >= L + service_warps(T, LC)) return;  // a block sized for more labels
        const bool sums = !two || wib == L, inputs = !two || wib > L;
        const uint32_t tx = (uint32_t)L * (3u * Seg<ES>::cols * ES + 2u * Seg<4>::cols * 4u) +
                            (has_al ? 2u : 1u) * Seg<4>::cols * 4u;
        const int x4 = cfirst - off4, xs = cfirst - offs;
        // one map a lane (q_x, q_y, p, u, p_s, C, alpha): its box, its slot's
        // offset (one lane issuing a row's seven boxes held the rows up: 2048^2,
        // L = 4 float32 63.5 -> 61.5 us, float16 69.6 -> 63.9; 4096^2, L = 16
        // 975 -> 937)
        const int nmaps = has_al ? 7 : 6;
        const CUtensorMap* const map = &M.qx + (lane < nmaps ? lane : 0);
        const int mx = lane < 3 ? xs : x4;
        const int moff = lane < 4 ? lane * Y::fs
                                  : Y::o_aux + (lane == 5 ? 0 : Y::f4 + (lane == 6 ? Y::f1 : 0));
        auto issue = [&](int i) {
            if (i > il) return;
            uint64_t* fb = bar + (i & (kAux - 1));
            if (lane == 0) mbar_arrive_expect_tx(fb, tx);
            __syncwarp();
            unsigned char* d =
                dsm + moff + (lane < 4 ? (i & (kState - 1)) * Y::state : (i & (kAux - 1)) * Y::aux);
            if (lane < nmaps) tma_load_3d(d, map, fb, mx, rf + i, 0);
        };
        int issued = 0;  // input rows issued
        if (inputs)
            for (; issued < kState; ++issued) issue(issued);
        // p_s^{k+1} of a row from p_s^k and the L shares of a slot, summed in
        // label order
        auto update = [&](float2 p_s, const unsigned char* base) {
            float2 a, b = make_float2(0.f, 0.f);
            if (TILE && SIMPLE) {
                const float4* q = reinterpret_cast<const float4*>(base) + lane;
                a = b;
                for (int l = 0; l < L; ++l) {
                    const float4 v = q[32 * l];
                    const float2 d = make_float2(v.x, v.y);
                    a = fused ? fma2(d, K.rho_p, a) : add2(a, mul2(d, K.rho_p));
                    b = add2(b, make_float2(v.z, v.w));
                }
            } else {
                const float2* q = reinterpret_cast<const float2*>(base) + lane;
                float2 v[LC];
#pragma unroll
                for (int l = 0; l < LC; ++l)
                    if (l < L) v[l] = q[32 * l];
                a = v[0];
#pragma unroll
                for (int l = 1; l < LC; ++l)
                    if (l < L) a = add2(a, v[l]);
            }
            return make_float2(potts_ps_update(K, p_s.x, a.x, b.x),
                               potts_ps_update(K, p_s.y, a.y, b.y));
        };
        auto store_ps = [&](int t, float2 n) {
            float* o = s1.ps + t * G.pitch + c;
            if (pair) Pair<float>::st(o, n.x, n.y);
            else o[0] = n.x;
        };
        float2* const psr = reinterpret_cast<float2*>(dsm + Y::o_ps) + lane;
        const int kl = sums ? ke : last_input_step(il);
        int k = 0;
        for (; k <= kl; ++k) {
            const int s = js + k;
            ok = mbar_wait(b_sf + 8 * (k & 3), (k >> 2) & 1);
            if (!ok) break;
            if (sums) {
                const float2 ps0 = *reinterpret_cast<const float2*>(
                    dsm + Y::o_aux + ((k + 1) & (kAux - 1)) * Y::aux + Y::f4 +
                    4 * (off4 + 2 * lane));
                const float2 n = update(ps0, dsm + Y::o_sha + (k & 3) * Y::sh);
                if (T == 2) {
                    psr[(k & (kPs - 1)) * 32] = n;
                    __syncwarp();
                    if (lane == 0) mbar_arrive(b_pr + 8 * ((k + 2) & 3));
                    if (s - 3 >= r0) {
                        const float2 nb = update(psr[((k - 3) & (kPs - 1)) * 32],
                                                 dsm + Y::o_shb + ((k - 3) & 3) * Y::sh);
                        if (own) store_ps(s - 3, nb);
                    }
                } else if (s >= r0 && own) {
                    store_ps(s, n);
                }
            }
            if (inputs) {
                __syncwarp();
                for (; issued < issued_after(k); ++issued) issue(issued);
            }
        }
        if (!ok && sums && lane == 0) {
            // a label never arrived (one that gives up does not): report it and
            // let the copies in flight land before the block's shared memory
            // goes; with two service warps the rows issued by then follow from
            // the step
            atomicExch(err, kErrWaitTimeout);
            const int n =
                min(!two ? issued : (k > 0 ? issued_after(k - 1) : kState), il + 1);
            for (int i = max(0, n - kAux); i < n; ++i)
                mbar_wait(b_full + 8 * (i & (kAux - 1)), (i / kAux) & 1);
        }
        return;
    }

    // ---- label warps -------------------------------------------------------
    const int l = wib;
    // 0/1 weights of the x differences (0 left of the grid, at the last
    // column and right of it)
    const float mxe = (c >= 0 && c < G.W - 1) ? 1.f : 0.f;
    const float mxo = (c + 1 >= 0 && c + 1 < G.W - 1) ? 1.f : 0.f;
    const float wxe = mxe * K.inv_a, wxo = mxo * K.inv_a;
    const unsigned char* const st_s = dsm + l * Seg<ES>::cols * ES + ES * (offs + 2 * lane);
    const unsigned char* const st_u =
        dsm + 3 * Y::fs + l * Seg<4>::cols * 4 + 4 * (off4 + 2 * lane);
    const unsigned char* const ax = dsm + Y::o_aux + 4 * (off4 + 2 * lane);
    const unsigned char* const axc = ax + l * Seg<4>::cols * 4;
    unsigned char* const sh = dsm + Y::o_sha + (l * 32 + lane) * (TILE && SIMPLE ? 16 : 8);
    const unsigned char* const psr = dsm + Y::o_ps + lane * 8;
    // the strip's last pair is a single column
    const bool odd_strip = cfirst + 63 >= G.W && (G.W & 1);

    auto f2 = [](const unsigned char* q) { return *reinterpret_cast<const float2*>(q); };
    auto sp = [](const unsigned char* q) {
        return *reinterpret_cast<const typename PS::T*>(q);
    };
    // 1 where row t has a y difference, else 0 (also above the grid)
    auto row_w = [&](int t) { return (unsigned)t < (unsigned)(G.H - 1) ? 1.f : 0.f; };
    // g = div q + p_i - p_s - u_i / c, given the row above's q_y and q_x at
    // the column to the left; wy: the row's weight
    auto g_of = [&](const Row<S>& x, float left, float2 p_s, typename PS::T qyu, float wy) {
        const float2 qx = PS::f2(x.qx);
        float2 g = make_float2(fmaf(mxe, qx.x, -left), fmaf(mxo, qx.y, -qx.x));
        g = fma2(PS::f2(x.qy), wy, g);
        g = sub2(g, PS::f2(qyu));
        g = add2(g, PS::f2(x.p));
        g = sub2(g, p_s);
        return fma2(x.u, -K.inv_c, g);
    };
    auto left_of = [&](float v) { return __shfl_up_sync(full_mask, v, 1); };
    auto right_of = [&](float v) { return __shfl_down_sync(full_mask, v, 1); };
    // new flows of a row (rounded) from its state and g at the row (gr: at
    // the column to the right) and the row below
    auto flows = [&](const Row<S>& x, float2 g, float gr, float2 gn, float2 al, float wy,
                     Row<S>& y) {
        const float2 qx = PS::f2(x.qx), qy = PS::f2(x.qy);
        const float my = wy * K.inv_a;
        float txe = fmaf(g.y - g.x, wxe, qx.x), txo = fmaf(gr - g.y, wxo, qx.y);
        float tye = fmaf(gn.x - g.x, my, qy.x), tyo = fmaf(gn.y - g.y, my, qy.y);
        project1<ANISO, false>(txe, tye, al.x);
        project1<ANISO, ES == 4 && !TILE>(txo, tyo, al.y);
        y.qx = PS::pk(txe, txo);
        y.qy = PS::pk(tye, tyo);
    };
    // the row's divergence, p_i^{k+1}, v_i and the label's share of the p_s
    // update (written to its slot); up: the new q_y of the row above (updated)
    auto finish = [&](const Row<S>& x, float2 p_s, float2 g, float txl, float2 cl, float wy,
                      float2& up, Row<S>& y, unsigned char* slot) {
        const float2 tx = PS::f2(y.qx), ty = PS::f2(y.qy);
        float2 d = make_float2(fmaf(mxe, tx.x, -txl), fmaf(mxo, tx.y, -tx.x));
        d = sub2(fma2(ty, wy, d), up);
        up = ty;
        const float2 p0 = PS::f2(x.p);
        float2 p1, share;
        if (SIMPLE) {
            const float2 e = sub2(p0, p_s);
            const float2 b = fma2(e, K.rho_p, mul2(x.u, -K.inv_c));
            const float2 rd = mul2(d, K.rho_p);
            share = TILE && fused ? fma2(d, K.rho_p, b) : add2(b, rd);
            p1 = fma2(share, -K.inv_a1, p0);
            y.p = PS::pk(fminf(p1.x, cl.x), fminf(p1.y, cl.y));
            p1 = PS::f2(y.p);
            const float2 h = fma2(e, -K.omr, p1);
            y.u = sub2(x.u, mul2(TILE && fused ? fma2(d, K.rho_p, h) : add2(h, rd), K.cu));
            if (TILE) {
                *reinterpret_cast<float4*>(slot) = make_float4(d.x, d.y, b.x, b.y);
                return;
            }
        } else {
            float sa = 0.f, sb = 0.f, ta = 0.f, tb = 0.f;
            p1.x = potts_label_pu<S>(K, g.x, d.x, p0.x, p_s.x, x.u.x, cl.x, sa, sb, y.u.x);
            p1.y = potts_label_pu<S>(K, g.y, d.y, p0.y, p_s.y, x.u.y, cl.y, ta, tb, y.u.y);
            y.p = PS::pk(p1.x, p1.y);
            share = make_float2(sa + sb, ta + tb);
        }
        *reinterpret_cast<float2*>(slot) = share;
    };
    auto load_row = [&](int slot, Row<S>& x) {
        const unsigned char* q = st_s + slot * Y::state;
        x.qx = sp(q);
        x.qy = sp(q + Y::fs);
        x.p = sp(q + 2 * Y::fs);
        x.u = f2(st_u + slot * Y::state);
    };
    // output: element index of the next row to store (the planes of all
    // labels hold less than 2^32 elements)
    uint32_t o = (uint32_t)l * (uint32_t)G.plane +
                 (uint32_t)((T == 2 ? js - 3 : js) * G.pitch + c);
    auto store_row = [&](const Row<S>& y, int t) {
        if (t >= r0 && own) {
            if (!odd_strip || pair) {
                *reinterpret_cast<typename PS::T*>(s1.qx + o) = y.qx;
                *reinterpret_cast<typename PS::T*>(s1.qy + o) = y.qy;
                *reinterpret_cast<typename PS::T*>(s1.p + o) = y.p;
                *reinterpret_cast<float2*>(s1.u + o) = y.u;
            } else {  // the last column alone
                St::st(s1.qx + o, PS::f2(y.qx).x);
                St::st(s1.qy + o, PS::f2(y.qy).x);
                St::st(s1.p + o, PS::f2(y.p).x);
                s1.u[o] = y.u.x;
            }
        }
        o += G.pitch;
    };

    // rows rf (its q_y only) and rf + 1
    Row<S> x[2], y[4];  // stage A's input rows j, j+1; its rows j .. j-3
    float2 ps[2], g[2];
    float2 qn_up = make_float2(0.f, 0.f);
    float2 gb = qn_up, qb_up = qn_up, psb = qn_up;  // stage B: g, p_s of row j-3
    float wya = 0.f, wyb = 0.f;                     // weights of rows j and j-3
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        y[i].qx = y[i].qy = y[i].p = PS::zero();
        y[i].u = qn_up;
    }
    ok = mbar_wait(b_full, 0) && mbar_wait(b_full + 8, 0);
    if (ok) {
        Row<S> xf;
        load_row(0, xf);
        load_row(1, x[0]);
        ps[0] = f2(ax + Y::aux + Y::f4);
        x[0].u = fma2(ps[0], cu_in, x[0].u);
        wya = row_w(js);
        g[0] = g_of(x[0], left_of(PS::f2(x[0].qx).y), ps[0], xf.qy, wya);
    }
    // One step, k = 8 n + U: every ring position is a constant; par = n & 1.
    auto body = [&](auto uc, int k, uint32_t par) -> bool {
        constexpr int U = decltype(uc)::value;
        constexpr int A = U & 1, B = A ^ 1;
        const int j = js + k;
        // aux slots of rows j + 1, j, j - 3
        constexpr int a1 = ((U + 2) & 7) * Y::aux, a0 = ((U + 1) & 7) * Y::aux,
                      ab = ((U + 6) & 7) * Y::aux;
        Row<S>&y2 = y[(U + 2) & 3], &y3 = y[(U + 1) & 3], &yn = y[U & 3];  // rows j-2, j-3, j
        if (label_waits_row(k, il))  // row j + 1 (the ones behind rl are made up and not used)
            if (!mbar_wait(b_full + 8 * ((U + 2) & 7), U < 6 ? par : par ^ 1)) return false;
        if (T == 2 && !mbar_wait(b_pr + 8 * (U & 3), U >> 2)) return false;
        if (T == 2) {
            // Stage B, before stage A: both at once take more than the 96
            // registers that 17 or 18 warps leave a thread.
            // p_s^{k+1} of row j-2 completes its u^{k+1} and g
            const float2 psn = f2(psr + ((U + 6) & 7) * 256);
            const float2 al = f2(ax + ab + Y::f4 + Y::f1), cl = f2(axc + ab);
            const float left = left_of(PS::f2(y2.qx).y);
            y2.u = fma2(psn, K.cu, y2.u);
            const float wyn = row_w(j - 2);
            const float2 gn = g_of(y2, left, psn, y3.qy, wyn);
            Row<S> z;
            flows(y3, gb, right_of(gb.x), gn, al, wyb, z);
            const float txl = left_of(PS::f2(z.qx).y);
            finish(y3, psb, gb, txl, cl, wyb, qb_up, z,
                   sh + (Y::o_shb - Y::o_sha) + ((U + 1) & 3) * Y::sh);
            gb = gn;
            psb = psn;
            wyb = wyn;
            store_row(z, j - 3);
        }
        load_row((U + 2) & (kState - 1), x[B]);
        ps[B] = f2(ax + a1 + Y::f4);
        const float2 al = f2(ax + a0 + Y::f4 + Y::f1), cl = f2(axc + a0);
        const float left = left_of(PS::f2(x[B].qx).y);
        x[B].u = fma2(ps[B], cu_in, x[B].u);
        const float wyn = row_w(j + 1);
        g[B] = g_of(x[B], left, ps[B], x[A].qy, wyn);
        flows(x[A], g[A], right_of(g[A].x), g[B], al, wya, yn);
        const float txl = left_of(PS::f2(yn.qx).y);
        finish(x[A], ps[A], g[A], txl, cl, wya, qn_up, yn, sh + (U & 3) * Y::sh);
        wya = wyn;
        __syncwarp();
        if (lane == 0) mbar_arrive(b_sf + 8 * (U & 3));
        if (T == 1) store_row(yn, j);
        return true;
    };
    if (ok) {
        uint32_t par = 0;
#pragma unroll 1
        for (int k = 0; k <= ke; k += 8, par ^= 1) {
#define CMF_STEP(U)                                                                  \
    if (k + U > ke || !(ok = body(std::integral_constant<int, U>(), k + U, par))) break
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

// One launch of the single-problem solver.
template <typename S, bool ANISO, bool SIMPLE, int T, int LC, bool TILE>
__global__ void __launch_bounds__(32 * (LC + rows::service_warps(T, LC)),
                                  LC == 4 ? 4 : (LC == 8 ? 2 : 1))
    k_potts_rows(const __grid_constant__ PottsRowsMaps M, PottsProblem P, PottsState<S> s1,
                 AdmmCoef K, float cu_in, int R, int nstrips, int fused, int* err) {
    const int r0 = (blockIdx.x / nstrips) * R;
    potts_rows_block<S, ANISO, SIMPLE, T, LC, TILE>(
        M, P, s1, K, cu_in, r0, min(r0 + R, P.g.H),
        (int)(blockIdx.x % nstrips) * (T == 2 ? 56 : 60) - (T == 2 ? 4 : 2), fused, err);
}

// ---- host side -------------------------------------------------------------

template <typename S, bool ANISO, bool SIMPLE, int T, int LC, bool TILE>
static cudaError_t launch_potts_rows(const PottsProblem& P, const PottsState<S>& b,
                                     const AdmmCoef& K, float cu_in, const PottsRowsMaps& M,
                                     int fused, int* err, cudaStream_t st) {
    auto kern = k_potts_rows<S, ANISO, SIMPLE, T, LC, TILE>;
    constexpr size_t dyn = rows::Layout<LC, (int)sizeof(S), TILE>::bytes;
    static std::atomic<long long> limit[kMaxDevices];
    cudaError_t e = raise_dyn_smem(limit, kern, dyn);
    if (e != cudaSuccess) return e;
    // blocks resident per device and label count
    static std::atomic<long long> memo[LC + 1][kMaxDevices];
    const int threads = 32 * (P.L + rows::service_warps(T, LC));
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
    constexpr int OUT = T == 2 ? 56 : 60;
    const int nstrips = (G.W + OUT - 1) / OUT;
    // band height: whole rounds of resident blocks, each costing its rows
    // plus the rows that fill and drain the pipeline (swept from 1 row up at
    // 128^2 to 2048^2, L = 2 to 16: within 2% of the best height throughout)
    constexpr int kFill = T == 2 ? 8 : 4;
    long long best = -1;
    int R = G.H;
    for (int rounds = 1; rounds <= 8; ++rounds) {
        long long bands = rounds * resident / nstrips;
        bands = bands < 1 ? 1 : (bands > G.H ? G.H : bands);
        const int r = (int)((G.H + bands - 1) / bands);
        const long long items = (long long)nstrips * ((G.H + r - 1) / r);
        const long long cost = (items + resident - 1) / resident * (r + kFill);
        if (best < 0 || cost < best) {
            best = cost;
            R = r;
        }
    }
    const int nitems = nstrips * ((G.H + R - 1) / R);
    kern<<<nitems, threads, dyn, st>>>(M, P, b, K, cu_in, R, nstrips, fused, err);
    return cudaGetLastError();
}

template <typename S, bool ANISO, bool SIMPLE, int T, bool TILE>
static cudaError_t potts_rows_lc(const PottsProblem& P, const PottsState<S>& b, const AdmmCoef& K,
                                 float cu_in, const PottsRowsMaps& M, int fused, int* err,
                                 cudaStream_t st) {
#define CMF_ROWS(LC) \
    launch_potts_rows<S, ANISO, SIMPLE, T, LC, TILE>(P, b, K, cu_in, M, fused, err, st)
    return P.L <= 4 ? CMF_ROWS(4) : (P.L <= 8 ? CMF_ROWS(8) : CMF_ROWS(rows::kMaxLabels));
#undef CMF_ROWS
}

template <typename S, bool SIMPLE, bool TILE>
static cudaError_t potts_rows_step_s(const PottsProblem& P, const PottsStateV& b, bool aniso,
                                     const AdmmCoef& K, float cu_in, int iters,
                                     const PottsRowsMaps& M, int fused, int* err,
                                     cudaStream_t st) {
    const PottsState<S> B = b.as<S>();
#define CMF_ROWS(AN, IT) \
    potts_rows_lc<S, AN, SIMPLE, IT, TILE>(P, B, K, cu_in, M, fused, err, st)
    if (iters == 2) return aniso ? CMF_ROWS(true, 2) : CMF_ROWS(false, 2);
    return aniso ? CMF_ROWS(true, 1) : CMF_ROWS(false, 1);
#undef CMF_ROWS
}

}  // namespace cmf
