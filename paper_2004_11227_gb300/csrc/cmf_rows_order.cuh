// Which input rows are issued when, and who waits for whom, in the kernels that
// couple warps by mbarriers with the labels side by side (cmf_potts_rows.cuh,
// cmf_potts_cert.cuh): apart from the arithmetic and free of device code, so that
// a host test can replay the order of events for any schedule of the warps.
//
// A wait on an mbarrier tells phases apart by parity alone: a warp that comes to
// a wait two phases late finds the parity it does not wait for, and waits out the
// limit.  So whoever waits for a barrier's phase has to be one whom the next phase
// but one cannot do without.
#pragma once

#ifdef __CUDACC__
#define CMF_ORDER __host__ __device__ constexpr
#else
#define CMF_ORDER constexpr
#endif

namespace cmf {
namespace rows {

constexpr int kState = 4;  // state rows in shared memory
constexpr int kAux = 8;    // cost / p_s / alpha rows in shared memory
constexpr int kSh = 4;     // share slots of each stage
constexpr int kPs = 8;     // p_s^{k+1} rows

// Service warps of a block: two iterations per launch and many labels keep
// one warp busy with the label sums alone.
CMF_ORDER int service_warps(int T, int LC) { return T == 2 && LC > 4 ? 2 : 1; }
// Input rows issued once every label is done with step k: row k + 2 is in the
// labels' registers, so its state slot is free for the last of them.
CMF_ORDER int issued_after(int k) { return k + 3 + kState; }
// Whether a label waits for an input row (k + 2) at step k; il: the last row.
CMF_ORDER bool label_waits_row(int k, int il) { return k + 2 <= il; }
// The last step of the labels that a service warp without the sums waits for: the
// one behind which it issues its last row.  From then on no label waits for it, and
// if it came late it would find the barriers of later steps used again.
CMF_ORDER int last_input_step(int il) { return il > 2 + kState ? il - 2 - kState : 0; }

}  // namespace rows

namespace cert {

constexpr int kRing = 8;  // rows of every kind in shared memory

// Warps that find the simplex thresholds, rows in turn.
CMF_ORDER int theta_warps(int LC) { return LC / 4; }
// A label waits before step k for the thresholds of rows thresholds_from(k) to
// k + 1: of row 0 too, which it does not use, for row kRing is issued into row 0's
// slot when every label is done with step 0, and the warp that finds row 0's
// thresholds has to have read that row by then.
CMF_ORDER int thresholds_from(int k) { return k == 0 ? 0 : k + 1; }

}  // namespace cert
}  // namespace cmf
