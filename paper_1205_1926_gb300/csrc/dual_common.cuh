// Device helpers for the orthonormal constraint matrix B (Sec. 4.1) acting
// between multiplier space and the interface copy slots of the subdomains.
#pragma once
#include "dev.h"

namespace tfeti {

// Adds the entries of a B^T row after its first one (copies shared by more than two subdomains).
__device__ __forceinline__ double bt_rest(const DevMesh& M, const double* __restrict__ x, int row, int rest, double s) {
  const int r0 = (rest >> 8) & 0xff, j = rest & 0xff;
  for (int r = r0 + 1; r < (rest >> 16); ++r) s += __ldg(M.helm + r * 8 + j) * x[row + r - r0];
  return s;
}

// (B^T x) at U copy slots at once (slot < 0 gives 0): the slots' records, then their first entries'
// gathers, so that the U chains of dependent loads overlap.
template <int U>
__device__ __forceinline__ void bt_at_slots(const DevMesh& M, const double* __restrict__ x, const long long* slot,
                                            double* out) {
  int4 rec[U];   // SlotRow
#pragma unroll
  for (int k = 0; k < U; ++k)
    rec[k] = slot[k] >= 0 ? __ldg(reinterpret_cast<const int4*>(M.slot_row + slot[k])) : make_int4(-1, 0, 0, 0);
  double xv[U];
#pragma unroll
  for (int k = 0; k < U; ++k) xv[k] = rec[k].x >= 0 ? x[rec[k].x] : 0.0;
#pragma unroll
  for (int k = 0; k < U; ++k)
    out[k] = bt_rest(M, x, rec[k].x, rec[k].y, __hiloint2double(rec[k].w, rec[k].z) * xv[k]);
}

__device__ __forceinline__ double bt_at_slot(const DevMesh& M, const double* __restrict__ x, long long slot) {
  double v;
  bt_at_slots<1>(M, x, &slot, &v);
  return v;
}

// (B v)[row] for copy-slot values v.
__device__ __forceinline__ double b_at_row(const DevMesh& M, const double* __restrict__ v, long long row) {
  const int4 q = __ldg(reinterpret_cast<const int4*>(M.row_slots + row));   // RowSlots
  const double v0 = v[q.x];
  if (q.y < 0) return v0;
  double s = __ldg(M.helm + q.z * 8) * v0 + __ldg(M.helm + q.z * 8 + 1) * v[q.y];
  for (int j = 2; j <= q.z; ++j) s += M.helm[q.z * 8 + j] * v[M.groups[q.w].slot[j]];
  return s;
}

// Scalar logic of the inner PCGP (state in sc, see PcgScalar): pre -- after y.w of the
// iteration: the finiteness and stop tests; mid -- after p.Fp: the breakdown test; post -- at the
// end of a body run: the counters and the done flag; returns whether another body run follows.
__device__ __forceinline__ void pcg_pre_logic(double* sc) {
  if (sc[kDone] != 0.0) return;
  const double ww = sc[kWW], yw = sc[kYW];
  sc[kLastWW] = ww;
  if (!isfinite(ww) || !isfinite(yw)) {
    sc[kDone] = 1.0;
    sc[kStatus] = 8.0;
    return;
  }
  if (sc[kFirst] != 0.0 && !(ww > 0.0)) {   // w^0 = 0: nothing to do
    sc[kDone] = 1.0;
    sc[kStopAfter] = 1.0;
    return;
  }
  sc[kStopAfter] = ww <= sc[kTol2] ? 1.0 : 0.0;
}

__device__ __forceinline__ void pcg_mid_logic(double* sc) {
  if (sc[kDone] != 0.0) return;
  if (!(sc[kPFP] > 0.0)) {
    sc[kDone] = 1.0;
    sc[kStatus] = 7.0;
  }
}

// Closes one body run; returns whether the WHILE loop goes on.
__device__ __forceinline__ bool pcg_post_logic(double* sc) {
  sc[kBodyRuns] += 1.0;
  if (sc[kDone] == 0.0) {
    sc[kYWPrev] = sc[kYW];
    sc[kIter] += 1.0;
    sc[kFirst] = 0.0;
    if (sc[kStopAfter] != 0.0 || sc[kIter] >= sc[kMaxit]) sc[kDone] = 1.0;
  }
  return sc[kDone] == 0.0 && sc[kBodyRuns] < 2.0 * sc[kMaxit] + 4.0;
}

}  // namespace tfeti
