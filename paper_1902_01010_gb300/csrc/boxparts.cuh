// Two boxes for 32 consecutive members of a curve. Where the curve jumps (Morton at octant
// edges; Hilbert too, on the cells that a flat or elongated halo occupies of its cube), the
// members lie in two clumps, and one box would reach everything between them.
#pragma once
#include "vr_internal.cuh"

namespace vr {

// One warp: lane k holds member q of a run whose members are lanes [0, last] (lanes beyond it
// repeat one of them); [lo, hi] is the run's box. Writes the boxes of the members up to a cut and
// beyond it, cut where the two volumes are least, each extent with an eighth of the box's largest
// added; returns the cut (0 for a single member, whose second part holds none). To be followed by
// __syncwarp() before plo / phi (shared memory) are read.
__device__ __forceinline__ int box_parts(int4 q, int last, int4 lo, int4 hi, int4 *plo, int4 *phi) {
  const unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  int4 alo = q, ahi = q, zlo = q, zhi = q;  // boxes of the members up to each lane, and from it on
  auto from = [&](int4 a, int src) {
    return make_int4(__shfl_sync(FULL, a.x, src), __shfl_sync(FULL, a.y, src), __shfl_sync(FULL, a.z, src), 0);
  };
  auto join = [](int4 &l, int4 &h, int4 ol, int4 oh) {
    l.x = min(l.x, ol.x); l.y = min(l.y, ol.y); l.z = min(l.z, ol.z);
    h.x = max(h.x, oh.x); h.y = max(h.y, oh.y); h.z = max(h.z, oh.z);
  };
  for (int o = 1; o < 32; o <<= 1) {
    const int4 al = from(alo, lane - o), ah = from(ahi, lane - o), zl = from(zlo, lane + o), zh = from(zhi, lane + o);
    if (lane >= o) join(alo, ahi, al, ah);
    if (lane + o <= last) join(zlo, zhi, zl, zh);
  }
  const float m = 0.125f * (float)max(hi.x - lo.x, max(hi.y - lo.y, hi.z - lo.z));
  auto vol = [&](int4 l, int4 h) {
    return ((float)(h.x - l.x) + m) * ((float)(h.y - l.y) + m) * ((float)(h.z - l.z) + m);
  };
  const int4 nlo = from(zlo, lane + 1), nhi = from(zhi, lane + 1);
  float best = lane < last ? vol(alo, ahi) + vol(nlo, nhi) : __int_as_float(0x7f800000);
  int at = lane;
  for (int o = 16; o; o >>= 1) {
    const float ob = __shfl_xor_sync(FULL, best, o);
    const int oa = __shfl_xor_sync(FULL, at, o);
    if (ob < best || (ob == best && oa < at)) {
      best = ob;
      at = oa;
    }
  }
  if (lane == at) {
    plo[0] = alo;
    phi[0] = ahi;
    plo[1] = last > 0 ? nlo : alo;
    phi[1] = last > 0 ? nhi : ahi;
  }
  return at;
}

}  // namespace vr
