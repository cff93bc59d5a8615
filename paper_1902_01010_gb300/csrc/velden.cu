// Local velocity density f_l (Sec. 2.2): Epanechnikov estimate from the N_v nearest in
// velocity among the N_se nearest in position, inside each halo.
//
// GB300 design (no neighbour list is ever materialised):
//  - halo members are Morton-ordered inside their halo (halos.cu); each run of 32
//    consecutive members is a "bucket" with an integer bounding box, and 32 consecutive
//    buckets of one halo form a "super-bucket";
//  - one warp handles one bucket: lane k is the query particle k. Each lane first bounds
//    its N_se-th neighbour distance by the N_se-th smallest distance among the 4 N_se
//    members around the bucket in Morton order (to within one of 64 histogram bins);
//    every later pass visits only the buckets whose boxes come within the largest
//    per-lane bounds of the boxes of the warp's two parts (super-bucket boxes prune first),
//    and within some lane's bound of that lane;
//  - each visited bucket is staged once in shared memory and read back by every lane
//    with broadcast 16-byte loads; every lane keeps its own 64-bin histogram of the exact
//    key (d^2 << 22 | local index). Histogram passes narrow the key range until the bin
//    holding the N_se-th key has at most 32 keys; a last pass feeds every key below that
//    bin, plus the right number from the bin, into a per-lane list of the N_v smallest
//    |dv|^2 (shared memory);
//  - h^2 is the largest kept |dv|^2, and the kernel sum runs over the kept list only
//    (every neighbour with |dv| < h is in it).
// Position keys are exact integers, so the N_se set equals the oracle's; velocity
// differences and sums are FP32. Squared separations are 64-bit integers, or 32-bit ones
// wherever the two boxes involved (query bucket and candidate bucket or window) bound
// every separation by kNarrow lattice units per axis, which makes them exact in 32 bits.
//
// What bounds it: the issue slots (76 % taken at 7 warps a scheduler on a 256^3 box), by phase
// the window's bound 7 %, the histogram levels 38 %, the collect pass 42 % (most of it list
// insertions, whose lanes diverge), the keys of the final bin 13 %. Its code has to stay small:
// with every loop over 32 members unrolled whole, warps in different phases put each other's
// instructions out of the cache. k_velden_big over a 256^3 box (16.8 M particles, one launch):
// 30.3 ms, 55.6 with subtractions in 64 or 32 bits, a launch per size bin and bounds that stay
// what they were at the start of a level; over 1 M particles 2.73 ms, before 5.00.
// Halos with at most N_se members use every member (one pass, no position search).
#include <math.h>

#include <vector>

#include "boxparts.cuh"
#include "halos.cuh"
#include "tuning.cuh"
#include "vr_workspace.h"

namespace vr {

namespace {

constexpr int kNVMax = 64;
constexpr int kBinBits = 6;      // histogram levels resolve kBinBits bits of the key
constexpr int kBins = 1 << kBinBits;
constexpr int kBuf = 32;
// A bin's 16-bit count is held at kFull: above N_se + kBuf (1,024 + 32) its value no longer
// matters, and 16 buckets add at most 512 before it is looked at again.
constexpr int kFull = 32768;
// Lanes that want a bucket, up to which the collect pass takes it a lane per member and query by
// query (about 22 instructions a query) instead of a lane per query (about 300 for the 32 members).
// With it the f_l call of a 256^3 box took 33.3 ms, without 34.5. In the levels the counts would
// then need shared-memory atomics, so not there.
constexpr int kFewLanes = 12;
constexpr int kWarps = 4;        // warps per block

// Optional instrumentation (compile with -DVR_VELDEN_STATS): warp-level counts of the
// buckets staged per pass, kept in the status block's info[] words. Off in normal builds.
constexpr int kStatPass0 = 1;    // info[1 + pass]: 0 window, 1.. histogram levels, 7 collect
#ifdef VR_VELDEN_STATS
#define VR_STAT(st, slot, val) \
  do { if ((threadIdx.x & 31) == 0) atomicAdd((unsigned long long *)&(st)->info[(slot)], (unsigned long long)(val)); } while (0)
#else
#define VR_STAT(st, slot, val) do { } while (0)
#endif
constexpr int kWindow = 4;       // window of kWindow * N_se members for the first bound

// Per-warp shared memory. The key histogram is used only by the bound and histogram
// passes and the top-N_v list only by the collect pass, so the two share storage and the
// slots of the final bin are in local memory: 6.3 KB a warp, so that registers, not this, limit
// the warps in flight. Counts have 16 bits, since 32 would leave room for fewer warps.
template <int NVM>
struct WarpSmem {
  int4 su[32];
  float4 sv[32];
  union {
    uint16_t hist[kBins + 2][32];  // keys below the bins, the bins, keys beyond them
    float top[NVM][32];
  };
  int4 blo[32], bhi[32];  // boxes of 32 candidate buckets
  int4 qlo[2], qhi[2];    // boxes of the query bucket's two parts
};

template <int NVM>
struct SmallSmem {
  float4 sv[32];
  float top[NVM][32];
};

// Per-lane list of the nv smallest values, kept as a binary max-heap in the lane's
// shared-memory column (top[0] is the largest kept value), with its size and maximum.
struct TopV {
  int c, im;
  float m;
};

// Offers v to the list: while fewer than nv values are kept, v is added (sifted up);
// after that v replaces the largest when it is smaller (sifted down from the root), so
// a replacement costs log2(nv) steps instead of a scan of all nv values.
__device__ __forceinline__ void top_insert(float (*top)[32], int lane, TopV &t, int nv, float v) {
  if (t.c < nv) {
    int i = t.c++;
    while (i > 0) {
      const int p = (i - 1) >> 1;
      const float pv = top[p][lane];
      if (pv >= v) break;
      top[i][lane] = pv;
      i = p;
    }
    top[i][lane] = v;
    t.m = top[0][lane];
  } else if (v < t.m) {
    int i = 0;
    for (;;) {
      const int l = 2 * i + 1;
      if (l >= nv) break;
      int ch = l;
      float cv = top[l][lane];
      if (l + 1 < nv) {
        const float rv = top[l + 1][lane];
        if (rv > cv) {
          ch = l + 1;
          cv = rv;
        }
      }
      if (cv <= v) break;
      top[i][lane] = cv;
      i = ch;
    }
    top[i][lane] = v;
    t.m = top[0][lane];
  }
}

// f_l from the kept list: h^2 = largest kept |dv|^2 (the N_v-th smallest);
// f_l = 15/(8 pi h^3) * sum_{|dv| < h} (1 - |dv|^2/h^2) / N_se_eff.
__device__ __forceinline__ float top_density(float (*top)[32], int lane, const TopV &t,
                                             int nse_eff) {
  float h2 = t.m;
  if (!(h2 > 0.0f)) return INFINITY;
  float inv = 1.0f / h2;
  float sum = 0.0f;
  for (int q = 0; q < t.c; ++q) {
    float x = top[q][lane];
    if (x < h2) sum += 1.0f - x * inv;
  }
  float h = sqrtf(h2);
  const float c = 15.0f / (8.0f * 3.14159265358979f);
  return c / (h2 * h) * sum / (float)nse_eff;
}

__device__ __forceinline__ float dv2f(float4 a, float4 b) {
  float dx = a.x - b.x, dy = a.y - b.y, dz = a.z - b.z;
  return dx * dx + dy * dy + dz * dz;
}

__device__ __forceinline__ long long d2i(int4 a, int4 b) {
  long long dx = a.x - b.x, dy = a.y - b.y, dz = a.z - b.z;
  return dx * dx + dy * dy + dz * dz;
}
// The 32-bit route. When the query box is at most kNarrow wide and every separation between a
// point of it and one of the candidates' box has all components within kNarrow, d^2 < 2^31
// and, with coordinates relative to the query box's corner o, |q|^2 < 2^31. Then d^2 =
// |c|^2 - 2 q.c + |q|^2 in 32-bit arithmetic (what wraps on the way wraps back, and d^2 -
// |q|^2 fits a signed word), so a candidate staged as (c, |c|^2) costs three multiply-adds,
// and |q|^2 goes into the thresholds.
constexpr int kNarrow = 26754;  // 3 kNarrow^2 < 2^31

struct Rel {  // a query's side
  uint32_t ax, ay, az;  // -2 (q - o)
  int q2;               // |q - o|^2
};
__device__ __forceinline__ Rel rel_query(int4 q, int4 o) {
  const uint32_t x = (uint32_t)(q.x - o.x), y = (uint32_t)(q.y - o.y), z = (uint32_t)(q.z - o.z);
  return Rel{0u - 2u * x, 0u - 2u * y, 0u - 2u * z, (int)(x * x + y * y + z * z)};
}
__device__ __forceinline__ int4 rel_member(int4 p, int4 o) {
  const uint32_t x = (uint32_t)(p.x - o.x), y = (uint32_t)(p.y - o.y), z = (uint32_t)(p.z - o.z);
  return make_int4((int)x, (int)y, (int)z, (int)(x * x + y * y + z * z));
}
// d^2 - |q - o|^2
__device__ __forceinline__ int rel_d2(const Rel &r, int4 c) {
  return (int)(r.ax * (uint32_t)c.x + (r.ay * (uint32_t)c.y + (r.az * (uint32_t)c.z + (uint32_t)c.w)));
}

// True when the query box A is at most kNarrow wide and every separation between a point of
// it and a point of box B has all components within kNarrow.
__device__ __forceinline__ bool fits32(int4 alo, int4 ahi, int4 blo, int4 bhi) {
  const int ex = max(ahi.x - min(alo.x, blo.x), bhi.x - alo.x),
            ey = max(ahi.y - min(alo.y, blo.y), bhi.y - alo.y),
            ez = max(ahi.z - min(alo.z, blo.z), bhi.z - alo.z);
  return max(ex, max(ey, ez)) <= kNarrow;
}

// A bound on d^2 for the 32-bit route, where d^2 < 2^31.
__device__ __forceinline__ int clamp31(u64 x) { return x > 0x7fffffffull ? 0x7fffffff : (int)x; }

// ---------------------------------------------------------------- small halos
// Halos of at most N_se members: every member is a neighbour. A warp takes 32 consecutive
// slots of [m0, m1), a lane per slot, and the halos they belong to one after the other: the
// halo's members are staged 32 at a time and offered to its lanes. The offers are a serial
// chain, so the work is cut by slots and not by halos: a warp per halo made the 8 x 256
// offers of a 256-member halo one after the other (660 to 680 us for a 32^3 box and for 1 M
// particles alike; now 115 and 151 us, and over a 256^3 box 1.07 -> 0.51 ms).
template <int NVM>
__global__ void __launch_bounds__(32 * kWarps) k_velden_small(
    const uint32_t *__restrict__ hoff, const uint32_t *__restrict__ hid, int64_t m0, int64_t m1,
    const float4 *__restrict__ v, int nse, int nv, float *__restrict__ f_l) {
  __shared__ SmallSmem<NVM> sm[kWarps];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t s0 = m0 + ((int64_t)blockIdx.x * kWarps + w) * 32;
  if (s0 >= m1) return;
  const int64_t k = s0 + lane;
  const uint32_t h = hid[k < m1 ? k : m1 - 1];
  unsigned todo = __ballot_sync(0xffffffffu, k < m1);
  float(*top)[32] = sm[w].top;
  while (todo) {
    const uint32_t hh = __shfl_sync(0xffffffffu, h, __ffs(todo) - 1);
    const bool mine = k < m1 && h == hh;
    todo &= ~__ballot_sync(0xffffffffu, mine);
    const uint32_t hs = hoff[hh], he = hoff[hh + 1];
    const int nh = (int)(he - hs);
    if (nh > nse) continue;
    const int nv_eff = nv < nh ? nv : nh;
    const float4 vq = v[mine ? k : hs];
    TopV t = {0, 0, 0.0f};
    for (uint32_t jb = hs; jb < he; jb += 32) {
      const uint32_t j = jb + lane;
      __syncwarp();
      if (j < he) sm[w].sv[lane] = v[j];
      __syncwarp();
      const int cnt = (int)min(32u, he - jb);
      if (mine)
        for (int tt = 0; tt < cnt; ++tt) top_insert(top, lane, t, nv_eff, dv2f(sm[w].sv[tt], vq));
    }
    if (mine) f_l[__float_as_int(vq.w)] = top_density(top, lane, t, nh);
  }
}

// ------------------------------------------------------------- bucket boxes
// Super-buckets are laid out halo by halo in the size order (largest first), so that the
// buckets of each halo-size bin form one contiguous range. Halo h owns super-buckets
// [sbs[h], sbe[h]); its bucket b (0-based) holds slots [hoff[h] + 32 b,
// min(hoff[h+1], hoff[h] + 32 b + 32)) and has the global index 32 sbs[h] + b.
__global__ void k_sb_count(const uint32_t *__restrict__ hoff, const uint32_t *__restrict__ horder,
                           int64_t H, int nse, uint32_t *__restrict__ sbr) {
  int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (r > H) return;
  if (r == H) {
    sbr[H] = 0;
    return;
  }
  const uint32_t h = horder[r];
  uint32_t nh = hoff[h + 1] - hoff[h];
  uint32_t nb = (nh + 31) / 32;
  sbr[r] = nh > (uint32_t)nse ? (nb + 31) / 32 : 0;
}

__global__ void k_sb_fill(const uint32_t *__restrict__ sbr, const uint32_t *__restrict__ horder,
                          int64_t H, uint32_t *__restrict__ sbs, uint32_t *__restrict__ sbe,
                          uint32_t *__restrict__ sbhalo) {
  int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= H) return;
  const uint32_t h = horder[r];
  sbs[h] = sbr[r];
  sbe[h] = sbr[r + 1];
  for (uint32_t s = sbr[r]; s < sbr[r + 1]; ++s) sbhalo[s] = h;
}

// First super-bucket of the halos of at most kVBinEdge0 and at most kVBinEdge1 members
// (sizes decrease along the order; the total when no halo is that small).
__global__ void k_bin_edges(const uint32_t *__restrict__ hoff, const uint32_t *__restrict__ horder,
                            const uint32_t *__restrict__ sbr, int64_t H, uint32_t *__restrict__ edges) {
  int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= H) return;
  const uint32_t hr = horder[r];
  const uint32_t nr = hoff[hr + 1] - hoff[hr];
  uint32_t np = 0xffffffffu;
  if (r > 0) {
    const uint32_t hp = horder[r - 1];
    np = hoff[hp + 1] - hoff[hp];
  }
  const uint32_t e[2] = {kVBinEdge0, kVBinEdge1};
  for (int k = 0; k < 2; ++k) {
    if (np > e[k] && nr <= e[k]) edges[k] = sbr[r];
    if (r == H - 1 && nr > e[k]) edges[k] = sbr[H];
  }
}

__global__ void k_bucket_boxes(const uint32_t *__restrict__ hoff, const uint32_t *__restrict__ sbs,
                               const uint32_t *__restrict__ sbhalo, int64_t nbpad,
                               const int4 *__restrict__ u, int4 *__restrict__ bmin,
                               int4 *__restrict__ bmax) {
  int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= nbpad) return;
  uint32_t h = sbhalo[b >> 5];
  uint32_t local = (uint32_t)b - 32u * sbs[h];
  uint32_t s0 = hoff[h] + 32u * local, s1 = min(s0 + 32u, hoff[h + 1]);
  int4 lo = make_int4(0x7fffffff, 0x7fffffff, 0x7fffffff, 0);
  int4 hi = make_int4(-0x7fffffff, -0x7fffffff, -0x7fffffff, 0);
  for (uint32_t m = s0; m < s1; ++m) {
    int4 p = u[m];
    lo.x = min(lo.x, p.x); lo.y = min(lo.y, p.y); lo.z = min(lo.z, p.z);
    hi.x = max(hi.x, p.x); hi.y = max(hi.y, p.y); hi.z = max(hi.z, p.z);
  }
  bmin[b] = lo;  // empty (padding) buckets keep an inverted box
  bmax[b] = hi;
}

__global__ void k_superbucket_boxes(int64_t nsb, const int4 *__restrict__ bmin,
                                    const int4 *__restrict__ bmax, int4 *__restrict__ smin,
                                    int4 *__restrict__ smax) {
  int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= nsb) return;
  int4 lo = make_int4(0x7fffffff, 0x7fffffff, 0x7fffffff, 0);
  int4 hi = make_int4(-0x7fffffff, -0x7fffffff, -0x7fffffff, 0);
  for (int k = 0; k < 32; ++k) {
    int4 a = bmin[32 * s + k], c = bmax[32 * s + k];
    lo.x = min(lo.x, a.x); lo.y = min(lo.y, a.y); lo.z = min(lo.z, a.z);
    hi.x = max(hi.x, c.x); hi.y = max(hi.y, c.y); hi.z = max(hi.z, c.z);
  }
  smin[s] = lo;
  smax[s] = hi;
}

__device__ __forceinline__ long long gap1(int alo, int ahi, int blo, int bhi) {
  long long g = 0;
  if (blo > ahi) g = (long long)blo - ahi;
  else if (alo > bhi) g = (long long)alo - bhi;
  return g;
}
__device__ __forceinline__ long long box_d2(int4 alo, int4 ahi, int4 blo, int4 bhi) {
  long long gx = gap1(alo.x, ahi.x, blo.x, bhi.x), gy = gap1(alo.y, ahi.y, blo.y, bhi.y),
            gz = gap1(alo.z, ahi.z, blo.z, bhi.z);
  return gx * gx + gy * gy + gz * gz;
}
__device__ __forceinline__ long long pt_box_d2(int4 p, int4 blo, int4 bhi) {
  return box_d2(p, p, blo, bhi);
}

__device__ __forceinline__ int bitlen64(unsigned long long x) { return x ? 64 - __clzll(x) : 0; }

// ---------------------------------------------------------------- big halos
// Launch shape (tuning.cuh): BATCH candidates computed side by side, at most MAXREG
// registers, any number of warps per block up to 8 (blockDim.x / 32).
template <int NVM, int BATCH, int MAXREG>
__global__ void __launch_bounds__(256) __maxnreg__(MAXREG) k_velden_big(
    const uint32_t *__restrict__ hoff, const uint32_t *__restrict__ sbs,
    const uint32_t *__restrict__ sbe, const uint32_t *__restrict__ sbhalo, int64_t b0,
    int64_t b1, const int4 *__restrict__ u,
    const float4 *__restrict__ v, const int4 *__restrict__ bmin, const int4 *__restrict__ bmax,
    const int4 *__restrict__ smin, const int4 *__restrict__ smax, int nse, int nv,
    float *__restrict__ f_l, DevStatus *st) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  WarpSmem<NVM> &sm = reinterpret_cast<WarpSmem<NVM> *>(smem_raw)[threadIdx.x >> 5];
  const int lane = threadIdx.x & 31;
  const unsigned FULL = 0xffffffffu;
  const int64_t b = b0 + (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);  // buckets [b0, b1)
  if (b >= b1) return;
  const uint32_t h = sbhalo[b >> 5];
  const uint32_t hs = hoff[h], he = hoff[h + 1];
  const uint32_t nh = he - hs;
  const uint32_t sb0 = sbs[h], sb1 = sbe[h];
  const uint32_t local = (uint32_t)b - 32u * sb0;
  const uint32_t nbh = (nh + 31) / 32;
  if (local >= nbh) return;  // padding bucket
  const uint32_t qs = hs + 32u * local, qe = min(qs + 32u, he);
  const uint32_t k = qs + lane;
  const bool valid = k < qe;
  const int4 q = u[valid ? k : qs];
  const float4 vq = v[valid ? k : qs];
  const int nse_eff = nse;  // nh > nse here
  const int nv_eff = nv;
  int pass_id = 0;  // instrumentation only
  auto warp_max = [&](long long x) {
    for (int o = 16; o; o >>= 1) {
      long long y = __shfl_xor_sync(FULL, x, o);
      x = y > x ? y : x;
    }
    return x;
  };
  // stages slots [s0, s0 + cnt) in shared memory (positions; velocities if asked); the
  // remaining entries get a sentinel position far outside any bound (d^2 > 2^58), so the
  // candidate loops always run 32 fixed iterations
  // (`rel`: relative to the query box's corner, for the 32-bit route)
  const int4 qlo = bmin[b], qhi = bmax[b];
  const Rel rq = rel_query(q, qlo);
  auto stage = [&](uint32_t s0, int cnt, bool with_v, bool rel) {
    __syncwarp();
    if (rel) {  // beyond `cnt`: the last one again
      const uint32_t m = s0 + min(lane, cnt - 1);
      sm.su[lane] = rel_member(u[m], qlo);
      if (with_v) sm.sv[lane] = v[m];
    } else if (lane < cnt) {
      sm.su[lane] = u[s0 + lane];
      if (with_v) sm.sv[lane] = v[s0 + lane];
    } else {
      sm.su[lane] = make_int4(0x3fffffff, 0x3fffffff, 0x3fffffff, 0);
    }
    __syncwarp();
    VR_STAT(st, kStatPass0 + pass_id, 1);
  };
  // 1. bound from the window of kWindow * N_se members around the bucket: the N_se-th
  //    smallest distance among them, rounded up to a histogram bin edge. When the window's
  //    box and the bucket's box bound every separation by kNarrow per axis (a warp-uniform
  //    test), the distances are exact in 32-bit arithmetic.
  long long r2 = 0;
  {
    const int W = (int)min((uint32_t)(kWindow * nse), nh);
    int64_t w0 = (int64_t)qs + 16 - W / 2;
    if (w0 + W > (int64_t)he) w0 = (int64_t)he - W;
    if (w0 < (int64_t)hs) w0 = hs;
    int4 wlo = make_int4(0x7fffffff, 0x7fffffff, 0x7fffffff, 0);
    int4 whi = make_int4(-0x7fffffff, -0x7fffffff, -0x7fffffff, 0);
    for (int c = lane; c < W; c += 32) {
      const int4 pw = u[w0 + c];
      wlo.x = min(wlo.x, pw.x); wlo.y = min(wlo.y, pw.y); wlo.z = min(wlo.z, pw.z);
      whi.x = max(whi.x, pw.x); whi.y = max(whi.y, pw.y); whi.z = max(whi.z, pw.z);
    }
    for (int o = 16; o; o >>= 1) {
      wlo.x = min(wlo.x, __shfl_xor_sync(FULL, wlo.x, o));
      wlo.y = min(wlo.y, __shfl_xor_sync(FULL, wlo.y, o));
      wlo.z = min(wlo.z, __shfl_xor_sync(FULL, wlo.z, o));
      whi.x = max(whi.x, __shfl_xor_sync(FULL, whi.x, o));
      whi.y = max(whi.y, __shfl_xor_sync(FULL, whi.y, o));
      whi.z = max(whi.z, __shfl_xor_sync(FULL, whi.z, o));
    }
    const bool wn = fits32(qlo, qhi, wlo, whi);  // warp-uniform
    long long wmax = 0;
    int wmax32 = -0x7fffffff;  // of d^2 - |q - o|^2
    for (int c = 0; c < W; c += 32) {
      const int cnt = min(32, W - c);
      stage((uint32_t)(w0 + c), cnt, false, wn);
      if (wn) {
#pragma unroll 1
        for (int t0 = 0; t0 < 32; t0 += BATCH) {
#pragma unroll
          for (int j = 0; j < BATCH; ++j) wmax32 = max(wmax32, rel_d2(rq, sm.su[t0 + j]));
        }
      } else {
#pragma unroll 1
        for (int t0 = 0; t0 < 32; t0 += BATCH) {
          long long d[BATCH];
#pragma unroll
          for (int j = 0; j < BATCH; ++j) d[j] = d2i(q, sm.su[t0 + j]);
#pragma unroll
          for (int j = 0; j < BATCH; ++j) wmax = (t0 + j < cnt && d[j] > wmax) ? d[j] : wmax;
        }
      }
    }
    if (wn) wmax = (long long)wmax32 + rq.q2;
#pragma unroll 4
    for (int cb = 0; cb < kBins; ++cb) sm.hist[cb][lane] = 0;
    int sh0 = bitlen64((unsigned long long)wmax) - kBinBits;  // kBins bins over [0, 2^bitlen)
    if (sh0 < 0) sh0 = 0;
    for (int c = 0; c < W; c += 32) {
      const int cnt = min(32, W - c);
      stage((uint32_t)(w0 + c), cnt, false, wn);
      if (wn) {  // wmax < 2^31, so sh0 <= 25
        int d[BATCH];
#pragma unroll 1
        for (int t0 = 0; t0 < 32; t0 += BATCH) {
#pragma unroll
          for (int j = 0; j < BATCH; ++j) d[j] = rel_d2(rq, sm.su[t0 + j]) + rq.q2;
#pragma unroll
          for (int j = 0; j < BATCH; ++j) sm.hist[d[j] >> sh0][lane]++;
        }
        sm.hist[d[BATCH - 1] >> sh0][lane] -= 32 - cnt;  // the repeated last one
      } else {
#pragma unroll 1
        for (int t0 = 0; t0 < 32; t0 += BATCH) {
          long long d[BATCH];
#pragma unroll
          for (int j = 0; j < BATCH; ++j) d[j] = d2i(q, sm.su[t0 + j]);
#pragma unroll
          for (int j = 0; j < BATCH; ++j)
            if (t0 + j < cnt) sm.hist[(unsigned)(d[j] >> sh0)][lane]++;
        }
      }
    }
    int cum = 0, bs = kBins - 1;
#pragma unroll 4
    for (int cb = 0; cb < kBins; ++cb) {
      cum += sm.hist[cb][lane];
      if (cum >= nse_eff) {
        bs = cb;
        break;
      }
    }
    r2 = (((long long)bs + 1) << sh0) - 1;  // every distance in bins <= bs is <= r2
    if (r2 > wmax) r2 = wmax;
  }
  if (__any_sync(FULL, r2 >= (1LL << 41))) {  // all lanes leave, so that none waits for one that left
    if (r2 >= (1LL << 41)) raise_error(st, VR_ERR_UNSUPPORTED, 1);
    return;
  }
  // Two parts of the query bucket (a bucket whose box spanned a jump of the curve, in a halo of
  // 564 k members, tested 27,000 others one by one for 437 to visit: 25 M cycles; the longest warp
  // of any is 9 M cycles with two parts).
  const int cut = box_parts(q, (int)(qe - qs) - 1, qlo, qhi, sm.qlo, sm.qhi);
  __syncwarp();
  // Candidate buckets are enumerated on the fly in every pass: super-bucket boxes, then
  // bucket boxes, against the query bucket's box grown by the largest per-lane bound;
  // f(bucket index) is called warp-uniformly for every bucket that passes.
  // f(bucket index, this lane wants it, it fits the 32-bit route) returns true when it lowered
  // a lane's bound.
  auto for_each_bucket = [&](const long long &r2lane, auto &&f) {
    long long ra, rz;  // largest bounds in the query bucket's parts
    auto bounds = [&]() {
      ra = warp_max(lane <= cut ? r2lane : -1);
      rz = warp_max(lane <= cut ? -1 : r2lane);
    };
    auto reach = [&](int4 lo, int4 hi) {
      return box_d2(sm.qlo[0], sm.qhi[0], lo, hi) <= ra || box_d2(sm.qlo[1], sm.qhi[1], lo, hi) <= rz;
    };
    auto gap = [](int lo, int hi, int c) { return max(max(lo - c, c - hi), 0); };
    bounds();
    for (uint32_t sbase = sb0; sbase < sb1; sbase += 32) {
      uint32_t sx = sbase + lane;
      bool hit = sx < sb1 && reach(smin[sx], smax[sx]);
      unsigned hm = __ballot_sync(FULL, hit);
      while (hm) {
        int t = __ffs(hm) - 1;
        hm &= hm - 1;
        const uint32_t bb = 32u * (sbase + t) + lane;
        bool in = false, near = false;
        if (bb - 32u * sb0 < nbh) {
          const int4 lo = bmin[bb], hi = bmax[bb];
          in = reach(lo, hi);
          near = fits32(qlo, qhi, lo, hi);
          sm.blo[lane] = lo;
          sm.bhi[lane] = hi;
        }
        unsigned bm = __ballot_sync(FULL, in);
        const unsigned nm = __ballot_sync(FULL, near);
        __syncwarp();
        while (bm) {
          const int tb = __ffs(bm) - 1;
          bm &= bm - 1;
          const bool fits = (nm >> tb) & 1u;
          const int4 lo = sm.blo[tb], hi = sm.bhi[tb];
          bool want;
          if (fits) {
            const int ax = gap(lo.x, hi.x, q.x), ay = gap(lo.y, hi.y, q.y), az = gap(lo.z, hi.z, q.z);
            want = ax * ax + ay * ay + az * az <= (r2lane < 0 ? -1 : clamp31((u64)r2lane));
          } else {
            want = pt_box_d2(q, lo, hi) <= r2lane;
          }
          if (__any_sync(FULL, want) && f(32u * (sbase + t) + (uint32_t)tb, want, fits)) bounds();
        }
        __syncwarp();
      }
    }
  };
  // 2. histogram passes over the exact keys (d^2 << 22 | local index). The first level
  //    spreads its bins over [r2/4, r2] only (the N_se-th key lies near the bound) and
  //    counts the keys below in one register; later levels split the chosen bin.
  u64 klo = (u64)(r2 >> 2) << 22;
  int sh = bitlen64((((u64)(r2 + 1)) << 22) - klo - 1) - kBinBits;
  if (sh < 0) sh = 0;
  int need = nse_eff;
  bool settled = !valid;
  u64 fin_lo = 0, fin_hi = 0;
  int need_in = 0;
  long long rcur = r2;  // per-lane bound on d^2 of keys still of interest
  bool focus = true;    // this lane's current level is the focused first level
  for (int level = 0; level < 16; ++level) {
    pass_id = level < 5 ? 1 + level : 5;
    int below = 0, visits = 0;
    long long rlev = settled ? -1 : rcur;  // bound on d^2 of the keys that this level has to count
    if (!settled)
#pragma unroll 4
      for (int c = 0; c < kBins + 2; ++c) sm.hist[c][lane] = 0;
    for_each_bucket(rlev, [&](uint32_t bb, bool want, bool fits) {
      const uint32_t s0 = hs + 32u * (bb - 32u * sb0);
      const int cnt = (int)min(32u, he - s0);
      // 32-bit route: the boxes are near enough and the bins of every lane are whole units of
      // d^2, so a key's bin depends on d^2 alone (klo is a multiple of 2^22): bin =
      // (d^2 - (klo >> 22)) >> (sh - 22), and its row one more (65 << (sh - 22) fits 31 bits)
      const bool narrow = fits && __all_sync(FULL, !want || (sh >= 22 && sh < 47 && (klo & 0x3fffffull) == 0));
      stage(s0, cnt, false, narrow);
      if (narrow) {
        // without a branch per member: what lies below the bins or beyond the bound (all of it
        // for a lane that wants none) counts in a row of its own
        const int far = (want ? clamp31((u64)rlev) : -1) - rq.q2, shd = want ? sh - 22 : 0;
        const uint32_t off = (uint32_t)rq.q2 - (uint32_t)clamp31(klo >> 22) + (1u << shd);
        auto row_of = [&](int x) { return x > far ? kBins + 1 : max((int)((uint32_t)x + off) >> shd, 0); };
        int d[BATCH];
#pragma unroll 1
        for (int t0 = 0; t0 < 32; t0 += BATCH) {
#pragma unroll
          for (int j = 0; j < BATCH; ++j) d[j] = rel_d2(rq, sm.su[t0 + j]);
#pragma unroll
          for (int j = 0; j < BATCH; ++j) sm.hist[row_of(d[j])][lane]++;
        }
        sm.hist[row_of(d[BATCH - 1])][lane] -= 32 - cnt;  // the repeated last one
      } else if (want) {
#pragma unroll 1
        for (int t0 = 0; t0 < 32; t0 += BATCH) {
          long long d[BATCH];
#pragma unroll
          for (int j = 0; j < BATCH; ++j) d[j] = d2i(q, sm.su[t0 + j]);
#pragma unroll
          for (int j = 0; j < BATCH; ++j) {
            if (d[j] <= rlev) {
              u64 key = ((u64)d[j] << 22) | (u64)sm.su[t0 + j].w;
              if (key >= klo) {
                u64 rel = (key - klo) >> sh;
                if (rel < kBins) sm.hist[1 + rel][lane]++;
              } else if (focus) {
                ++below;
              }
            }
          }
        }
      }
      // Every 16 buckets: the bins counted so far bound the N_se-th key already, and nothing beyond
      // the bin that reaches it matters. The count of that bin is held at kFull, since the buckets
      // to come may hold more of its keys than 16 bits count (a halo has up to 2^22 members, and
      // coincident ones all fall in one bin); the rows before it hold fewer than N_se in all.
      if (++visits & 15) return false;
      if (rlev >= 0) {
        int cum = below + (int)sm.hist[0][lane];
        if (!focus) cum = 0;
        if (cum >= need) {
          rlev = -1;  // it lies below the focused range: nothing more to count here
        } else {
#pragma unroll 4
          for (int c = 0; c < kBins; ++c) {
            const int hc = sm.hist[1 + c][lane];
            cum += hc;
            if (cum >= need) {
              if (hc > kFull) sm.hist[1 + c][lane] = (uint16_t)kFull;
              const long long top_d = (long long)((klo + ((u64)(c + 1) << sh) - 1) >> 22);
              rlev = top_d < rlev ? top_d : rlev;
              break;
            }
          }
        }
      }
      return true;
    });
    if (!settled) {
      below += sm.hist[0][lane];
      if (focus && below >= need) {
        // the N_se-th key lies below the focused range: bin [0, klo) next
        const u64 hi = klo;
        klo = 0;
        sh = bitlen64(hi - 1) - kBinBits;
        if (sh < 0) sh = 0;
        const long long top_d = (long long)((hi - 1) >> 22);
        rcur = top_d < rcur ? top_d : rcur;
        focus = false;
      } else {
        if (focus) need -= below;  // every key below the focused range is in
        focus = false;
        int cum = 0, bs = kBins - 1;
#pragma unroll 4
        for (int c = 0; c < kBins; ++c) {
          int hc = sm.hist[1 + c][lane];
          if (cum + hc >= need) {
            bs = c;
            break;
          }
          cum += hc;
        }
        int hc = sm.hist[1 + bs][lane];
        if (hc <= kBuf || sh == 0) {
          fin_lo = klo + ((u64)bs << sh);
          fin_hi = fin_lo + ((u64)1 << sh);
          need_in = need - cum;
          settled = true;
        } else {
          klo += (u64)bs << sh;
          need -= cum;
          const long long top_d = (long long)((klo + ((u64)1 << sh) - 1) >> 22);
          rcur = top_d < rcur ? top_d : rcur;
          sh = sh >= kBinBits ? sh - kBinBits : 0;
        }
      }
    }
    if (__all_sync(FULL, settled)) break;
  }
  // 3. collect: keys below the final bin are in; the final bin is buffered
  if (valid) {
    const long long top_d = (long long)((fin_hi - 1) >> 22);
    rcur = top_d < r2 ? top_d : r2;
  } else {
    rcur = -1;
  }
  float(*top)[32] = sm.top;
  TopV tv = {0, 0, 0.0f};
  int nbuf = 0;
  uint32_t bslot[kBuf];  // member slots of the keys in the final bin (a few, in local memory)
  pass_id = 6;
  for_each_bucket(rcur, [&](uint32_t bb, bool want, bool fits) {
    const uint32_t s0 = hs + 32u * (bb - 32u * sb0);
    const int cnt = (int)min(32u, he - s0);
    // 32-bit route as in the histogram passes: with both final-bin edges multiples of
    // 2^22, key < edge iff d^2 < edge >> 22
    const bool narrow = fits && __all_sync(FULL, !want || ((fin_lo | fin_hi) & 0x3fffffull) == 0);
    stage(s0, cnt, true, narrow);
    uint32_t in = 0, fin = 0;  // members below the final bin, and in it
    const unsigned who = __ballot_sync(FULL, want);
    const bool few = __popc(who) <= kFewLanes;
    if (narrow) {
      const int none = -0x7fffffff - 1;
      const int flo = want ? clamp31(fin_lo >> 22) - rq.q2 : none,
                last = want ? min(clamp31((fin_hi >> 22) - 1), clamp31((u64)rcur)) - rq.q2 : none;
      if (few) {  // a lane per member, query by query
        const int4 c = sm.su[lane];
#pragma unroll 1
        for (unsigned w = who; w; w &= w - 1u) {
          const int l = __ffs(w) - 1;
          Rel o;
          o.ax = __shfl_sync(FULL, rq.ax, l);
          o.ay = __shfl_sync(FULL, rq.ay, l);
          o.az = __shfl_sync(FULL, rq.az, l);
          const int d = rel_d2(o, c), ofl = __shfl_sync(FULL, flo, l), ola = __shfl_sync(FULL, last, l);
          const unsigned bi = __ballot_sync(FULL, d < ofl), bf = __ballot_sync(FULL, d <= ola);
          in = lane == l ? bi : in;
          fin = lane == l ? bf : fin;
        }
      } else {
#pragma unroll 1
        for (int t0 = 0; t0 < 32; t0 += BATCH) {
          uint32_t bi = 0, bf = 0;
#pragma unroll
          for (int j = 0; j < BATCH; ++j) {
            const int d = rel_d2(rq, sm.su[t0 + j]);
            bi |= d < flo ? 1u << j : 0u;
            bf |= d <= last ? 1u << j : 0u;
          }
          in |= bi << t0;
          fin |= bf << t0;
        }
      }
    } else if (few) {
      const int4 c = sm.su[lane];
#pragma unroll 1
      for (unsigned w = who; w; w &= w - 1u) {
        const int l = __ffs(w) - 1;
        const int4 o = make_int4(__shfl_sync(FULL, q.x, l), __shfl_sync(FULL, q.y, l), __shfl_sync(FULL, q.z, l), 0);
        const long long d = d2i(o, c);
        const u64 key = ((u64)d << 22) | (u64)c.w, olo = __shfl_sync(FULL, fin_lo, l);
        const unsigned bi = __ballot_sync(FULL, key < olo);
        const u64 ohi = __shfl_sync(FULL, fin_hi, l);
        const long long orc = __shfl_sync(FULL, rcur, l);
        const unsigned bf = __ballot_sync(FULL, key < ohi && d <= orc);
        in = lane == l ? bi : in;
        fin = lane == l ? bf : fin;
      }
    } else if (want) {
#pragma unroll 1
      for (int t0 = 0; t0 < 32; t0 += BATCH) {
        uint32_t bi = 0, bf = 0;
#pragma unroll
        for (int j = 0; j < BATCH; ++j) {
          const int4 pc = sm.su[t0 + j];
          const long long d = d2i(q, pc);
          const u64 key = ((u64)d << 22) | (u64)pc.w;
          bi |= key < fin_lo ? 1u << j : 0u;
          bf |= key < fin_hi && d <= rcur ? 1u << j : 0u;
        }
        in |= bi << t0;
        fin |= bf << t0;
      }
    }
    if (cnt < 32) {
      in &= (1u << cnt) - 1u;
      fin &= (1u << cnt) - 1u;
    }
    fin &= ~in;
    for (; fin; fin &= fin - 1u)
      if (nbuf < kBuf) bslot[nbuf++] = s0 + (uint32_t)(__ffs(fin) - 1);
    // What the lists turn away already is passed over side by side first, where that is most of it:
    // of N_se members a list takes about N_v (1 + ln(N_se / N_v)). With N_se 256 and N_v 32 the f_l
    // call of a 256^3 box took 34.4 ms with this and 35.5 without; with 64 and 16, where the lists
    // take 60 %, that of a catalogue 24.4 and 24.1, so not there.
    if (nse_eff >= 6 * nv_eff && __reduce_max_sync(FULL, (unsigned)__popc(in)) > 10u) {
      uint32_t drop = 0;
#pragma unroll 1
      for (uint32_t some = __reduce_or_sync(FULL, in); some; some &= some - 1u) {
        const int k = __ffs(some) - 1;
        drop |= dv2f(sm.sv[k], vq) < tv.m ? 0u : 1u << k;
      }
      if (tv.c >= nv_eff) in &= ~drop;
    }
    // each lane its own next member: as many rounds as the lane with the most has
    for (; in; in &= in - 1u) top_insert(top, lane, tv, nv_eff, dv2f(sm.sv[__ffs(in) - 1], vq));
    return false;
  });
  if (!valid) return;
  // the need_in smallest keys of the final bin, in order
  if (need_in > 0) {
    u64 bkey[kBuf];
    for (int e = 0; e < nbuf; ++e) {
      const int4 pe = u[bslot[e]];
      bkey[e] = ((u64)d2i(q, pe) << 22) | (u64)pe.w;
    }
    for (int r = 0; r < min(need_in, nbuf); ++r) {
      int best = 0;
      u64 bk = bkey[0];
      for (int e = 1; e < nbuf; ++e) {
        const u64 x = bkey[e];
        if (x < bk) {
          bk = x;
          best = e;
        }
      }
      bkey[best] = ~0ULL;
      top_insert(top, lane, tv, nv_eff, dv2f(v[bslot[best]], vq));
    }
  }
  f_l[__float_as_int(vq.w)] = top_density(top, lane, tv, nse_eff);
}

__global__ void k_fill_f32(float *__restrict__ a, int64_t n, float val) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) a[i] = val;
}

}  // namespace

// Buckets with their padding: a halo of more than N_se members pads its buckets to a
// multiple of 32, at most 31 per such halo.
inline int64_t bucket_bound(int64_t n, int nse) { return n / 32 + 32 * (n / (nse + 1) + 2) + 64; }

size_t velden_bytes(int64_t n, int nmin, int nse) {
  Arena ar;
  int64_t hmax = n / (nmin > 0 ? nmin : 1) + 2;
  int64_t nbmax = bucket_bound(n, nse);
  ar.take<uint32_t>(hmax + 1);  // sbr
  ar.take<uint32_t>(hmax);      // sbs
  ar.take<uint32_t>(hmax);      // sbe
  ar.take<uint32_t>(4);         // bin edges
  ar.take<uint32_t>(nbmax / 32 + 1);  // sbhalo
  ar.take<int4>(nbmax);   // bmin
  ar.take<int4>(nbmax);   // bmax
  ar.take<int4>(nbmax / 32 + 1);  // smin
  ar.take<int4>(nbmax / 32 + 1);  // smax
  ar.take<char>(scan_scratch_bytes<uint32_t>(hmax + 1));
  return ar.off;
}

namespace {

// The f_l kernel instance for launch shape `shape` (tuning.cuh); N_v above 32 always uses
// the default shape.
template <int NVM>
void *big_kernel(int shape) {
  if (NVM > 32) return (void *)k_velden_big<NVM, 4, 64>;
  switch (kVShapes[shape].batch) {
    case 2: return (void *)k_velden_big<NVM, 2, 64>;
    case 8: return (void *)k_velden_big<NVM, 8, 80>;
    default: return (void *)k_velden_big<NVM, 4, 64>;
  }
}

}  // namespace

// Runs the f_l stage on an existing segmentation; f_l must already hold NaN outside
// halos.
vr_status run_velden(vr_ctx *ctx, const HaloSeg &g, const vr_params *p, Arena &ar, float *f_l,
                     cudaStream_t s, const uint32_t *hoff_host, cudaEvent_t ev_big) {
  if (g.H == 0) {
    if (ev_big) VR_CUDA(ctx, cudaEventRecord(ev_big, s));
    return VR_OK;
  }
  const int64_t H = g.H;
  int64_t hmax = g.n / (p->nmin > 0 ? p->nmin : 1) + 2;
  int64_t nbmax = bucket_bound(g.n, p->nse);
  uint32_t *sbr = ar.take<uint32_t>(hmax + 1);
  uint32_t *sbs = ar.take<uint32_t>(hmax);
  uint32_t *sbe = ar.take<uint32_t>(hmax);
  uint32_t *edges = ar.take<uint32_t>(4);
  uint32_t *sbhalo = ar.take<uint32_t>(nbmax / 32 + 1);
  int4 *bmin = ar.take<int4>(nbmax);
  int4 *bmax = ar.take<int4>(nbmax);
  int4 *smin = ar.take<int4>(nbmax / 32 + 1);
  int4 *smax = ar.take<int4>(nbmax / 32 + 1);
  void *scr = ar.take<char>(scan_scratch_bytes<uint32_t>(hmax + 1));
  if (!ar.ok()) return set_error(ctx, VR_ERR_WORKSPACE_TOO_SMALL, "workspace too small");
  const int T = 256;
  // small halos: all members are neighbours
  auto small = [&](int64_t a, int64_t z) {
    const int grid = grid_for(z - a, 32 * kWarps);
    if (p->nv <= 32)
      k_velden_small<32><<<grid, 32 * kWarps, 0, s>>>(g.hoff, g.hid, a, z, g.v, p->nse, p->nv, f_l);
    else
      k_velden_small<kNVMax><<<grid, 32 * kWarps, 0, s>>>(g.hoff, g.hid, a, z, g.v, p->nse, p->nv, f_l);
  };
  if (hoff_host) {  // one launch per halo
    for (int64_t h = 0; h < H; ++h) {
      if (hoff_host[h + 1] - hoff_host[h] > (uint32_t)p->nse) continue;
      small(hoff_host[h], hoff_host[h + 1]);
      VR_LAUNCHED(ctx, "k_velden_small");
    }
  } else {
    VR_TIMED(ctx, "velden_small", s, small(0, g.NHP));
    VR_LAUNCHED(ctx, "k_velden_small");
  }
  k_sb_count<<<grid_for(H + 1, T), T, 0, s>>>(g.hoff, g.horder, H, p->nse, sbr);
  VR_LAUNCHED(ctx, "k_sb_count");
  VR_CUDA(ctx, exclusive_scan<uint32_t>(sbr, sbr, H + 1, scr, s));
  k_bin_edges<<<grid_for(H, T), T, 0, s>>>(g.hoff, g.horder, sbr, H, edges);
  VR_LAUNCHED(ctx, "k_bin_edges");
  VR_CUDA(ctx, cudaMemcpyAsync(ctx->h_pinned + 34, sbr + H, sizeof(uint32_t),
                               cudaMemcpyDeviceToHost, s));
  VR_CUDA(ctx, cudaMemcpyAsync(ctx->h_pinned + 35, edges, 2 * sizeof(uint32_t),
                               cudaMemcpyDeviceToHost, s));
  VR_CUDA(ctx, cudaStreamSynchronize(s));
  uint32_t nsb = 0, eg[2] = {0, 0};
  memcpy(&nsb, ctx->h_pinned + 34, 4);
  memcpy(eg, ctx->h_pinned + 35, 8);
  if (nsb == 0) {
    if (ev_big) VR_CUDA(ctx, cudaEventRecord(ev_big, s));
    return VR_OK;
  }
  int64_t nbpad = 32LL * nsb;
  k_sb_fill<<<grid_for(H, T), T, 0, s>>>(sbr, g.horder, H, sbs, sbe, sbhalo);
  VR_LAUNCHED(ctx, "k_sb_fill");
  k_bucket_boxes<<<grid_for(nbpad, T), T, 0, s>>>(g.hoff, sbs, sbhalo, nbpad, g.u, bmin, bmax);
  VR_LAUNCHED(ctx, "k_bucket_boxes");
  k_superbucket_boxes<<<grid_for(nsb, T), T, 0, s>>>(nsb, bmin, bmax, smin, smax);
  VR_LAUNCHED(ctx, "k_superbucket_boxes");
  const size_t wsm = p->nv <= 32 ? sizeof(WarpSmem<32>) : sizeof(WarpSmem<kNVMax>);
  for (int sh = 0; sh < kNVShapes; ++sh) {
    void *kf = p->nv <= 32 ? big_kernel<32>(sh) : big_kernel<kNVMax>(sh);
    VR_CUDA(ctx, cudaFuncSetAttribute(kf, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(8 * wsm)));
  }
  // buckets [a, z) with launch shape `sh`
  auto big = [&](int sh, int64_t a, int64_t z) -> cudaError_t {
    const int w = p->nv <= 32 ? kVShapes[sh].warps : 4;
    void *kf = p->nv <= 32 ? big_kernel<32>(sh) : big_kernel<kNVMax>(sh);
    const int nse = p->nse, nv = p->nv;
    DevStatus *st = ctx->d_status;
    void *args[] = {(void *)&g.hoff, (void *)&sbs, (void *)&sbe, (void *)&sbhalo, (void *)&a,
                    (void *)&z, (void *)&g.u, (void *)&g.v, (void *)&bmin, (void *)&bmax,
                    (void *)&smin, (void *)&smax, (void *)&nse, (void *)&nv, (void *)&f_l,
                    (void *)&st};
    return cudaLaunchKernel(kf, dim3(grid_for(z - a, w)), dim3(32 * w), args, w * wsm, s);
  };
  if (hoff_host) {  // one launch per halo
    std::vector<uint32_t> s0(H), s1(H);
    VR_CUDA(ctx, cudaMemcpyAsync(s0.data(), sbs, H * sizeof(uint32_t), cudaMemcpyDeviceToHost, s));
    VR_CUDA(ctx, cudaMemcpyAsync(s1.data(), sbe, H * sizeof(uint32_t), cudaMemcpyDeviceToHost, s));
    VR_CUDA(ctx, cudaStreamSynchronize(s));
    for (int64_t h = 0; h < H; ++h) {
      if (s1[h] == s0[h]) continue;
      VR_CUDA(ctx, big(0, 32LL * s0[h], 32LL * s1[h]));
      VR_LAUNCHED(ctx, "k_velden_big");
    }
    return VR_OK;
  }
  // a shape per halo-size bin; a bin still to be tuned is run once per candidate shape (same
  // results each time) and keeps the fastest. Neighbouring bins of one shape share a launch,
  // so that the last, long warps of one run beside the next (alone, the launch of the largest
  // halos left a third of the chip's time idle), unless `ev_big` has to mark the end of the first
  // bin.
  const int64_t lo[kVBins] = {0, 32LL * eg[0], 32LL * eg[1]};
  const int64_t hi[kVBins] = {32LL * eg[0], 32LL * eg[1], nbpad};
  timer_begin(ctx, "velden_big", s);
  for (int k = 0; k < kVBins; ++k) {
    if (hi[k] <= lo[k]) {
      if (k == 0 && ev_big) VR_CUDA(ctx, cudaEventRecord(ev_big, s));
      continue;
    }
    if (p->nv <= 32 && vmeasure(ctx, k)) {
      Tuning *tn = ctx->tune;
      cudaEvent_t e0, e1;
      VR_CUDA(ctx, cudaEventCreate(&e0));
      VR_CUDA(ctx, cudaEventCreate(&e1));
      int best = 0;
      for (int sh = 0; sh < kNVShapes; ++sh) {
        VR_CUDA(ctx, cudaEventRecord(e0, s));
        VR_CUDA(ctx, big(sh, lo[k], hi[k]));
        VR_LAUNCHED(ctx, "k_velden_big");
        VR_CUDA(ctx, cudaEventRecord(e1, s));
        VR_CUDA(ctx, cudaEventSynchronize(e1));
        float ms = 0.f;
        VR_CUDA(ctx, cudaEventElapsedTime(&ms, e0, e1));
        tn->vms[k][sh] = ms;
        if (ms < tn->vms[k][best]) best = sh;
      }
      cudaEventDestroy(e0);
      cudaEventDestroy(e1);
      tn->vshape[k] = best;
      tn->vtuned[k] = 1;
    } else {
      const int sh = p->nv <= 32 ? vshape_for(ctx, k, nbpad) : 0;
      const int64_t first = lo[k];
      while (k + 1 < kVBins && !(k == 0 && ev_big) &&
             (p->nv > 32 || (!vmeasure(ctx, k + 1) && vshape_for(ctx, k + 1, nbpad) == sh)))
        ++k;
      for (int j = 0; j < kVBins; ++j)
        if (hi[j] > lo[j] && lo[j] >= first && hi[j] <= hi[k] && vshape_by_size(ctx, j)) ctx->vshape_last[j] = sh;
      VR_CUDA(ctx, big(sh, first, hi[k]));
      VR_LAUNCHED(ctx, "k_velden_big");
    }
    if (k == 0 && ev_big) VR_CUDA(ctx, cudaEventRecord(ev_big, s));  // halos > kVBinEdge0 done
  }
  timer_end(ctx, "velden_big", s);
  return VR_OK;
}

vr_status fill_f32(vr_ctx *ctx, float *a, int64_t n, float val, cudaStream_t s) {
  k_fill_f32<<<grid_for(n, 256), 256, 0, s>>>(a, n, val);
  VR_LAUNCHED(ctx, "k_fill_f32");
  return VR_OK;
}

}  // namespace vr
