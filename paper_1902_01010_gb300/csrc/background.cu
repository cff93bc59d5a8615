// Background velocity model and outlier ratio (Sec. 2.2).
//
//  k_halo_frame*  a warp, a block or a cluster of blocks per halo: FP64 mean velocity and
//                 dispersion tensor about it (divided by N_H), sigma_host = |Sigma|^(1/6),
//                 halo table row.
//  k_cells_*      a block or a cluster of blocks per searched halo: entropy kd-tree (Eq. S)
//                 down to cells of at most N_cell members, built node by node in global
//                 working arrays; split value = element floor(n/2) of the node in (coordinate,
//                 local index) order found by a radix select; FP64 cell moments (Eqs. meanpos,
//                 meanvel, meandispvel) per leaf.
//  k_ratio        one thread per member: own cell plus the cells across its six faces
//                 (point location by descending the tree), inverse-distance weights
//                 (Eq. cellinterp), FP64 Cholesky, ln f_bg (Eq. fvbg), R = ln f_l - ln f_bg.
// Readings of points the paper leaves open (fixed identically in the oracle): bins
// n_b = max(2, floor(n^(1/3))) over [min, max] with bin = (x - min) n_b / (max - min + 1);
// argmax S with ties within 1e-12 going to the lower axis; an axis whose split leaves
// the left side empty is skipped for the next-best one; regions are half-open boxes;
// a face neighbour is the leaf containing the member's position moved to lo - 1 (or hi)
// along that axis, skipped outside the root region and counted once.
#include <math.h>

#include <algorithm>
#include <vector>

#include <cooperative_groups.h>

#include "halos.cuh"
#include "vr_workspace.h"
#include "background.cuh"

namespace cg = cooperative_groups;

namespace vr {

namespace {

constexpr int kFrameT = 256;       // threads per halo-frame CTA
constexpr int kSmallT = 256;       // threads per tree-building CTA, halos below kMidHalo
constexpr int kBigT = 1024;        // threads per tree-building CTA, larger halos
constexpr int64_t kMidHalo = 8192, kBigHalo = 65536;
constexpr int kMaxBins = 162;      // floor((2^22)^(1/3)) + 1

__device__ __forceinline__ int64_t ncell_of(int64_t nh, double f_cell, int ncell_min) {
  int64_t nc = (int64_t)floor(__dmul_rn(f_cell, (double)nh));
  if (nc < ncell_min) {
    nc = ncell_min;
    if (nh / 8 < nc) nc = nh / 8;
  }
  return nc < 1 ? 1 : nc;
}

__device__ __forceinline__ int64_t icbrt_dev(int64_t n) {
  int64_t m = (int64_t)cbrt((double)n);
  while (m > 0 && m * m * m > n) --m;
  while ((m + 1) * (m + 1) * (m + 1) <= n) ++m;
  return m;
}

// ---- block reductions (256 threads) ----
template <int NT, class T, class Op>
__device__ __forceinline__ T block_reduce(T v, Op op, T *sbuf) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int o = 16; o; o >>= 1) v = op(v, __shfl_xor_sync(0xffffffffu, v, o));
  __syncthreads();
  if (lane == 0) sbuf[w] = v;
  __syncthreads();
  T r = sbuf[0];
  for (int k = 1; k < NT / 32; ++k) r = op(r, sbuf[k]);
  __syncthreads();
  return r;
}

struct MinOp { __device__ int operator()(int a, int b) const { return a < b ? a : b; } };
struct MaxOp { __device__ int operator()(int a, int b) const { return a > b ? a : b; } };
struct AddD { __device__ double operator()(double a, double b) const { return a + b; } };
struct AddF { __device__ float operator()(float a, float b) const { return a + b; } };

// Entropy bin floor(d nbins / ext) of a member d lattice units above its node's minimum (0 <=
// d < ext < 2^22, nbins <= 162): the quotient in FP32, put right where it is one off.
__device__ __forceinline__ int entropy_bin(int d, int64_t nbins, int ext) {
  const uint32_t x = (uint32_t)d * (uint32_t)nbins;  // below 2^30
  int q = (int)(__fdividef((float)x, (float)ext));
  const int r = (int)x - q * ext;
  if (r < 0) --q;
  if (r >= ext) ++q;
  return q;
}

__device__ __forceinline__ int coord(const int4 &p, int a) { return a == 0 ? p.x : (a == 1 ? p.y : p.z); }

}  // namespace

// Halo table row for every halo (searched or not): FP64 frame and sigma_host, by a team of
// kFrameTeam blocks of a cluster, one block, or one warp, by the halo's size. Both passes over
// the velocities and the reductions are FP64, of which an SM does two lanes a cycle: a halo
// of 500,000 members on one SM took 0.92 ms, and a block of 256 threads for every small halo
// spent 864 warp additions on its nine sums, where a warp spends 45 (200^3 box, all halos: one
// block each 1.20 ms, the three classes 0.14, 0.11 and 0.22).
constexpr int kFrameTeam = 8;
constexpr uint32_t kFrameBlock = 1024, kFrameBig = 16384;  // members from which a block, a cluster works

__device__ void frame_row(double *row, const double *mean, const double *S, uint32_t label, uint32_t nh,
                          int nsearch_min) {
  const double det = S[0] * (S[1] * S[2] - S[5] * S[5]) - S[3] * (S[3] * S[2] - S[5] * S[4]) +
                     S[4] * (S[3] * S[5] - S[1] * S[4]);
  row[VR_H_LABEL] = (double)label;
  row[VR_H_NH] = (double)nh;
  row[VR_H_SEARCHED] = nh >= (uint32_t)nsearch_min ? 1.0 : 0.0;
  row[VR_H_RBAR] = NAN;
  row[VR_H_SIGR] = NAN;
  row[VR_H_VFX] = mean[0];
  row[VR_H_VFY] = mean[1];
  row[VR_H_VFZ] = mean[2];
  row[VR_H_SIGMA] = det > 0.0 ? pow(det, 1.0 / 6.0) : 0.0;
  row[VR_H_LX2] = NAN;
  row[VR_H_LV2] = NAN;
  row[VR_H_NCELLS] = 0.0;
}

__device__ __forceinline__ double warp_add(double x) {
#pragma unroll
  for (int o = 16; o; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  return x;
}

// Sums of K values over the threads of a block, and of the cluster's blocks when TEAM > 1, to
// every thread. `sd` is the block's, one use per buffer.
template <int NT, int TEAM, int K>
__device__ __forceinline__ void team_add(double *x, double (*sd)[K], double *tot) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
  for (int k = 0; k < K; ++k) x[k] = warp_add(x[k]);
  if (lane == 0)
    for (int k = 0; k < K; ++k) sd[w][k] = x[k];
  __syncthreads();
  if (threadIdx.x < K) {
    double s = 0.0;
    for (int q = 0; q < NT / 32; ++q) s += sd[q][threadIdx.x];
    tot[threadIdx.x] = s;
  }
  if (TEAM > 1) cg::this_cluster().sync(); else __syncthreads();
#pragma unroll
  for (int k = 0; k < K; ++k) {
    if (TEAM > 1) {
      double s = 0.0;
      for (int q = 0; q < TEAM; ++q) s += cg::this_cluster().map_shared_rank(tot, q)[k];
      x[k] = s;
    } else {
      x[k] = tot[k];
    }
  }
}

template <int NT, int TEAM>
__device__ __forceinline__ void frame_team(int64_t h, int part, const uint32_t *__restrict__ hoff,
                                           const uint32_t *__restrict__ hlabel,
                                           const float4 *__restrict__ v, int nsearch_min,
                                           double *__restrict__ hs_out) {
  __shared__ double s_a[NT / 32][3], s_b[NT / 32][6], s_ta[3], s_tb[6];
  const uint32_t b = hoff[h], e = hoff[h + 1];
  const double nh = (double)(e - b);
  double s[3] = {0, 0, 0};
#pragma unroll 4
  for (uint32_t m = b + part * NT + threadIdx.x; m < e; m += NT * TEAM) {
    const float4 q = v[m];
    s[0] += (double)q.x;
    s[1] += (double)q.y;
    s[2] += (double)q.z;
  }
  team_add<NT, TEAM, 3>(s, s_a, s_ta);
  const double mean[3] = {s[0] / nh, s[1] / nh, s[2] / nh};
  double c[6] = {0, 0, 0, 0, 0, 0};
#pragma unroll 4
  for (uint32_t m = b + part * NT + threadIdx.x; m < e; m += NT * TEAM) {
    const float4 q = v[m];
    const double d0 = (double)q.x - mean[0], d1 = (double)q.y - mean[1], d2 = (double)q.z - mean[2];
    c[0] += d0 * d0; c[1] += d1 * d1; c[2] += d2 * d2;
    c[3] += d0 * d1; c[4] += d0 * d2; c[5] += d1 * d2;
  }
  team_add<NT, TEAM, 6>(c, s_b, s_tb);
  if (part == 0 && threadIdx.x == 0) {
    for (int k = 0; k < 6; ++k) c[k] /= nh;
    frame_row(hs_out + h * VR_HALO_COLS, mean, c, hlabel[h], e - b, nsearch_min);
  }
}

__global__ void __launch_bounds__(kFrameT) __cluster_dims__(kFrameTeam, 1, 1) k_halo_frame_big(
    const uint32_t *__restrict__ hoff, const uint32_t *__restrict__ hlabel,
    const uint32_t *__restrict__ horder, int64_t first, int64_t last, const float4 *__restrict__ v,
    int nsearch_min, double *__restrict__ hs_out) {
  const int64_t at = first + blockIdx.x / kFrameTeam;  // the same for the whole cluster
  if (at >= last) return;
  const int64_t h = horder[at];  // largest halos first
  if (hoff[h + 1] - hoff[h] < kFrameBig) return;  // each size class has its own launch
  frame_team<kFrameT, kFrameTeam>(h, (int)cg::this_cluster().block_rank(), hoff, hlabel, v, nsearch_min, hs_out);
  cg::this_cluster().sync();  // the others may still read this block's sums
}

__global__ void __launch_bounds__(kFrameT) k_halo_frame(
    const uint32_t *__restrict__ hoff, const uint32_t *__restrict__ hlabel,
    const uint32_t *__restrict__ horder, int64_t first, int64_t last, const float4 *__restrict__ v,
    int nsearch_min, double *__restrict__ hs_out) {
  if (first + (int64_t)blockIdx.x >= last) return;
  const int64_t h = horder[first + blockIdx.x];  // largest halos first
  const uint32_t nh = hoff[h + 1] - hoff[h];
  if (nh < kFrameBlock || nh >= kFrameBig) return;  // each size class has its own launch
  frame_team<kFrameT, 1>(h, 0, hoff, hlabel, v, nsearch_min, hs_out);
}

__global__ void __launch_bounds__(kFrameT) k_halo_frame_small(
    const uint32_t *__restrict__ hoff, const uint32_t *__restrict__ hlabel,
    const uint32_t *__restrict__ horder, int64_t first, int64_t last, const float4 *__restrict__ v,
    int nsearch_min, double *__restrict__ hs_out) {
  const int lane = threadIdx.x & 31;
  const int64_t at = first + (int64_t)blockIdx.x * (kFrameT / 32) + (threadIdx.x >> 5);
  if (at >= last) return;
  const int64_t h = horder[at];
  const uint32_t b = hoff[h], e = hoff[h + 1];
  if (e - b >= kFrameBlock) return;  // each size class has its own launch
  const double nh = (double)(e - b);
  double s[3] = {0, 0, 0};
  for (uint32_t m = b + lane; m < e; m += 32) {
    const float4 q = v[m];
    s[0] += (double)q.x;
    s[1] += (double)q.y;
    s[2] += (double)q.z;
  }
  double mean[3];
  for (int k = 0; k < 3; ++k) mean[k] = warp_add(s[k]) / nh;
  double c[6] = {0, 0, 0, 0, 0, 0};
  for (uint32_t m = b + lane; m < e; m += 32) {
    const float4 q = v[m];
    const double d0 = (double)q.x - mean[0], d1 = (double)q.y - mean[1], d2 = (double)q.z - mean[2];
    c[0] += d0 * d0; c[1] += d1 * d1; c[2] += d2 * d2;
    c[3] += d0 * d1; c[4] += d0 * d2; c[5] += d1 * d2;
  }
  for (int k = 0; k < 6; ++k) c[k] = warp_add(c[k]) / nh;
  if (lane == 0) frame_row(hs_out + h * VR_HALO_COLS, mean, c, hlabel[h], e - b, nsearch_min);
}

// Rows of the halos [a, z) of the size order, a launch per size class; the larger ones are its
// first entries, at most NHP / (their least size) of them.
static vr_status halo_frames(vr_ctx *ctx, const HaloSeg &g, int64_t a, int64_t z, int nsearch_min,
                             double *halo_stats, cudaStream_t s) {
  const int64_t zb = std::min(z, g.NHP / (int64_t)kFrameBig), zm = std::min(z, g.NHP / (int64_t)kFrameBlock);
  if (zb > a) {
    k_halo_frame_big<<<(unsigned)(kFrameTeam * (zb - a)), kFrameT, 0, s>>>(g.hoff, g.hlabel, g.horder, a, zb, g.v,
                                                                          nsearch_min, halo_stats);
    VR_LAUNCHED(ctx, "k_halo_frame_big");
  }
  if (zm > a) {
    k_halo_frame<<<(unsigned)(zm - a), kFrameT, 0, s>>>(g.hoff, g.hlabel, g.horder, a, zm, g.v, nsearch_min,
                                                       halo_stats);
    VR_LAUNCHED(ctx, "k_halo_frame");
  }
  k_halo_frame_small<<<grid_for(z - a, kFrameT / 32), kFrameT, 0, s>>>(g.hoff, g.hlabel, g.horder, a, z, g.v,
                                                                      nsearch_min, halo_stats);
  VR_LAUNCHED(ctx, "k_halo_frame_small");
  return VR_OK;
}

vr_status run_halo_frame(vr_ctx *ctx, const HaloSeg &g, int nsearch_min, double *halo_stats,
                         cudaStream_t s) {
  if (g.H == 0) return VR_OK;
  timer_begin(ctx, "halo_frame", s);
  const vr_status st = halo_frames(ctx, g, 0, g.H, nsearch_min, halo_stats, s);
  timer_end(ctx, "halo_frame", s);
  return st;
}

// Node-capacity bound per halo (node table slots), 0 for halos not searched.
__global__ void k_node_caps(const uint32_t *__restrict__ hoff, int64_t H, int nsearch_min,
                            double f_cell, int ncell_min, uint32_t *__restrict__ caps) {
  int64_t h = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (h > H) return;
  if (h == H) {
    caps[H] = 0;
    return;
  }
  int64_t nh = hoff[h + 1] - hoff[h];
  if (nh < nsearch_min) {
    caps[h] = 0;
    return;
  }
  int64_t nc = ncell_of(nh, f_cell, ncell_min);
  caps[h] = (uint32_t)(kNodeFactor * ((nh + nc) / (nc + 1)) + 16);
}

constexpr int kStackCap = 128;  // depth of a node stack
// Per-warp scratch of the tree build (dynamic shared memory, one per warp): axis
// histograms, the radix digit counts of a median selection and the warp's node stack.
struct WarpTree {
  int hist[3][kMaxBins];
  uint32_t dig[256];
  int stack[kStackCap];
};
constexpr int kPendCap = 256;  // nodes handed from the block to its warps

// The digit holding the need-th (1-based) key of a warp's 256 digit counts and the
// number of keys in the digits below it (warp-uniform).
__device__ __forceinline__ int warp_digit(const uint32_t *dig, int lane, uint32_t need,
                                          uint32_t *below) {
  uint32_t c[8], tot = 0;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    c[i] = dig[8 * lane + i];
    tot += c[i];
  }
  uint32_t inc = tot;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += y;
  }
  const unsigned m = __ballot_sync(0xffffffffu, inc >= need);
  const int L = m ? __ffs(m) - 1 : 31;
  uint32_t run = inc - tot, bel = run;
  int bin = 8 * lane + 7;
  bool done = false;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    if (!done && run + c[i] >= need) {
      bin = 8 * lane + i;
      bel = run;
      done = true;
    }
    run += c[i];
  }
  *below = __shfl_sync(0xffffffffu, bel, L);
  return __shfl_sync(0xffffffffu, bin, L);
}

// Axes with an extent by decreasing (split_rule 0) or increasing S, ties within 1e-12 to the
// lower axis; returns their number.
__device__ __forceinline__ int axis_order(const double *S, const bool *ok, int split_rule, int *order) {
  int no = 0;
  bool used[3] = {false, false, false};
  for (int r = 0; r < 3; ++r) {
    int best = -1;
    for (int a = 0; a < 3; ++a) {
      if (!ok[a] || used[a]) continue;
      if (best < 0) { best = a; continue; }
      if (split_rule == 0 ? (S[a] > S[best] + 1e-12) : (S[a] < S[best] - 1e-12)) best = a;
    }
    if (best < 0) break;
    used[best] = true;
    order[no++] = best;
  }
  return no;
}

// True when FP32 entropies may order two axes differently from FP64 ones: at most 162 terms
// f ln f, each within 3e-7 of its size, make S accurate to about 1e-5.
__device__ __forceinline__ bool close32(const double *S, const bool *ok) {
  return (ok[0] && ok[1] && fabs(S[0] - S[1]) < 1e-4) || (ok[0] && ok[2] && fabs(S[0] - S[2]) < 1e-4) ||
         (ok[1] && ok[2] && fabs(S[1] - S[2]) < 1e-4);
}

// Children of node `id` (split at xs along a, nleft members left); node numbers from the
// halo's counter. Returns the first child's number, or -1 with an error raised.
__device__ __forceinline__ int make_children(CellNode *nodes, uint32_t base, uint32_t cap, int id,
                                             int a, int xs, int nleft, int *counter, DevStatus *st) {
  CellNode *nd = &nodes[base + id];
  const int c0 = atomicAdd(counter, 2);
  if ((uint32_t)(c0 + 2) > cap) {
    raise_error(st, VR_ERR_UNSUPPORTED, 3);
    atomicSub(counter, 2);
    nd->axis = -1;
    return -1;
  }
  CellNode *L = &nodes[base + c0], *R = &nodes[base + c0 + 1];
  for (int k = 0; k < 3; ++k) {
    L->lo[k] = R->lo[k] = nd->lo[k];
    L->hi[k] = R->hi[k] = nd->hi[k];
  }
  L->hi[a] = xs;
  R->lo[a] = xs;
  L->beg = nd->beg;
  L->end = nd->beg + nleft;
  R->beg = nd->beg + nleft;
  R->end = nd->end;
  L->axis = R->axis = -1;
  nd->axis = a;
  nd->split = xs;
  nd->left = c0;
  nd->right = c0 + 1;
  return c0;
}

// Splits the subtree rooted at node `root` of one halo with a single warp, depth first:
// the same rules as the block path (entropy of n_b bins per axis, axis order by S with
// ties within 1e-12 to the lower axis, split at element floor(n/2) in (coordinate, local
// index) order, left = {x < split}, an axis leaving the left side empty skipped, stable
// partition), with warp shuffles and per-warp shared counts instead of block barriers.
// New nodes are numbered by an atomic counter; results do not depend on the numbering.
// The split value is the coordinate of element floor(n/2), so the selection needs the
// coordinates only, and the members below it are those the selection has passed over.
__device__ void warp_build(int root, uint32_t base, uint32_t cap, int64_t ncell, int split_rule,
                           const int4 *__restrict__ u, uint32_t *perm,
                           uint32_t *tmp, CellNode *nodes,
                           int *s_count, WarpTree &wt, DevStatus *st) {
  const int lane = threadIdx.x & 31;
  const unsigned FULL = 0xffffffffu, lt = (1u << lane) - 1u;
  int sp = 0;
  if (lane == 0) wt.stack[0] = root;
  sp = 1;
  __syncwarp();
  while (sp > 0) {
    const int id = wt.stack[--sp];
    __syncwarp();
    CellNode *nd = &nodes[base + id];
    const uint32_t nb_ = nd->beg, ne_ = nd->end;
    const int64_t n = ne_ - nb_;
    if (n <= ncell) {
      if (lane == 0) nd->axis = -1;
      continue;
    }
    int amin[3] = {0x7fffffff, 0x7fffffff, 0x7fffffff}, amax[3] = {-0x7fffffff, -0x7fffffff, -0x7fffffff};
#pragma unroll 4
    for (uint32_t i = nb_ + lane; i < ne_; i += 32) {
      const int4 p = u[perm[i]];
      amin[0] = min(amin[0], p.x); amin[1] = min(amin[1], p.y); amin[2] = min(amin[2], p.z);
      amax[0] = max(amax[0], p.x); amax[1] = max(amax[1], p.y); amax[2] = max(amax[2], p.z);
    }
    bool ok[3];
    for (int a = 0; a < 3; ++a) {
      amin[a] = __reduce_min_sync(FULL, amin[a]);
      amax[a] = __reduce_max_sync(FULL, amax[a]);
      ok[a] = amax[a] > amin[a];
    }
    const int64_t nbins = max((int64_t)2, icbrt_dev(n));
    for (int k = lane; k < 3 * kMaxBins; k += 32) (&wt.hist[0][0])[k] = 0;
    __syncwarp();
#pragma unroll 2
    for (uint32_t i = nb_ + lane; i < ne_; i += 32) {
      const int4 p = u[perm[i]];
      for (int a = 0; a < 3; ++a)
        if (ok[a]) atomicAdd(&wt.hist[a][entropy_bin(coord(p, a) - amin[a], nbins, amax[a] - amin[a] + 1)], 1);
    }
    __syncwarp();
    // Shannon entropy per axis (Eq. S); every lane ends with the same sums
    double S[3];
    const float inv_n = 1.0f / (float)n, inv_l = 1.0f / logf((float)nbins);
    for (int a = 0; a < 3; ++a) {
      float part = 0.0f;
      if (ok[a])
        for (int b = lane; b < nbins; b += 32) {
          const int c = wt.hist[a][b];
          if (c > 0) {
            const float f = (float)c * inv_n;
            part -= f * logf(f);
          }
        }
      for (int o = 16; o; o >>= 1) part += __shfl_xor_sync(FULL, part, o);
      S[a] = ok[a] ? (double)(part * inv_l) : 0.0;
    }
    if (close32(S, ok)) {
      for (int a = 0; a < 3; ++a) {
        double part = 0.0;
        if (ok[a])
          for (int b = lane; b < nbins; b += 32) {
            const int c = wt.hist[a][b];
            if (c > 0) {
              const double f = (double)c / (double)n;
              part -= f * log(f);
            }
          }
        for (int o = 16; o; o >>= 1) part += __shfl_xor_sync(FULL, part, o);
        S[a] = ok[a] ? part / log((double)nbins) : 0.0;
      }
    }
    int order[3];
    const int norder = axis_order(S, ok, split_rule, order);
    bool split_done = false;
    for (int r = 0; r < norder && !split_done; ++r) {
      const int a = order[r];
      const int lo_a = amin[a];
      // coordinate of rank floor(n/2) by 8-bit radix selection from the top digit
      const int bits = 32 - __clz(amax[a] - lo_a);
      uint32_t prefix = 0, rank = (uint32_t)(n / 2);
      for (int d = (bits + 7) / 8 - 1; d >= 0; --d) {
        const int sh = 8 * d;
        for (int k = lane; k < 256; k += 32) wt.dig[k] = 0u;
        __syncwarp();
#pragma unroll 4
        for (uint32_t i = nb_ + lane; i < ne_; i += 32) {
          const uint32_t key = (uint32_t)(coord(u[perm[i]], a) - lo_a);
          if ((key >> sh) >> 8 == (prefix >> sh) >> 8) atomicAdd(&wt.dig[(key >> sh) & 0xffu], 1u);
        }
        __syncwarp();
        uint32_t below;
        const int dg = warp_digit(wt.dig, lane, rank + 1u, &below);
        prefix |= (uint32_t)dg << sh;
        rank -= below;
        __syncwarp();
      }
      const int xs = lo_a + (int)prefix;
      const int nleft = (int)(n / 2) - (int)rank;  // rank: members at xs before element floor(n/2)
      if (nleft == 0) continue;  // left side empty: next axis
      // stable partition: chunks of 32 in the node's order, left block then right block
      uint32_t offl = 0, offr = 0;
      for (uint32_t cb = nb_; cb < ne_; cb += 32) {
        const uint32_t i = cb + lane;
        const bool okm = i < ne_;
        uint32_t pm = 0;
        bool isl = false;
        if (okm) {
          pm = perm[i];
          isl = coord(u[pm], a) < xs;
        }
        const unsigned bl = __ballot_sync(FULL, okm && isl);
        const unsigned br = __ballot_sync(FULL, okm && !isl);
        if (okm) {
          if (isl) tmp[nb_ + offl + __popc(bl & lt)] = pm;
          else tmp[nb_ + nleft + offr + __popc(br & lt)] = pm;
        }
        offl += __popc(bl);
        offr += __popc(br);
      }
      __syncwarp();
      for (uint32_t i = nb_ + lane; i < ne_; i += 32) perm[i] = tmp[i];
      __syncwarp();
      int c0 = 0;
      if (lane == 0) {
        if (sp + 2 <= kStackCap) {
          c0 = make_children(nodes, base, cap, id, a, xs, nleft, s_count, st);
        } else {
          raise_error(st, VR_ERR_UNSUPPORTED, 3);
          nd->axis = -1;
          c0 = -1;
        }
        if (c0 >= 0) {
          wt.stack[sp] = c0 + 1;
          wt.stack[sp + 1] = c0;
        }
      }
      c0 = __shfl_sync(FULL, c0, 0);
      if (c0 >= 0) sp += 2;
      __syncwarp();
      split_done = true;
    }
    if (!split_done && lane == 0) nd->axis = -1;
    __syncwarp();
  }
}

constexpr int kDigBits = 11;  // of a median selection by a block: coordinates in two passes
// Shared memory of a block of the tree build, besides the warps' scratch.
template <int NT>
struct BlockTree {
  int hist[3][kMaxBins];
  uint32_t dig[2][1 << kDigBits];  // by parity of the pass
  int ri[NT / 32];
  float rf[NT / 32];
  double rd[NT / 32];
  uint32_t scan[NT / 32];
  uint32_t wl[NT / 32], wr[NT / 32];
  int mm[2][6];      // extents of a node's members, by parity of the node
  int nl[2];         // members left of the split in this block's part, by parity
  int stack[64];     // nodes the block has yet to split
  int pend[kPendCap];
  int sp, npend, nleaves;
  uint32_t prefix, rank;
  int count;         // nodes of the halo (of the cluster: in its first block)
};

// One block, or the blocks of a cluster each with one part of every node's members: `part` of
// `parts`. A cluster adds up what its blocks counted through distributed shared memory.
template <int NT, int PARTS>
struct TreeTeam {
  BlockTree<NT> &s;
  int part;
  __device__ __forceinline__ void sync() const {
    if (PARTS > 1) cg::this_cluster().sync(); else __syncthreads();
  }
  template <class T>
  __device__ __forceinline__ T *of(T *p, int q) const {  // p of block q
    return PARTS > 1 ? cg::this_cluster().map_shared_rank(p, q) : p;
  }
};

// Splits node `id` (n members, more than ncell) with the whole team. Returns the first
// child's number (-1: none). `turn` alternates the buffers: a block reads the others' counts
// after one barrier, and writes to the same buffer again two barriers later at the earliest.
template <int NT, int PARTS>
__device__ int team_split(const TreeTeam<NT, PARTS> &tm, int id, uint32_t base, uint32_t cap, int split_rule,
                          const int4 *__restrict__ u, uint32_t *perm, uint32_t *tmp,
                          CellNode *nodes, int *counter, int &turn, int *child, DevStatus *st) {
  BlockTree<NT> &s = tm.s;
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  CellNode *nd = &nodes[base + id];
  const uint32_t nb_ = nd->beg, ne_ = nd->end;
  const int64_t n = ne_ - nb_;
  const uint32_t c0 = nb_ + (uint32_t)(n * tm.part / PARTS), c1 = nb_ + (uint32_t)(n * (tm.part + 1) / PARTS);
  // extent of the node's members per axis
  int amin[3], amax[3];
  {
    int mn[3] = {0x7fffffff, 0x7fffffff, 0x7fffffff}, mx[3] = {-0x7fffffff, -0x7fffffff, -0x7fffffff};
#pragma unroll 4
    for (uint32_t i = c0 + t; i < c1; i += NT) {
      const int4 p = u[perm[i]];
      mn[0] = min(mn[0], p.x); mn[1] = min(mn[1], p.y); mn[2] = min(mn[2], p.z);
      mx[0] = max(mx[0], p.x); mx[1] = max(mx[1], p.y); mx[2] = max(mx[2], p.z);
    }
    turn ^= 1;
    if (t < 6) s.mm[turn][t] = t < 3 ? 0x7fffffff : -0x7fffffff;
    for (int k = t; k < 3 * kMaxBins; k += NT) (&s.hist[0][0])[k] = 0;
    __syncthreads();
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const int l = __reduce_min_sync(0xffffffffu, mn[a]), h = __reduce_max_sync(0xffffffffu, mx[a]);
      if (lane == 0) {
        atomicMin(&s.mm[turn][a], l);
        atomicMax(&s.mm[turn][3 + a], h);
      }
    }
    tm.sync();
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      amin[a] = 0x7fffffff;
      amax[a] = -0x7fffffff;
      for (int q = 0; q < PARTS; ++q) {
        amin[a] = min(amin[a], tm.of(&s.mm[turn][a], q)[0]);
        amax[a] = max(amax[a], tm.of(&s.mm[turn][3 + a], q)[0]);
      }
    }
  }
  const bool ok[3] = {amax[0] > amin[0], amax[1] > amin[1], amax[2] > amin[2]};
  const int64_t nbins = max((int64_t)2, icbrt_dev(n));
#pragma unroll 4
  for (uint32_t i = c0 + t; i < c1; i += NT) {
    const int4 p = u[perm[i]];
#pragma unroll
    for (int a = 0; a < 3; ++a)
      if (ok[a]) atomicAdd(&s.hist[a][entropy_bin(coord(p, a) - amin[a], nbins, amax[a] - amin[a] + 1)], 1);
  }
  tm.sync();
  // Shannon entropy per axis (Eq. S): every thread sums the bins it owns, then a block
  // reduction; FP64 where FP32 leaves the order open
  double S[3];
  int cnt[3] = {0, 0, 0};  // this thread's bin (at most kMaxBins < NT of them)
#pragma unroll
  for (int a = 0; a < 3; ++a)
    if (ok[a] && t < nbins)
      for (int q = 0; q < PARTS; ++q) cnt[a] += tm.of(&s.hist[a][t], q)[0];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const float f = (float)cnt[a] / (float)n;
    const float part = block_reduce<NT>(cnt[a] > 0 ? -f * logf(f) : 0.0f, AddF(), s.rf);
    S[a] = ok[a] ? (double)(part / logf((float)nbins)) : 0.0;
  }
  if (close32(S, ok)) {
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const double f = (double)cnt[a] / (double)n;
      const double part = block_reduce<NT>(cnt[a] > 0 ? -(f * log(f)) : 0.0, AddD(), s.rd);
      S[a] = ok[a] ? part / log((double)nbins) : 0.0;
    }
  }
  int order[3];
  const int norder = axis_order(S, ok, split_rule, order);
  for (int r = 0; r < norder; ++r) {
    const int a = order[r];
    const int lo_a = amin[a];
    // coordinate of rank floor(n/2) by radix selection from the top digit
    const int bits = 32 - __clz(amax[a] - lo_a);
    uint32_t prefix = 0, rank = (uint32_t)(n / 2);
    for (int sh = (bits - 1) / kDigBits * kDigBits; sh >= 0; sh -= kDigBits) {
      turn ^= 1;
      uint32_t *dig = s.dig[turn];
      for (int k = t; k < (1 << kDigBits); k += NT) dig[k] = 0;
      __syncthreads();
#pragma unroll 4
      for (uint32_t i = c0 + t; i < c1; i += NT) {
        const uint32_t key = (uint32_t)(coord(u[perm[i]], a) - lo_a);
        if ((key >> sh) >> kDigBits == (prefix >> sh) >> kDigBits)
          atomicAdd(&dig[(key >> sh) & ((1u << kDigBits) - 1u)], 1u);
      }
      tm.sync();
      constexpr int kPer = (1 << kDigBits) / NT;  // digits of a thread
      uint32_t c[kPer], sum = 0;
#pragma unroll
      for (int q = 0; q < kPer; ++q) {
        c[q] = 0;
        for (int b = 0; b < PARTS; ++b) c[q] += tm.of(&dig[kPer * t + q], b)[0];
        sum += c[q];
      }
      uint32_t incl = sum;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t x = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += x;
      }
      if (lane == 31) s.scan[w] = incl;
      __syncthreads();
      for (int q = 0; q < w; ++q) incl += s.scan[q];
      uint32_t run = incl - sum;
#pragma unroll
      for (int q = 0; q < kPer; ++q) {
        if (run <= rank && rank < run + c[q]) {
          s.prefix = prefix | ((uint32_t)(kPer * t + q) << sh);
          s.rank = rank - run;
        }
        run += c[q];
      }
      __syncthreads();
      prefix = s.prefix;
      rank = s.rank;
      __syncthreads();
    }
    const int xs = lo_a + (int)prefix;
    const int nleft = (int)(n / 2) - (int)rank;  // rank: members at xs before element floor(n/2)
    if (nleft == 0) continue;  // left side empty: next axis
    // stable partition into tmp (left block, then right block, each in the node's order): per
    // chunk, every warp's ballot counts are scanned across the warps, so the member order,
    // and with it every later FP64 sum, does not depend on warp scheduling
    uint32_t offl = 0, offr = 0;
    if (PARTS > 1) {  // members left of the split in the parts before this one
      turn ^= 1;
      if (t == 0) s.nl[turn] = 0;
      __syncthreads();
      int cl = 0;
#pragma unroll 4
      for (uint32_t i = c0 + t; i < c1; i += NT) cl += coord(u[perm[i]], a) < xs ? 1 : 0;
      cl = __reduce_add_sync(0xffffffffu, cl);
      if (lane == 0) atomicAdd(&s.nl[turn], cl);
      tm.sync();
      for (int q = 0; q < tm.part; ++q) offl += (uint32_t)tm.of(&s.nl[turn], q)[0];
      offr = (c0 - nb_) - offl;
    }
    const unsigned lt = (1u << lane) - 1u;
    for (uint32_t cb = c0; cb < c1; cb += NT) {
      const uint32_t i = cb + t;
      const bool okm = i < c1;
      uint32_t pm = 0;
      bool isl = false;
      if (okm) {
        pm = perm[i];
        isl = coord(u[pm], a) < xs;
      }
      const unsigned bl = __ballot_sync(0xffffffffu, okm && isl);
      const unsigned br = __ballot_sync(0xffffffffu, okm && !isl);
      if (lane == 0) {
        s.wl[w] = (uint32_t)__popc(bl);
        s.wr[w] = (uint32_t)__popc(br);
      }
      __syncthreads();
      // inclusive scan of the per-warp counts, redone by every warp
      uint32_t xl = lane < NT / 32 ? s.wl[lane] : 0u, xr = lane < NT / 32 ? s.wr[lane] : 0u;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t yl = __shfl_up_sync(0xffffffffu, xl, o);
        const uint32_t yr = __shfl_up_sync(0xffffffffu, xr, o);
        if (lane >= o) {
          xl += yl;
          xr += yr;
        }
      }
      const uint32_t basel = offl + __shfl_sync(0xffffffffu, xl, w) - (uint32_t)__popc(bl);
      const uint32_t baser = offr + __shfl_sync(0xffffffffu, xr, w) - (uint32_t)__popc(br);
      offl += __shfl_sync(0xffffffffu, xl, 31);
      offr += __shfl_sync(0xffffffffu, xr, 31);
      if (okm) {
        if (isl) tmp[nb_ + basel + __popc(bl & lt)] = pm;
        else tmp[nb_ + nleft + baser + __popc(br & lt)] = pm;
      }
      __syncthreads();  // wl / wr are rewritten by the next chunk
    }
    tm.sync();
#pragma unroll 4
    for (uint32_t i = c0 + t; i < c1; i += NT) perm[i] = tmp[i];
    if (tm.part == 0 && t == 0) *child = make_children(nodes, base, cap, id, a, xs, nleft, counter, st);
    tm.sync();
    return tm.of(child, 0)[0];
  }
  if (tm.part == 0 && t == 0) nd->axis = -1;
  tm.sync();
  return -1;
}

// Builds the subtree of node `root` with one block: nodes of at most tw members are left to
// single warps (whole subtrees), the larger ones are split by the block, the smaller child
// first, so that the stack holds at most one node per halving.
template <int NT>
__device__ void block_build(BlockTree<NT> &s, int root, int64_t tw, uint32_t base, uint32_t cap, int64_t ncell,
                            int split_rule, const int4 *__restrict__ u, uint32_t *perm, uint32_t *tmp,
                            CellNode *nodes, int *counter, int *child, WarpTree *wt,
                            DevStatus *st) {
  const int t = threadIdx.x;
  const TreeTeam<NT, 1> tm{s, 0};
  int turn = 0;
  __syncthreads();
  if (t == 0) {
    s.stack[0] = root;
    s.sp = 1;
    s.npend = 0;
  }
  __syncthreads();
  while (s.sp > 0) {
    const int id = s.stack[s.sp - 1];
    const int64_t n = nodes[base + id].end - nodes[base + id].beg;
    const bool leaf = n <= ncell, hand = !leaf && n <= tw && s.npend < kPendCap;
    __syncthreads();
    if (t == 0) {
      --s.sp;
      if (leaf) nodes[base + id].axis = -1;
      if (hand) s.pend[s.npend++] = id;
    }
    __syncthreads();
    if (leaf || hand) continue;
    const int c0 = team_split<NT, 1>(tm, id, base, cap, split_rule, u, perm, tmp, nodes, counter, turn, child, st);
    if (t == 0 && c0 >= 0) {
      const CellNode &L = nodes[base + c0], &R = nodes[base + c0 + 1];
      const bool left_small = L.end - L.beg <= R.end - R.beg;
      s.stack[s.sp++] = left_small ? c0 + 1 : c0;
      s.stack[s.sp++] = left_small ? c0 : c0 + 1;
    }
    __syncthreads();
  }
  const int np = s.npend;
  for (int k = t >> 5; k < np; k += NT / 32)
    warp_build(s.pend[k], base, cap, ncell, split_rule, u, perm, tmp, nodes, counter, wt[t >> 5], st);
  __syncthreads();
}

// FP64 moments and membership of the leaves among the halo's first `count` nodes, one warp
// per leaf: warp `first` of `step`. Returns the leaves this warp took.
__device__ int leaf_moments(int first, int step, int count, uint32_t base, const int4 *__restrict__ u,
                            const float4 *__restrict__ v, const uint32_t *perm, uint32_t *leaf_of,
                            const CellNode *nodes, double *__restrict__ mom) {
  const int lane = threadIdx.x & 31;
  const unsigned FULL = 0xffffffffu;
  int nleaves = 0;
  for (int cur = first; cur < count; cur += step) {
    const CellNode *nd = &nodes[base + cur];
    if (nd->axis >= 0) continue;  // the same node for the whole warp
    ++nleaves;
    const uint32_t b = nd->beg, e = nd->end;
    const double M = (double)(e - b);
    long long sx[3] = {0, 0, 0};
    double sv[3] = {0, 0, 0};
#pragma unroll 2
    for (uint32_t i = b + lane; i < e; i += 32) {
      const uint32_t m = perm[i];
      leaf_of[m] = base + cur;
      const int4 p = u[m];
      const float4 q = v[m];
      sx[0] += p.x; sx[1] += p.y; sx[2] += p.z;
      sv[0] += (double)q.x; sv[1] += (double)q.y; sv[2] += (double)q.z;
    }
    for (int o = 16; o; o >>= 1)
      for (int k = 0; k < 3; ++k) {
        sx[k] += __shfl_xor_sync(FULL, sx[k], o);
        sv[k] += __shfl_xor_sync(FULL, sv[k], o);
      }
    double xm[3], vm[3];
    for (int k = 0; k < 3; ++k) {
      xm[k] = (double)sx[k] / M;
      vm[k] = sv[k] / M;
    }
    double c[6] = {0, 0, 0, 0, 0, 0};
#pragma unroll 2
    for (uint32_t i = b + lane; i < e; i += 32) {
      const float4 q = v[perm[i]];
      const double d0 = (double)q.x - vm[0], d1 = (double)q.y - vm[1], d2 = (double)q.z - vm[2];
      c[0] += d0 * d0; c[1] += d1 * d1; c[2] += d2 * d2;
      c[3] += d0 * d1; c[4] += d0 * d2; c[5] += d1 * d2;
    }
    for (int o = 16; o; o >>= 1)
      for (int k = 0; k < 6; ++k) c[k] += __shfl_xor_sync(FULL, c[k], o);
    if (lane == 0) {
      double *out = mom + 13 * (int64_t)(base + cur);
      out[0] = M;
      for (int k = 0; k < 3; ++k) { out[1 + k] = xm[k]; out[4 + k] = vm[k]; }
      for (int k = 0; k < 6; ++k) out[7 + k] = c[k] / M;
    }
  }
  return nleaves;
}

// Size classes of the tree build, each with its own launch: halos below kMidHalo members with
// a block of 256 threads, below kBigHalo with one of 1,024, the rest with a cluster of kTeam
// such blocks. A halo of 500,000 members on one SM took 10.2 ms: 6.5 levels of passes over its
// members, bound by their latency, 127 entropies and the leaves' moments in FP64, of which an
// SM does two lanes a cycle (now 1.5 ms; the launches of a 200^3 box 15.5 -> 4.7 ms in all).
constexpr int kTeam = 8;

template <int NT>
__global__ void __launch_bounds__(NT) k_cells_build(
    const uint32_t *__restrict__ hoff, const uint32_t *__restrict__ horder,
    const uint32_t *__restrict__ nodeoff, int64_t first, int64_t last,
    const int4 *__restrict__ u, const float4 *__restrict__ v, int nsearch_min, double f_cell,
    int ncell_min, int split_rule, uint32_t *perm, uint32_t *tmp,
    CellNode *nodes, double *__restrict__ mom, uint32_t *leaf_of,
    double *__restrict__ hs_out, DevStatus *st, int64_t szlo, int64_t szhi) {
  __shared__ BlockTree<NT> s;
  __shared__ int s_child;
  extern __shared__ __align__(16) unsigned char tree_smem[];
  if (first + (int64_t)blockIdx.x >= last) return;
  const int64_t h = horder[first + blockIdx.x];  // largest halos first
  const uint32_t hb = hoff[h], he = hoff[h + 1];
  const int64_t nh = he - hb;
  if (nh < nsearch_min || nh < szlo || nh >= szhi) return;  // each size class has its own launch
  const int64_t ncell = ncell_of(nh, f_cell, ncell_min);
  const uint32_t base = nodeoff[h], cap = nodeoff[h + 1] - base;
  const int t = threadIdx.x;
  for (uint32_t m = hb + t; m < he; m += NT) perm[m] = m;
  // root region: [min, max + 1)
  {
    int mn[3] = {0x7fffffff, 0x7fffffff, 0x7fffffff}, mx[3] = {-0x7fffffff, -0x7fffffff, -0x7fffffff};
#pragma unroll 4
    for (uint32_t m = hb + t; m < he; m += NT) {
      int4 p = u[m];
      mn[0] = min(mn[0], p.x); mn[1] = min(mn[1], p.y); mn[2] = min(mn[2], p.z);
      mx[0] = max(mx[0], p.x); mx[1] = max(mx[1], p.y); mx[2] = max(mx[2], p.z);
    }
    for (int a = 0; a < 3; ++a) {
      int lo = block_reduce<NT>(mn[a], MinOp(), s.ri);
      int hi = block_reduce<NT>(mx[a], MaxOp(), s.ri);
      if (t == 0) {
        nodes[base].lo[a] = lo;
        nodes[base].hi[a] = hi + 1;
      }
    }
    if (t == 0) {
      nodes[base].beg = hb;
      nodes[base].end = he;
      nodes[base].axis = -1;
      s.count = 1;
      s.nleaves = 0;
    }
  }
  __syncthreads();
  WarpTree *wt = reinterpret_cast<WarpTree *>(tree_smem);
  block_build<NT>(s, 0, max((int64_t)1024, nh / (2 * (NT / 32))), base, cap, ncell, split_rule, u, perm, tmp,
                  nodes, &s.count, &s_child, wt, st);
  const int nl = leaf_moments(t >> 5, NT / 32, s.count, base, u, v, perm, leaf_of, nodes, mom);
  if ((t & 31) == 0) atomicAdd(&s.nleaves, nl);
  __syncthreads();
  if (t == 0) hs_out[h * VR_HALO_COLS + VR_H_NCELLS] = (double)s.nleaves;
}

// The largest halos, a cluster each: the nodes of more than an eighth of the halo are split by
// the whole cluster, the subtrees below them by single blocks.
template <int NT>
__global__ void __launch_bounds__(NT) __cluster_dims__(kTeam, 1, 1) k_cells_cluster(
    const uint32_t *__restrict__ hoff, const uint32_t *__restrict__ horder,
    const uint32_t *__restrict__ nodeoff, int64_t first, int64_t last,
    const int4 *__restrict__ u, const float4 *__restrict__ v, int nsearch_min, double f_cell,
    int ncell_min, int split_rule, uint32_t *perm, uint32_t *tmp,
    CellNode *nodes, double *__restrict__ mom, uint32_t *leaf_of,
    double *__restrict__ hs_out, DevStatus *st, int64_t szlo, int64_t szhi) {
  __shared__ BlockTree<NT> s;
  __shared__ int s_child;
  extern __shared__ __align__(16) unsigned char tree_smem[];
  cg::cluster_group cl = cg::this_cluster();
  const int part = (int)cl.block_rank(), t = threadIdx.x;
  const int64_t at = first + blockIdx.x / kTeam;  // the same for the whole cluster
  if (at >= last) return;
  const int64_t h = horder[at];  // largest halos first
  const uint32_t hb = hoff[h], he = hoff[h + 1];
  const int64_t nh = he - hb;
  if (nh < nsearch_min || nh < szlo || nh >= szhi) return;  // each size class has its own launch
  const int64_t ncell = ncell_of(nh, f_cell, ncell_min);
  const uint32_t base = nodeoff[h], cap = nodeoff[h + 1] - base;
  const TreeTeam<NT, kTeam> tm{s, part};
  int turn = 0;
  const uint32_t c0 = hb + (uint32_t)(nh * part / kTeam), c1 = hb + (uint32_t)(nh * (part + 1) / kTeam);
  {
    int mn[3] = {0x7fffffff, 0x7fffffff, 0x7fffffff}, mx[3] = {-0x7fffffff, -0x7fffffff, -0x7fffffff};
#pragma unroll 4
    for (uint32_t m = c0 + t; m < c1; m += NT) {
      const int4 p = u[m];
      perm[m] = m;
      mn[0] = min(mn[0], p.x); mn[1] = min(mn[1], p.y); mn[2] = min(mn[2], p.z);
      mx[0] = max(mx[0], p.x); mx[1] = max(mx[1], p.y); mx[2] = max(mx[2], p.z);
    }
    for (int a = 0; a < 3; ++a) {
      const int lo = block_reduce<NT>(mn[a], MinOp(), s.ri), hi = block_reduce<NT>(mx[a], MaxOp(), s.ri);
      if (t == 0) {
        s.mm[0][a] = lo;
        s.mm[0][3 + a] = hi;
      }
    }
    if (t == 0) {
      s.count = 1;
      s.nleaves = 0;
    }
  }
  cl.sync();
  int *counter = cl.map_shared_rank(&s.count, 0);
  if (part == 0 && t == 0) {
    for (int a = 0; a < 3; ++a) {
      int lo = 0x7fffffff, hi = -0x7fffffff;
      for (int q = 0; q < kTeam; ++q) {
        lo = min(lo, cl.map_shared_rank(&s.mm[0][a], q)[0]);
        hi = max(hi, cl.map_shared_rank(&s.mm[0][3 + a], q)[0]);
      }
      nodes[base].lo[a] = lo;
      nodes[base].hi[a] = hi + 1;
    }
    nodes[base].beg = hb;
    nodes[base].end = he;
    nodes[base].axis = -1;
  }
  cl.sync();
  // every block keeps the same list of nodes: 64 of them when the cluster stops splitting, or
  // fewer
  __shared__ int s_list[64];
  int nlist = 1;
  if (t == 0) s_list[0] = 0;
  __syncthreads();
  for (int k = 0; k < nlist;) {
    const int id = s_list[k];
    const int64_t n = nodes[base + id].end - nodes[base + id].beg;
    if (n <= ncell || n <= nh / kTeam || nlist >= 63) {
      ++k;
      continue;
    }
    const int ch = team_split<NT, kTeam>(tm, id, base, cap, split_rule, u, perm, tmp, nodes, counter, turn,
                                         &s_child, st);
    __syncthreads();
    if (ch >= 0) {  // the children take the node's place
      if (t == 0) {
        s_list[k] = ch;
        s_list[nlist] = ch + 1;
      }
      ++nlist;
    } else {
      if (t == 0) s_list[k] = -1;  // a leaf
      ++k;
    }
    __syncthreads();
  }
  cl.sync();  // the others may still read the first block's s_child, which it writes below
  WarpTree *wt = reinterpret_cast<WarpTree *>(tree_smem);
  for (int k = part; k < nlist; k += kTeam) {
    const int id = s_list[k];
    if (id < 0) continue;
    const int64_t n = nodes[base + id].end - nodes[base + id].beg;
    block_build<NT>(s, id, max((int64_t)1024, n / (2 * (NT / 32))), base, cap, ncell, split_rule, u, perm, tmp,
                    nodes, counter, &s_child, wt, st);
  }
  cl.sync();
  const int nl = leaf_moments(part * (NT / 32) + (t >> 5), kTeam * (NT / 32), *counter, base, u, v, perm,
                              leaf_of, nodes, mom);
  if ((t & 31) == 0) atomicAdd(cl.map_shared_rank(&s.nleaves, 0), nl);
  cl.sync();
  if (part == 0 && t == 0) hs_out[h * VR_HALO_COLS + VR_H_NCELLS] = (double)s.nleaves;
}

// Leaf containing point p, or -1 outside the root region.
__device__ __forceinline__ int locate(const CellNode *__restrict__ nodes, uint32_t base, const int *p) {
  const CellNode &r = nodes[base];
  for (int a = 0; a < 3; ++a)
    if (p[a] < r.lo[a] || p[a] >= r.hi[a]) return -1;
  uint32_t id = base;
  for (int guard = 0; guard < 4096; ++guard) {
    const CellNode &nd = nodes[id];
    if (nd.axis < 0) return (int)id;
    id = base + (p[nd.axis] < nd.split ? nd.left : nd.right);
  }
  return -1;
}

// Cholesky of (xx, yy, zz, xy, xz, yz); false if not positive definite.
__device__ __forceinline__ bool chol3(const double *s, double *L) {
  double a00 = s[0], a11 = s[1], a22 = s[2], a10 = s[3], a20 = s[4], a21 = s[5];
  if (!(a00 > 0.0)) return false;
  double l00 = sqrt(a00);
  double l10 = a10 / l00, l20 = a20 / l00;
  double d1 = a11 - l10 * l10;
  if (!(d1 > 0.0)) return false;
  double l11 = sqrt(d1);
  double l21 = (a21 - l20 * l10) / l11;
  double d2 = a22 - l20 * l20 - l21 * l21;
  if (!(d2 > 0.0)) return false;
  double l22 = sqrt(d2);
  L[0] = l00; L[1] = l10; L[2] = l11; L[3] = l20; L[4] = l21; L[5] = l22;
  return true;
}

__global__ void k_ratio(const uint32_t *__restrict__ hid, const uint32_t *__restrict__ nodeoff,
                        int64_t m0, int64_t m1, const int4 *__restrict__ u, const float4 *__restrict__ v,
                        const float *__restrict__ f_l, const CellNode *__restrict__ nodes,
                        const double *__restrict__ mom, const uint32_t *__restrict__ leaf_of,
                        float *__restrict__ R, unsigned long long *__restrict__ ndegen,
                        const uint32_t *__restrict__ hoff, uint32_t szlo, uint32_t szhi) {
  int64_t m = m0 + (int64_t)blockIdx.x * blockDim.x + threadIdx.x;  // members [m0, m1)
  if (m >= m1) return;
  const uint32_t h = hid[m];
  const uint32_t base = nodeoff[h];
  if (nodeoff[h + 1] == base) return;  // halo not searched
  const uint32_t nh = hoff[h + 1] - hoff[h];
  if (nh <= szlo || nh > szhi) return;  // another launch's halo
  const int4 p = u[m];
  const float4 q = v[m];
  const uint32_t own = leaf_of[m];
  const CellNode &nd = nodes[own];
  int cells[7];
  int nc = 0;
  cells[nc++] = (int)own;
  for (int a = 0; a < 3; ++a) {
    for (int side = 0; side < 2; ++side) {
      int pp[3] = {p.x, p.y, p.z};
      pp[a] = side == 0 ? nd.lo[a] - 1 : nd.hi[a];
      int c = locate(nodes, base, pp);
      if (c < 0) continue;
      bool dup = false;
      for (int k = 0; k < nc; ++k) dup |= cells[k] == c;
      if (!dup) cells[nc++] = c;
    }
  }
  double w[7];
  int zero = -1;
  for (int k = 0; k < nc; ++k) {
    const double *c = mom + 13 * (int64_t)cells[k];
    double dx = (double)p.x - c[1], dy = (double)p.y - c[2], dz = (double)p.z - c[3];
    const double d2 = dx * dx + dy * dy + dz * dz;
    if (d2 == 0.0) {
      zero = k;
      break;
    }
    w[k] = rsqrt(d2);  // 1 / |x - xbar|
  }
  double vb[3] = {0, 0, 0}, sg[6] = {0, 0, 0, 0, 0, 0};
  if (zero >= 0) {
    const double *c = mom + 13 * (int64_t)cells[zero];
    for (int k = 0; k < 3; ++k) vb[k] = c[4 + k];
    for (int k = 0; k < 6; ++k) sg[k] = c[7 + k];
  } else {
    double ws = 0.0;
    for (int k = 0; k < nc; ++k) ws += w[k];
    for (int k = 0; k < nc; ++k) {
      const double *c = mom + 13 * (int64_t)cells[k];
      double f = w[k] / ws;
      for (int j = 0; j < 3; ++j) vb[j] += f * c[4 + j];
      for (int j = 0; j < 6; ++j) sg[j] += f * c[7 + j];
    }
  }
  double L[6];
  const int pidx = __float_as_int(q.w);
  if (!chol3(sg, L)) {
    R[pidx] = NAN;
    atomicAdd(ndegen, 1ULL);
    return;
  }
  double d0 = (double)q.x - vb[0], d1 = (double)q.y - vb[1], d2 = (double)q.z - vb[2];
  double y0 = d0 / L[0];
  double y1 = (d1 - L[1] * y0) / L[2];
  double y2 = (d2 - L[3] * y0 - L[4] * y1) / L[5];
  double qf = y0 * y0 + y1 * y1 + y2 * y2;
  const double ln2pi = 1.8378770664093453;  // ln(2 pi)
  double lnfbg = -0.5 * qf - 1.5 * ln2pi - log(L[0] * L[2] * L[5]);  // ln det L
  R[pidx] = (float)(log((double)f_l[pidx]) - lnfbg);
}

size_t background_bytes(int64_t n, const vr_params *p) {
  Arena ar;
  int64_t hmax = n / (p->nmin > 0 ? p->nmin : 1) + 2;
  ar.take<uint32_t>(hmax + 1);                       // nodeoff
  ar.take<uint32_t>(n);                              // perm
  ar.take<uint32_t>(n);                              // tmp
  ar.take<uint32_t>(n);                              // leaf_of
  int64_t nodes = max_nodes(n, p);
  ar.take<CellNode>(nodes);
  ar.take<double>(13 * nodes);
  ar.take<char>(scan_scratch_bytes<uint32_t>(hmax + 1));
  return ar.off;
}

int64_t max_nodes(int64_t n, const vr_params *p) {
  // smallest N_cell over searched halos is that of the smallest searched halo
  int64_t ns = p->nsearch_min;
  int64_t nc = (int64_t)floor(p->f_cell * (double)ns);
  if (nc < p->ncell_min) {
    nc = p->ncell_min;
    if (ns / 8 < nc) nc = ns / 8;
  }
  if (nc < 1) nc = 1;
  return kNodeFactor * ((n + nc) / (nc + 1)) + 16 * (n / ns + 1) + 16;
}

vr_status run_background(vr_ctx *ctx, const HaloSeg &g, const vr_params *p, Arena &ar,
                         const float *f_l, float *R, double *halo_stats, Background *out,
                         cudaStream_t s, const uint32_t *hoff_host) {
  const int64_t H = g.H;
  int64_t hmax = g.n / (p->nmin > 0 ? p->nmin : 1) + 2;
  Background &bg = *out;
  bg.nodeoff = ar.take<uint32_t>(hmax + 1);
  uint32_t *perm = bg.scratch = ar.take<uint32_t>(g.n);
  uint32_t *tmp = ar.take<uint32_t>(g.n);
  bg.leaf_of = ar.take<uint32_t>(g.n);
  int64_t cap = max_nodes(g.n, p);
  bg.nodes = ar.take<CellNode>(cap);
  bg.mom = ar.take<double>(13 * cap);
  void *scr = ar.take<char>(scan_scratch_bytes<uint32_t>(hmax + 1));
  if (!ar.ok()) return set_error(ctx, VR_ERR_WORKSPACE_TOO_SMALL, "workspace too small");
  if (H == 0) return VR_OK;
  if (hoff_host) {
    for (int64_t i = 0; i < H; ++i) {
      const vr_status st = halo_frames(ctx, g, i, i + 1, p->nsearch_min, halo_stats, s);
      if (st != VR_OK) return st;
    }
  } else {
    vr_status st = run_halo_frame(ctx, g, p->nsearch_min, halo_stats, s);
    if (st != VR_OK) return st;
  }
  k_node_caps<<<grid_for(H + 1, 256), 256, 0, s>>>(g.hoff, H, p->nsearch_min, p->f_cell,
                                                   p->ncell_min, bg.nodeoff);
  VR_LAUNCHED(ctx, "k_node_caps");
  VR_CUDA(ctx, exclusive_scan<uint32_t>(bg.nodeoff, bg.nodeoff, H + 1, scr, s));
  const size_t smem_big = sizeof(WarpTree) * (kBigT / 32), smem_small = sizeof(WarpTree) * (kSmallT / 32);
  VR_CUDA(ctx, cudaFuncSetAttribute(k_cells_cluster<kBigT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_big));
  VR_CUDA(ctx, cudaFuncSetAttribute(k_cells_build<kBigT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_big));
  VR_CUDA(ctx, cudaFuncSetAttribute(k_cells_build<kSmallT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_small));
  // entries [a, z) of the size order: size class 0 (small), 1 (kMidHalo), 2 (kBigHalo)
  auto build = [&](int cls, cudaStream_t st, int64_t a, int64_t z) {
    const unsigned grid = (unsigned)(z - a);
    const int64_t inf = 1LL << 40;
    if (cls == 2)
      k_cells_cluster<kBigT><<<kTeam * grid, kBigT, smem_big, st>>>(
          g.hoff, g.horder, bg.nodeoff, a, z, g.u, g.v, p->nsearch_min, p->f_cell, p->ncell_min, p->split_rule,
          perm, tmp, bg.nodes, bg.mom, bg.leaf_of, halo_stats, ctx->d_status, kBigHalo, inf);
    else if (cls == 1)
      k_cells_build<kBigT><<<grid, kBigT, smem_big, st>>>(
          g.hoff, g.horder, bg.nodeoff, a, z, g.u, g.v, p->nsearch_min, p->f_cell, p->ncell_min, p->split_rule,
          perm, tmp, bg.nodes, bg.mom, bg.leaf_of, halo_stats, ctx->d_status, kMidHalo, kBigHalo);
    else
      k_cells_build<kSmallT><<<grid, kSmallT, smem_small, st>>>(
          g.hoff, g.horder, bg.nodeoff, a, z, g.u, g.v, p->nsearch_min, p->f_cell, p->ncell_min, p->split_rule,
          perm, tmp, bg.nodes, bg.mom, bg.leaf_of, halo_stats, ctx->d_status, 0, kMidHalo);
  };
  unsigned long long *ndeg = (unsigned long long *)&ctx->d_status->info[0];
  if (hoff_host) {
    // one launch per searched halo, in the size order, with the CTA size of its class
    std::vector<uint32_t> ord(H);
    VR_CUDA(ctx, cudaMemcpyAsync(ord.data(), g.horder, H * sizeof(uint32_t), cudaMemcpyDeviceToHost, s));
    VR_CUDA(ctx, cudaStreamSynchronize(s));
    for (int64_t i = 0; i < H; ++i) {
      const int64_t nh = hoff_host[ord[i] + 1] - hoff_host[ord[i]];
      if (nh < p->nsearch_min) continue;
      build(nh >= kBigHalo ? 2 : (nh >= kMidHalo ? 1 : 0), s, i, i + 1);
      VR_LAUNCHED(ctx, "k_cells_build");
    }
    for (int64_t h = 0; h < H; ++h) {
      const int64_t a = hoff_host[h], z = hoff_host[h + 1];
      if (z - a < p->nsearch_min) continue;
      k_ratio<<<grid_for(z - a, 256), 256, 0, s>>>(g.hid, bg.nodeoff, a, z, g.u, g.v, f_l, bg.nodes,
                                                  bg.mom, bg.leaf_of, R, ndeg, g.hoff, 0u,
                                                  0xffffffffu);
      VR_LAUNCHED(ctx, "k_ratio");
    }
    return VR_OK;
  }
  // The two larger classes, the first entries of the size order, run on the context's side
  // stream while all other halos run on stream s; the launches overlap.
  const int64_t nbig = g.NHP / kBigHalo < H ? g.NHP / kBigHalo : H;
  const int64_t nmid = g.NHP / kMidHalo < H ? g.NHP / kMidHalo : H;
  VR_CUDA(ctx, cudaEventRecord(ctx->ev_fork, s));
  VR_CUDA(ctx, cudaStreamWaitEvent(ctx->side, ctx->ev_fork, 0));
  timer_begin(ctx, "cells_build_big", ctx->side);
  if (nbig > 0) {
    build(2, ctx->side, 0, nbig);
    VR_LAUNCHED(ctx, "k_cells_cluster");
  }
  if (nmid > 0) {
    build(1, ctx->side, 0, nmid);
    VR_LAUNCHED(ctx, "k_cells_build<big>");
  }
  timer_end(ctx, "cells_build_big", ctx->side);
  VR_TIMED(ctx, "cells_build", s, build(0, s, 0, H));
  VR_LAUNCHED(ctx, "k_cells_build");
  VR_CUDA(ctx, cudaEventRecord(ctx->ev_join, ctx->side));
  VR_CUDA(ctx, cudaStreamWaitEvent(s, ctx->ev_join, 0));
  if (f_l) return background_ratio(ctx, g, bg, f_l, R, s);
  return VR_OK;
}

vr_status background_ratio(vr_ctx *ctx, const HaloSeg &g, const Background &bg, const float *f_l,
                           float *R, cudaStream_t s, uint32_t szlo, uint32_t szhi) {
  if (g.H == 0) return VR_OK;
  unsigned long long *ndeg = (unsigned long long *)&ctx->d_status->info[0];
  VR_TIMED(ctx, "ratio", s, k_ratio<<<grid_for(g.NHP, 256), 256, 0, s>>>(g.hid, bg.nodeoff, 0, g.NHP, g.u, g.v, f_l, bg.nodes,
                                               bg.mom, bg.leaf_of, R, ndeg, g.hoff, szlo, szhi));
  VR_LAUNCHED(ctx, "k_ratio");
  return VR_OK;
}

}  // namespace vr
