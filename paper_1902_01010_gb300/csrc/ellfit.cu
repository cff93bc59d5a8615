// Skew-Gaussian fit of each searched halo's R distribution (Eq. skewgaus) and the
// normalised ratio ell = (R - Rbar) / sigma_R (Eq. ell), in three kernels:
//  - k_fit_hist, a block per halo: median and MAD of the finite R values, exact (radix
//    selection on FP32 keys; the FP64 keys |R - median| only for the members that FP32 cannot
//    tell apart from the MAD), MAD' = 1.4826 MAD; nbins = clamp(ceil(sqrt(N)), min, max) equal
//    bins on [median - 6 MAD', median + 6 MAD'], bin = floor((R - lo) / width) evaluated
//    without fused multiply-add wherever FP32 does not settle it, so the counts equal those
//    of an FP64 reference fed the same R values;
//  - k_fit_lm, a warp per halo: Levenberg-Marquardt on the counts (unweighted least squares;
//    start A = max count, Rbar = centre of the first fullest bin, sigma = MAD', s = 1; lambda
//    1e-3, /10 on an accepted step, x10 on a rejected one; stop on a relative cost change
//    below 1e-15, or when a step changes no parameter: a larger lambda only shortens it, in
//    the norm that weights each parameter by its diagonal of J^T J);
//  - k_ell, a thread per member.
// One block per halo for all three left 7 of 8 warps and their registers waiting for the one
// that iterates, and read every R 14 times with 256 threads (200^3 box: 3.53 ms; k_fit_hist now
// 0.33, k_fit_lm 1.02). k_fit_lm is bound by the latency of its chain of FP64 operations.
#include <math.h>

#include <vector>

#include "halos.cuh"
#include "vr_workspace.h"
#include "background.cuh"
#include "fit_bracket.h"

namespace vr {

namespace {

constexpr int kFitT = 256;          // threads of a histogram block, halos below kFitBig
constexpr int kFitTBig = 1024;      // and of kFitBig members or more
constexpr uint32_t kFitBig = 16384;
constexpr int kMaxFitBins = 1024;
constexpr int kFitCand = 2048;      // keys a selection holds in shared memory
constexpr int kLmWarps = 4;

__device__ __forceinline__ uint32_t fkey(float x) {
  uint32_t b = __float_as_uint(x);
  return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}
__device__ __forceinline__ float fkey_inv(uint32_t k) {
  uint32_t b = (k & 0x80000000u) ? (k & 0x7fffffffu) : ~k;
  return __uint_as_float(b);
}

struct FitSmem {
  uint32_t dig[2048];  // digit counts, later the histogram
  unsigned long long cand[kFitCand];
  uint32_t scan[32];
  unsigned long long pre, big;
  int rank, cnt, n;
};

// k-th smallest (0-based) 64-bit key of `nbits` bits among the block's keys produced by get(i)
// for i in [0, n) where valid; radix selection by 11-bit digits from the top. Once the keys
// that share the digits found so far fit in shared memory, they are kept there and the
// remaining digits read no further than that.
template <int NT, class Get>
__device__ unsigned long long block_select(int n, int k, int nbits, Get get, FitSmem &s) {
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  constexpr int kPer = 2048 / NT;
  if (t == 0) {
    s.pre = 0ULL;
    s.rank = k;
  }
  int held = -1;      // >= 0: that many candidates are in s.cand
  int hi = nbits;     // bits [0, hi) are still open
  while (hi > 0) {
    const int sh = hi > 11 ? hi - 11 : 0;
    const uint32_t mask = (1u << (hi - sh)) - 1u;
#pragma unroll
    for (int q = 0; q < kPer; ++q) s.dig[q * NT + t] = 0;
    __syncthreads();
    const unsigned long long pre = hi >= 64 ? 0ULL : s.pre >> hi;
    if (held >= 0) {
      for (int i = t; i < held; i += NT) {
        const unsigned long long key = s.cand[i];
        if (hi >= 64 || key >> hi == pre) atomicAdd(&s.dig[(uint32_t)(key >> sh) & mask], 1u);
      }
    } else {
#pragma unroll 4
      for (int i = t; i < n; i += NT) {
        unsigned long long key;
        if (get(i, key) && (hi >= 64 || key >> hi == pre)) atomicAdd(&s.dig[(uint32_t)(key >> sh) & mask], 1u);
      }
    }
    __syncthreads();
    // the digit that holds rank s.rank: thread t owns digits [kPer t, kPer (t + 1))
    uint32_t c[kPer], sum = 0;
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
      c[q] = s.dig[kPer * t + q];
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
    const uint32_t rk = (uint32_t)s.rank;
    __syncthreads();
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
      if (run <= rk && rk < run + c[q]) {
        s.pre |= (unsigned long long)(kPer * t + q) << sh;
        s.rank = (int)(rk - run);
        s.n = (int)c[q];
        s.cnt = 0;
      }
      run += c[q];
    }
    __syncthreads();
    if (held < 0 && sh > 0 && s.n <= kFitCand) {  // keep what shares the digits
      const unsigned long long p2 = s.pre >> sh;
#pragma unroll 4
      for (int i = t; i < n; i += NT) {
        unsigned long long key;
        if (get(i, key) && key >> sh == p2) s.cand[atomicAdd(&s.cnt, 1)] = key;
      }
      __syncthreads();
      held = s.cnt;
    }
    hi = sh;
  }
  const unsigned long long r = s.pre;
  __syncthreads();
  return r;
}

__device__ __forceinline__ double warp_sum(double x) {
  for (int o = 16; o; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  return x;
}

// Solves (JtJ + lambda diag(JtJ)) x = b by Gaussian elimination with partial pivoting;
// jj holds the upper triangle of JtJ row by row.
__device__ bool solve4(const double *jj, double lambda, const double *b, double *x) {
  double a[4][5];
  int q = 0;
  for (int i = 0; i < 4; ++i)
    for (int j = i; j < 4; ++j) {
      a[i][j] = a[j][i] = jj[q++];
    }
  for (int i = 0; i < 4; ++i) {
    a[i][i] = a[i][i] + lambda * a[i][i];
    a[i][4] = b[i];
  }
  double inv[4];
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    // bring the largest of column c up, row by row (constant indices keep the rows in registers)
#pragma unroll
    for (int r = c + 1; r < 4; ++r)
      if (fabs(a[r][c]) > fabs(a[c][c])) {
#pragma unroll
        for (int j = 0; j < 5; ++j) {
          const double tt = a[c][j];
          a[c][j] = a[r][j];
          a[r][j] = tt;
        }
      }
    if (!(fabs(a[c][c]) > 0.0)) return false;
    inv[c] = 1.0 / a[c][c];
#pragma unroll
    for (int r = c + 1; r < 4; ++r) {
      const double f = a[r][c] * inv[c];
#pragma unroll
      for (int j = c; j < 5; ++j) a[r][j] -= f * a[c][j];
    }
  }
#pragma unroll
  for (int r = 3; r >= 0; --r) {
    double s = a[r][4];
#pragma unroll
    for (int j = r + 1; j < 4; ++j) s -= a[r][j] * x[j];
    x[r] = s * inv[r];
  }
  return true;
}

// R of every slot of the halos with szlo < N_H <= szhi, in slot order (the selections
// below read it many times).
__global__ void k_gather_r(const float4 *__restrict__ v, const float *__restrict__ R, int64_t nhp,
                           const uint32_t *__restrict__ hid, const uint32_t *__restrict__ hoff,
                           uint32_t szlo, uint32_t szhi, float *__restrict__ Rs) {
  const int64_t m = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (m >= nhp) return;
  const uint32_t h = hid[m], nh = hoff[h + 1] - hoff[h];
  if (nh > szlo && nh <= szhi) Rs[m] = R[__float_as_int(v[m].w)];
}

// The key of rank k - 1 given the key `a` of rank k (0-based, k >= 1) among the valid
// keys: `a` itself if fewer than k keys lie below it (a run of equal keys), else the
// largest key below `a`. One pass instead of a second selection.
template <int NT, class Get>
__device__ unsigned long long block_prev_rank(int n, int k, unsigned long long a, Get get, FitSmem &s) {
  const int t = threadIdx.x;
  if (t == 0) {
    s.big = 0ULL;
    s.cnt = 0;
  }
  __syncthreads();
  unsigned long long mx = 0ULL;
  int c = 0;
#pragma unroll 4
  for (int i = t; i < n; i += NT) {
    unsigned long long key;
    if (!get(i, key) || key >= a) continue;
    ++c;
    mx = key > mx ? key : mx;
  }
  c = __reduce_add_sync(0xffffffffu, c);
  for (int o = 16; o; o >>= 1) {
    const unsigned long long y = __shfl_xor_sync(0xffffffffu, mx, o);
    mx = y > mx ? y : mx;
  }
  if ((t & 31) == 0) {
    atomicAdd(&s.cnt, c);
    atomicMax(&s.big, mx);
  }
  __syncthreads();
  const unsigned long long r = s.cnt < k ? a : s.big;
  __syncthreads();
  return r;
}

// k-th smallest |x - med| (exact FP64 values), and with `even` the one before it: median of
// the two. FP32 distances d_f = |x - med_f| find a narrow bracket of it first (22 leading key
// bits); only members whose d_f lies within the rounding error of the bracket are
// evaluated in FP64. The one before is mostly below the bracket (a slice of 2^-14), and then
// found by one pass over the FP64 values: by d_f, two values on either side of a key's edge
// may come in the wrong order. Returns false where the bracket does not work out (many equal
// values, or a spread that FP32 does not resolve around med): the caller selects on FP64 keys.
template <int NT, class Val, class Get>
__device__ bool block_mad(int nh, int k, bool even, double med, Val val, Get getd, FitSmem &s, double *out) {
  const int t = threadIdx.x;
  const float mf = (float)med;
  auto getf = [&](int i, unsigned long long &key) {
    const float x = val(i);
    key = __float_as_uint(fabsf(x - mf)) >> kDistDrop;
    return (bool)isfinite(x);
  };
  const uint32_t top = (uint32_t)block_select<NT>(nh, k, kDistBits, getf, s);
  double lo, hi, err;  // [lo, hi] holds rank k
  if (!dist_bracket(top, med, &lo, &hi, &err)) return false;
  const float flo = (float)(lo - 4.0 * err), fhi = (float)(hi + 4.0 * err);
  if (t == 0) {
    s.cnt = 0;
    s.n = 0;
  }
  __syncthreads();
  int below = 0;
#pragma unroll 4
  for (int i = t; i < nh; i += NT) {
    const float x = val(i);
    if (!isfinite(x)) continue;
    const float d = fabsf(x - mf);
    if (d > fhi) continue;
    if (d < flo) {
      ++below;
      continue;
    }
    const double e = fabs(__dsub_rn((double)x, med));
    if (e < lo) {
      ++below;
    } else if (e <= hi) {
      const int at = atomicAdd(&s.cnt, 1);
      if (at < kFitCand) s.cand[at] = (unsigned long long)__double_as_longlong(e);
    }
  }
  below = __reduce_add_sync(0xffffffffu, below);
  if ((t & 31) == 0) atomicAdd(&s.n, below);
  __syncthreads();
  const int m = s.cnt, r = k - s.n;
  __syncthreads();
  if (m > kFitCand || r < 0 || r >= m) return false;
  // rank r (and r - 1) of the m keys in shared memory: every thread ranks its own
  for (int i = t; i < m; i += NT) {
    const unsigned long long key = s.cand[i];
    int less = 0, same = 0;
    for (int j = 0; j < m; ++j) {
      less += s.cand[j] < key;
      same += s.cand[j] == key;
    }
    if (less <= r && r < less + same) s.pre = key;
    if (r > 0 && less <= r - 1 && r - 1 < less + same) s.big = key;
  }
  __syncthreads();
  const unsigned long long ka = s.pre;
  unsigned long long kb = s.big;
  __syncthreads();
  if (even && r == 0) kb = block_prev_rank<NT>(nh, k, ka, getd, s);
  const double a = __longlong_as_double((long long)ka), b = __longlong_as_double((long long)kb);
  *out = even ? 0.5 * (b + a) : a;
  return true;
}

}  // namespace

// Median, MAD and histogram of a halo's R. The counts go to cnt[hoff[h] ...] and lo, width,
// MAD' and the number of bins (0: no fit) to the halo row's RBAR, SIGR, LX2 and LV2, for
// k_fit_lm, which leaves the row as documented.
template <int NT>
__global__ void __launch_bounds__(NT) k_fit_hist(const uint32_t *__restrict__ hoff,
                                                 const uint32_t *__restrict__ horder,
                                                 const uint32_t *__restrict__ nodeoff, int64_t first,
                                                 int64_t last, const float *__restrict__ Rs, int nb_min,
                                                 int nb_max, double *__restrict__ hs,
                                                 uint32_t *__restrict__ cnt, uint32_t szlo, uint32_t szhi) {
  __shared__ FitSmem s;
  if (first + (int64_t)blockIdx.x >= last) return;
  const int64_t h = horder[first + blockIdx.x];  // largest halos first
  if (nodeoff[h + 1] == nodeoff[h]) return;      // not searched
  const uint32_t hb = hoff[h], he = hoff[h + 1];
  const int nh = (int)(he - hb);
  if (he - hb <= szlo || he - hb > szhi) return;            // another launch's halo
  if ((NT == kFitTBig) != (he - hb >= kFitBig)) return;     // each size class has its own launch
  const int t = threadIdx.x;
  const float *Rh = Rs + hb;
  auto rval = [&](int i) { return Rh[i]; };
  // number of finite values
  if (t == 0) s.n = 0;
  __syncthreads();
  int c = 0;
#pragma unroll 4
  for (int i = t; i < nh; i += NT) c += isfinite(rval(i)) ? 1 : 0;
  c = __reduce_add_sync(0xffffffffu, c);
  if ((t & 31) == 0) atomicAdd(&s.n, c);
  __syncthreads();
  const int n = s.n;
  __syncthreads();
  double *row = hs + h * VR_HALO_COLS;
  if (n < 2) {
    if (t == 0) {
      row[VR_H_RBAR] = NAN;
      row[VR_H_SIGR] = NAN;
      row[VR_H_LV2] = 0.0;
    }
    return;
  }
  auto getf = [&](int i, unsigned long long &key) {
    float x = rval(i);
    if (!isfinite(x)) return false;
    key = fkey(x);
    return true;
  };
  double med;
  {
    const unsigned long long ka = block_select<NT>(nh, n / 2, 32, getf, s);
    float a = fkey_inv((uint32_t)ka);
    if (n & 1) {
      med = (double)a;
    } else {
      float b = fkey_inv((uint32_t)block_prev_rank<NT>(nh, n / 2, ka, getf, s));
      med = 0.5 * ((double)b + (double)a);
    }
  }
  auto getd = [&](int i, unsigned long long &key) {
    float x = rval(i);
    if (!isfinite(x)) return false;
    key = (unsigned long long)__double_as_longlong(fabs(__dsub_rn((double)x, med)));
    return true;
  };
  double mad;
  if (!block_mad<NT>(nh, n / 2, !(n & 1), med, rval, getd, s, &mad)) {
    const unsigned long long ka = block_select<NT>(nh, n / 2, 64, getd, s);
    mad = __longlong_as_double((long long)ka);
    if (!(n & 1))
      mad = 0.5 * (__longlong_as_double((long long)block_prev_rank<NT>(nh, n / 2, ka, getd, s)) + mad);
  }
  mad = __dmul_rn(1.4826, mad);
  if (!(mad > 0.0)) {
    if (t == 0) {
      row[VR_H_RBAR] = med;
      row[VR_H_SIGR] = NAN;
      row[VR_H_LV2] = 0.0;
    }
    return;
  }
  int nb = (int)ceil(sqrt((double)n));  // ceil(sqrt(n))
  while ((long long)nb * nb < n) ++nb;
  while (nb > 0 && (long long)(nb - 1) * (nb - 1) >= n) --nb;
  if (nb < nb_min) nb = nb_min;
  if (nb > nb_max) nb = nb_max;
  const double lo = __dsub_rn(med, __dmul_rn(6.0, mad));
  const double width = __ddiv_rn(__dmul_rn(12.0, mad), (double)nb);
  for (int b = t; b < nb; b += NT) s.dig[b] = 0;
  __syncthreads();
  // FP32 bin position f, within e of the FP64 one
  const float lof = (float)lo, invw = (float)(1.0 / width), fnb = (float)nb;
  const float e0 = 2.4e-7f * invw * fabsf(lof) + 1e-6f * fnb;
#pragma unroll 4
  for (int i = t; i < nh; i += NT) {
    float x = rval(i);
    if (!isfinite(x)) continue;
    const float f = (x - lof) * invw, e = e0 + 1e-6f * fabsf(f);
    if (f < -1.0f || f > fnb + 1.0f) {
      if (e < 0.5f) continue;
    } else if (f - floorf(f) > e && floorf(f) + 1.0f - f > e) {
      const int b = (int)floorf(f);
      if (b >= 0 && b < nb) atomicAdd(&s.dig[b], 1u);
      continue;
    }
    const double g = floor(__ddiv_rn(__dsub_rn((double)x, lo), width));
    if (g >= 0.0 && g < (double)nb) atomicAdd(&s.dig[(int)g], 1u);
  }
  __syncthreads();
  // a halo has one word per member for its counts: more bins than members (only with a
  // minimum number of bins above the halo's size) are kept as the members' bins instead
  const bool sparse = nb > nh;
  if (!sparse) {
    for (int b = t; b < nb; b += NT) cnt[hb + b] = s.dig[b];
  } else if (t == 0) {
    int at = 0;
    for (int b = 0; b < nb; ++b)
      for (uint32_t k = 0; k < s.dig[b]; ++k) cnt[hb + at++] = (uint32_t)b;
    while (at < nh) cnt[hb + at++] = 0xffffffffu;
  }
  if (t == 0) {
    row[VR_H_RBAR] = lo;
    row[VR_H_SIGR] = width;
    row[VR_H_LX2] = mad;
    row[VR_H_LV2] = (double)(sparse ? -nb : nb);
  }
}

// Eq. skewgaus at x and its gradient with respect to (A, Rbar, sigma, s), from parameters
// prepared once per step: the divisions are by the parameters only.
struct SgPar {
  double A, mu, il, ir, isg, is;  // 1 / (s sigma)^2, 1 / sigma^2, 1 / sigma, 1 / s
};
__device__ __forceinline__ SgPar sg_par(const double *p) {
  SgPar q;
  q.A = p[0];
  q.mu = p[1];
  q.isg = 1.0 / p[2];
  q.is = 1.0 / p[3];
  q.ir = q.isg * q.isg;
  q.il = q.ir * (q.is * q.is);
  return q;
}
__device__ __forceinline__ double sg_eval(double x, const SgPar &q, double *g) {
  const double d = x - q.mu;
  const bool left = d < 0.0;
  const double iw = left ? q.il : q.ir;
  const double di = d * iw;
  const double e = exp(-0.5 * (d * di));
  const double f = q.A * e;
  if (g) {
    g[0] = e;
    g[1] = f * di;
    const double g2 = g[1] * d;
    g[2] = g2 * q.isg;
    g[3] = left ? g2 * q.is : 0.0;
  }
  return f;
}

// Sums of 16 values over the warp: halving exchanges leave lane l with the sum of value l / 2,
// with 16 additions instead of 80 (an FP64 addition of a warp occupies its SM's FP64 lanes for
// 16 cycles), then every lane gets all of them.
__device__ __forceinline__ void warp_sum16(double *v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 16, m = 8; m; o >>= 1, m >>= 1) {
    const bool up = lane & o;
#pragma unroll
    for (int j = 0; j < m; ++j) {
      const double send = up ? v[j] : v[j + m], keep = up ? v[j + m] : v[j];
      v[j] = keep + __shfl_xor_sync(0xffffffffu, send, o);
    }
  }
  const double x = v[0] + __shfl_xor_sync(0xffffffffu, v[0], 1);
#pragma unroll
  for (int j = 0; j < 16; ++j) v[j] = __shfl_sync(0xffffffffu, x, 2 * j);
}

__global__ void __launch_bounds__(32 * kLmWarps) k_fit_lm(const uint32_t *__restrict__ hoff,
                                                          const uint32_t *__restrict__ horder,
                                                          const uint32_t *__restrict__ nodeoff,
                                                          int64_t first, int64_t last, int nb_max, int iters,
                                                          const uint32_t *__restrict__ cnt,
                                                          double *__restrict__ hs, uint32_t szlo,
                                                          uint32_t szhi) {
  extern __shared__ __align__(16) double s_bins[];  // per warp: counts, centres
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t r = first + (int64_t)blockIdx.x * kLmWarps + w;
  if (r >= last) return;
  const int64_t h = horder[r];  // largest halos first
  if (nodeoff[h + 1] == nodeoff[h]) return;  // not searched
  const uint32_t hb = hoff[h], nh = hoff[h + 1] - hb;
  if (nh <= szlo || nh > szhi) return;  // another launch's halo
  double *row = hs + h * VR_HALO_COLS;
  const double lo = row[VR_H_RBAR], width = row[VR_H_SIGR], mad = row[VR_H_LX2];
  const int nbs = (int)row[VR_H_LV2], nb = nbs < 0 ? -nbs : nbs;
  __syncwarp();
  if (lane == 0) row[VR_H_LX2] = row[VR_H_LV2] = NAN;
  if (nb == 0) return;
  double *s_cnt = s_bins + (size_t)w * 2 * nb_max, *s_x = s_cnt + nb_max;
  unsigned long long best = 0;  // first fullest bin: (count, ~bin) maximal
  for (int b = lane; b < nb; b += 32) s_cnt[b] = nbs < 0 ? 0.0 : (double)cnt[hb + b];
  __syncwarp();
  if (nbs < 0 && lane == 0)
    for (uint32_t i = 0; i < nh; ++i)
      if (cnt[hb + i] < (uint32_t)nb) s_cnt[cnt[hb + i]] += 1.0;
  __syncwarp();
  for (int b = lane; b < nb; b += 32) {
    const uint32_t c = (uint32_t)s_cnt[b];
    s_x[b] = __dadd_rn(lo, __dmul_rn((double)b + 0.5, width));
    const unsigned long long k = ((unsigned long long)c << 32) | (unsigned)~b;
    best = k > best ? k : best;
  }
  for (int o = 16; o; o >>= 1) {
    const unsigned long long y = __shfl_xor_sync(0xffffffffu, best, o);
    best = y > best ? y : best;
  }
  __syncwarp();
  const int mode = (int)~(uint32_t)best;
  double p[4] = {s_cnt[mode], s_x[mode], mad, 1.0};
  auto cost_of = [&](const double *pp) {
    const SgPar q = sg_par(pp);
    double c = 0.0;
    for (int b = lane; b < nb; b += 32) {
      const double d = s_cnt[b] - sg_eval(s_x[b], q, nullptr);
      c += d * d;
    }
    return warp_sum(c);
  };
  double cost = cost_of(p), lambda = 1e-3;
  // J^T J and J^T r depend on p alone: after a rejected step (p unchanged) the sums of
  // the previous iteration are reused as they are
  double jj[16];  // upper triangle of J^T J (10), J^T r (4)
  bool fresh = true;
  for (int it = 0; it < iters; ++it) {
    if (fresh) {
      const SgPar q = sg_par(p);
#pragma unroll
      for (int k = 0; k < 16; ++k) jj[k] = 0.0;
      for (int b = lane; b < nb; b += 32) {
        double g[4];
        const double d = s_cnt[b] - sg_eval(s_x[b], q, g);
        int k = 0;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          jj[10 + i] += g[i] * d;
#pragma unroll
          for (int j = i; j < 4; ++j) jj[k++] += g[i] * g[j];
        }
      }
      warp_sum16(jj);
      fresh = false;
    }
    double delta[4] = {0, 0, 0, 0};
    const bool ok = solve4(jj, lambda, jj + 10, delta);
    double qp[4];
    bool same = true;  // a step lost to rounding
    for (int i = 0; i < 4; ++i) {
      qp[i] = p[i] + (ok ? delta[i] : 0.0);
      same &= __double_as_longlong(qp[i]) == __double_as_longlong(p[i]);
    }
    if (ok && same) break;  // and with it every shorter one
    double ncost = INFINITY;
    if (ok && qp[2] > 0.0 && qp[3] > 0.0) ncost = cost_of(qp);
    if (ncost < cost) {
      const double rel = (cost - ncost) / cost;
      for (int i = 0; i < 4; ++i) p[i] = qp[i];
      cost = ncost;
      fresh = true;
      lambda /= 10.0;
      if (rel < 1e-15) break;
    } else {
      lambda *= 10.0;
      if (lambda > 1e30) break;
    }
  }
  if (lane == 0) {
    row[VR_H_RBAR] = p[1];
    row[VR_H_SIGR] = p[2];
  }
}

// ell of the members of the fitted halos (NaN where sigma_R is).
__global__ void k_ell(const uint32_t *__restrict__ hoff, const uint32_t *__restrict__ hid,
                      const uint32_t *__restrict__ nodeoff, int64_t m0, int64_t m1,
                      const float4 *__restrict__ v, const float *__restrict__ Rs,
                      const double *__restrict__ hs, float *__restrict__ ell, uint32_t szlo, uint32_t szhi) {
  const int64_t m = m0 + (int64_t)blockIdx.x * blockDim.x + threadIdx.x;  // slots [m0, m1)
  if (m >= m1) return;
  const uint32_t h = hid[m];
  if (nodeoff[h + 1] == nodeoff[h]) return;
  const uint32_t nh = hoff[h + 1] - hoff[h];
  if (nh <= szlo || nh > szhi) return;
  const double *row = hs + (int64_t)h * VR_HALO_COLS;
  ell[__float_as_int(v[m].w)] = (float)(((double)Rs[m] - row[VR_H_RBAR]) / row[VR_H_SIGR]);
}

vr_status run_fit(vr_ctx *ctx, const HaloSeg &g, const Background &bg, const vr_params *p,
                  const float *R, double *halo_stats, float *ell, cudaStream_t s, const uint32_t *hoff_host,
                  uint32_t szlo, uint32_t szhi) {
  if (g.H == 0) return VR_OK;
  if (p->fit_nbins_max > kMaxFitBins)
    return set_error(ctx, VR_ERR_INVALID_ARG, "fit_nbins_max above %d", kMaxFitBins);
  float *Rs = reinterpret_cast<float *>(g.scratch_u32_a);  // [n + 1] words, unused here
  if (hoff_host) szlo = 0, szhi = 0xffffffffu;
  k_gather_r<<<grid_for(g.NHP, 256), 256, 0, s>>>(g.v, R, g.NHP, g.hid, g.hoff, szlo, szhi, Rs);
  VR_LAUNCHED(ctx, "k_gather_r");
  // the attribute belongs to the function, not to this call: it is the same for every context, so
  // that another host thread's call cannot lower it between here and the launch
  constexpr size_t kLmRow = (size_t)kLmWarps * 2 * sizeof(double);
  VR_CUDA(ctx, cudaFuncSetAttribute(k_fit_lm, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)(kLmRow * kMaxFitBins)));
  const size_t lm_smem = kLmRow * p->fit_nbins_max;
  // halos [a, z) of the size order; the large ones are its first, at most NHP / kFitBig
  auto fit = [&](int64_t a, int64_t z) -> vr_status {
    const int64_t nbig = g.NHP / kFitBig, zb = nbig < z ? nbig : z;
    if (zb > a && szhi >= kFitBig) {
      k_fit_hist<kFitTBig><<<(unsigned)(zb - a), kFitTBig, 0, s>>>(
          g.hoff, g.horder, bg.nodeoff, a, zb, Rs, p->fit_nbins_min, p->fit_nbins_max, halo_stats, bg.scratch,
          szlo, szhi);
      VR_LAUNCHED(ctx, "k_fit_hist<big>");
    }
    if (szlo < kFitBig) {
      k_fit_hist<kFitT><<<(unsigned)(z - a), kFitT, 0, s>>>(
          g.hoff, g.horder, bg.nodeoff, a, z, Rs, p->fit_nbins_min, p->fit_nbins_max, halo_stats, bg.scratch,
          szlo, szhi);
      VR_LAUNCHED(ctx, "k_fit_hist");
    }
    k_fit_lm<<<grid_for(z - a, kLmWarps), 32 * kLmWarps, lm_smem, s>>>(
        g.hoff, g.horder, bg.nodeoff, a, z, p->fit_nbins_max, p->fit_iters, bg.scratch, halo_stats, szlo, szhi);
    VR_LAUNCHED(ctx, "k_fit_lm");
    return VR_OK;
  };
  auto normalise = [&](int64_t a, int64_t z) {
    k_ell<<<grid_for(z - a, 256), 256, 0, s>>>(g.hoff, g.hid, bg.nodeoff, a, z, g.v, Rs, halo_stats, ell, szlo,
                                               szhi);
  };
  if (hoff_host) {  // one launch per searched halo, in the size order
    std::vector<uint32_t> ord(g.H);
    VR_CUDA(ctx, cudaMemcpyAsync(ord.data(), g.horder, g.H * sizeof(uint32_t), cudaMemcpyDeviceToHost, s));
    VR_CUDA(ctx, cudaStreamSynchronize(s));
    for (int64_t i = 0; i < g.H; ++i) {
      const uint32_t a = hoff_host[ord[i]], z = hoff_host[ord[i] + 1];
      if (z - a < (uint32_t)p->nsearch_min) continue;
      const vr_status st = fit(i, i + 1);
      if (st != VR_OK) return st;
      normalise(a, z);
      VR_LAUNCHED(ctx, "k_ell");
    }
    return VR_OK;
  }
  timer_begin(ctx, "ell_fit", s);
  const vr_status st = fit(0, g.H);
  if (st != VR_OK) return st;
  normalise(0, g.NHP);
  VR_LAUNCHED(ctx, "k_ell");
  timer_end(ctx, "ell_fit", s);
  return VR_OK;
}

}  // namespace vr
