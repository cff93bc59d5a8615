// Device-wide primitives: exclusive prefix sum and a stable LSD radix sort of
// (key, value) pairs. Written for sm_103a: 256-thread blocks, warp-shuffle scans,
// __match_any_sync for stable in-tile ranking, 16-byte scan loads.
#include "vr_internal.cuh"

namespace vr {

namespace {

constexpr int kScanThreads = 256;
constexpr int kScanItems = 8;
constexpr int kScanTile = kScanThreads * kScanItems;  // 2048

template <class T>
__device__ __forceinline__ T warp_incl_scan(T v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    T u = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += u;
  }
  return v;
}

// Block-wide exclusive scan of one value per thread; returns the block total in *total.
template <class T>
__device__ __forceinline__ T block_excl_scan(T v, T *total, T *s_warp) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  T inc = warp_incl_scan(v);
  if (lane == 31) s_warp[w] = inc;
  __syncthreads();
  if (w == 0) {
    T x = lane < (kScanThreads / 32) ? s_warp[lane] : T(0);
    T xi = warp_incl_scan(x);
    if (lane < (kScanThreads / 32)) s_warp[lane] = xi - x;
    if (lane == (kScanThreads / 32) - 1) s_warp[kScanThreads / 32] = xi;
  }
  __syncthreads();
  T r = inc - v + s_warp[w];
  *total = s_warp[kScanThreads / 32];
  __syncthreads();
  return r;
}

// A thread's kScanItems consecutive values of the tile at `base` (zero beyond n), as
// 16-byte loads for a full tile at an aligned address.
template <class T>
__device__ __forceinline__ bool scan_wide(const T *p, int64_t base, int64_t n) {
  return base + kScanTile <= n && (reinterpret_cast<uintptr_t>(p) & 15) == 0;
}
template <class T>
__device__ __forceinline__ void scan_load(const T *in, int64_t base, int64_t n, T *v) {
  const int64_t i0 = base + (int64_t)threadIdx.x * kScanItems;
  if (scan_wide(in, base, n)) {
    const uint4 *q = reinterpret_cast<const uint4 *>(in + i0);
    constexpr int kVec = kScanItems * sizeof(T) / 16;
    uint4 *o = reinterpret_cast<uint4 *>(v);
#pragma unroll
    for (int k = 0; k < kVec; ++k) o[k] = q[k];
  } else {
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) v[k] = i0 + k < n ? in[i0 + k] : T(0);
  }
}

template <class T>
__global__ void __launch_bounds__(kScanThreads) k_scan_reduce(const T *in, int64_t n, T *sums) {
  __shared__ T s_warp[kScanThreads / 32 + 1];
  alignas(16) T v[kScanItems];
  scan_load(in, (int64_t)blockIdx.x * kScanTile, n, v);
  T acc = 0;
#pragma unroll
  for (int k = 0; k < kScanItems; ++k) acc += v[k];
  T tot;
  block_excl_scan(acc, &tot, s_warp);
  if (threadIdx.x == 0) sums[blockIdx.x] = tot;
}

// One block scan per tile, over the threads' sums of 8 consecutive values. A scan of 256
// values per round, 8 rounds of three barriers each, took 8 us for one tile, and a call of
// the substructure stages makes some 30 such launches (now 3.1 us).
template <class T>
__global__ void __launch_bounds__(kScanThreads) k_scan_apply(const T *in, T *out, int64_t n,
                                                              const T *offs) {
  __shared__ T s_warp[kScanThreads / 32 + 1];
  const int64_t base = (int64_t)blockIdx.x * kScanTile;
  alignas(16) T v[kScanItems];
  scan_load(in, base, n, v);
  T acc = 0;
#pragma unroll
  for (int k = 0; k < kScanItems; ++k) acc += v[k];
  T tot;
  T run = block_excl_scan(acc, &tot, s_warp) + (offs ? offs[blockIdx.x] : T(0));
#pragma unroll
  for (int k = 0; k < kScanItems; ++k) {
    const T x = v[k];
    v[k] = run;
    run += x;
  }
  const int64_t i0 = base + (int64_t)threadIdx.x * kScanItems;
  if (scan_wide(out, base, n)) {
    constexpr int kVec = kScanItems * sizeof(T) / 16;
    const uint4 *q = reinterpret_cast<const uint4 *>(v);
#pragma unroll
    for (int k = 0; k < kVec; ++k) reinterpret_cast<uint4 *>(out + i0)[k] = q[k];
  } else {
#pragma unroll
    for (int k = 0; k < kScanItems; ++k)
      if (i0 + k < n) out[i0 + k] = v[k];
  }
}

}  // namespace

template <class T>
size_t scan_scratch_bytes(int64_t n) {
  size_t b = 0;
  while (n > kScanTile) {
    n = ceil_div(n, kScanTile);
    b += ((size_t)n * sizeof(T) + 255) & ~(size_t)255;
  }
  return b + 256;
}

template <class T>
cudaError_t exclusive_scan(const T *in, T *out, int64_t n, void *scratch, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  if (n <= kScanTile) {
    k_scan_apply<T><<<1, kScanThreads, 0, s>>>(in, out, n, nullptr);
    count_launch();
    return cudaGetLastError();
  }
  int64_t nb = ceil_div(n, kScanTile);
  T *sums = (T *)scratch;
  char *rest = (char *)scratch + (((size_t)nb * sizeof(T) + 255) & ~(size_t)255);
  k_scan_reduce<T><<<(unsigned)nb, kScanThreads, 0, s>>>(in, n, sums);
  count_launch();
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  e = exclusive_scan<T>(sums, sums, nb, rest, s);
  if (e != cudaSuccess) return e;
  k_scan_apply<T><<<(unsigned)nb, kScanThreads, 0, s>>>(in, out, n, sums);
  count_launch();
  return cudaGetLastError();
}

template size_t scan_scratch_bytes<uint32_t>(int64_t);
template size_t scan_scratch_bytes<unsigned long long>(int64_t);
template cudaError_t exclusive_scan<uint32_t>(const uint32_t *, uint32_t *, int64_t, void *,
                                              cudaStream_t);
template cudaError_t exclusive_scan<unsigned long long>(const unsigned long long *,
                                                        unsigned long long *, int64_t, void *,
                                                        cudaStream_t);

// ------------------------------------------------------------------ radix sort
namespace {

constexpr int kRadThreads = 256;
constexpr int kRadWarps = kRadThreads / 32;
// Keys per thread: 16 where that fills the GPU, 4 below kRadSmall keys (8 tiles of 4,096
// keys of a 32^3 box leave 144 of 152 SMs idle: 18.8 -> 4.6 us a scatter, 10.2 -> 4.5 us
// a histogram).
constexpr int kRadItems = 16, kRadItemsSmall = 4;
constexpr int64_t kRadSmall = 1 << 20;
constexpr int kRadOne = kRadThreads * kRadItems;  // sorted by one block in one launch up to here

template <class K, int ITEMS>
__global__ void __launch_bounds__(kRadThreads) k_radix_hist(const K *keys, int64_t n, int shift,
                                                             int64_t ntiles, uint32_t *counts) {
  __shared__ uint32_t h[256];
  h[threadIdx.x] = 0;
  __syncthreads();
  const int64_t base = (int64_t)blockIdx.x * (kRadThreads * ITEMS);
#pragma unroll
  for (int r = 0; r < ITEMS; ++r) {
    int64_t i = base + r * kRadThreads + threadIdx.x;
    if (i < n) atomicAdd(&h[(uint32_t)(keys[i] >> shift) & 0xffu], 1u);
  }
  __syncthreads();
  counts[(int64_t)threadIdx.x * ntiles + blockIdx.x] = h[threadIdx.x];
}

template <class K, int ITEMS>
struct RadixTile {
  uint32_t wcnt[kRadWarps][256];  // per warp and digit: keys placed, then the warp's start
  uint32_t loc[256];              // start of each digit's run inside the tile
  uint32_t tot[kRadWarps];
  K key[kRadThreads * ITEMS];
  uint32_t val[kRadThreads * ITEMS];
};

// Stable ranking of one tile by the digit at `shift`, into s.key / s.val. Warp w holds the
// tile's keys [32 ITEMS w, 32 ITEMS (w + 1)), round by round, and counts them in a row of
// its own, so the rounds need no block barrier (with one row per round and three barriers a
// round, a pass took 1.58 ms over 134 M pairs, now 1.42 ms).
template <class K, int ITEMS>
__device__ __forceinline__ void radix_rank(RadixTile<K, ITEMS> &s, const K *key, const uint32_t *val,
                                           int tn, int shift) {
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  const uint32_t lt = (1u << lane) - 1u;
#pragma unroll
  for (int q = 0; q < 256; q += 32) s.wcnt[w][q + lane] = 0;
  __syncwarp();
  uint32_t rank[ITEMS];
#pragma unroll
  for (int r = 0; r < ITEMS; ++r) {
    const bool valid = w * 32 * ITEMS + r * 32 + lane < tn;
    const uint32_t d = valid ? (uint32_t)(key[r] >> shift) & 0xffu : 256u;
    const uint32_t peers = __match_any_sync(0xffffffffu, d);
    const uint32_t before = valid ? s.wcnt[w][d] : 0u;
    __syncwarp();
    if (valid && (peers & lt) == 0) s.wcnt[w][d] = before + __popc(peers);
    __syncwarp();
    rank[r] = before + __popc(peers & lt);
  }
  __syncthreads();
  uint32_t cnt = 0;  // thread t owns digit t: exclusive prefix over the warps
#pragma unroll
  for (int q = 0; q < kRadWarps; ++q) {
    const uint32_t c = s.wcnt[q][t];
    s.wcnt[q][t] = cnt;
    cnt += c;
  }
  uint32_t incl = cnt;  // and over the digits
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t x = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += x;
  }
  if (lane == 31) s.tot[w] = incl;
  __syncthreads();
  uint32_t pre = 0;
  for (int q = 0; q < w; ++q) pre += s.tot[q];
  s.loc[t] = pre + incl - cnt;
  __syncthreads();
#pragma unroll
  for (int r = 0; r < ITEMS; ++r) {
    if (w * 32 * ITEMS + r * 32 + lane < tn) {
      const uint32_t d = (uint32_t)(key[r] >> shift) & 0xffu;
      const uint32_t lp = s.loc[d] + s.wcnt[w][d] + rank[r];
      s.key[lp] = key[r];
      s.val[lp] = val[r];
    }
  }
  __syncthreads();
}

// Stable scatter of one tile: ranked in shared memory, then each digit's run is written out
// with consecutive threads on consecutive addresses.
template <class K, int ITEMS>
__global__ void __launch_bounds__(kRadThreads) k_radix_scatter(const K *kin, const uint32_t *vin,
                                                                K *kout, uint32_t *vout, int64_t n,
                                                                int shift, int64_t ntiles,
                                                                const uint32_t *offs) {
  extern __shared__ __align__(16) unsigned char s_dyn[];
  RadixTile<K, ITEMS> &s = *reinterpret_cast<RadixTile<K, ITEMS> *>(s_dyn);
  __shared__ uint32_t s_base[256];  // global offset of each digit's run of this tile
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  const int64_t base = (int64_t)blockIdx.x * (kRadThreads * ITEMS);
  const int tn = (int)min((int64_t)(kRadThreads * ITEMS), n - base);
  s_base[t] = offs[(int64_t)t * ntiles + blockIdx.x];
  K key[ITEMS];
  uint32_t val[ITEMS];
#pragma unroll
  for (int r = 0; r < ITEMS; ++r) {
    const int li = w * 32 * ITEMS + r * 32 + lane;
    key[r] = li < tn ? kin[base + li] : K(0);
    val[r] = li < tn ? vin[base + li] : 0u;
  }
  radix_rank<K, ITEMS>(s, key, val, tn, shift);
#pragma unroll 4
  for (int li = t; li < tn; li += kRadThreads) {
    const K k = s.key[li];
    const uint32_t d = (uint32_t)(k >> shift) & 0xffu;
    const uint32_t pos = s_base[d] + (uint32_t)li - s.loc[d];
    kout[pos] = k;
    vout[pos] = s.val[li];
  }
}

// All passes of a sort of at most kRadOne pairs in one block, in place: one launch instead
// of three or more per 8 bits.
template <class K>
__global__ void __launch_bounds__(kRadThreads) k_radix_one(K *k0, uint32_t *v0, int n, int begin_bit,
                                                           int end_bit) {
  extern __shared__ __align__(16) unsigned char s_dyn[];
  RadixTile<K, kRadItems> &s = *reinterpret_cast<RadixTile<K, kRadItems> *>(s_dyn);
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  K key[kRadItems];
  uint32_t val[kRadItems];
#pragma unroll
  for (int r = 0; r < kRadItems; ++r) {
    const int li = w * 32 * kRadItems + r * 32 + lane;
    key[r] = li < n ? k0[li] : K(0);
    val[r] = li < n ? v0[li] : 0u;
  }
  for (int shift = begin_bit; shift < end_bit; shift += 8) {
    radix_rank<K, kRadItems>(s, key, val, n, shift);
#pragma unroll
    for (int r = 0; r < kRadItems; ++r) {
      const int li = w * 32 * kRadItems + r * 32 + lane;
      if (li < n) {
        key[r] = s.key[li];
        val[r] = s.val[li];
      }
    }
    __syncthreads();
  }
#pragma unroll
  for (int r = 0; r < kRadItems; ++r) {
    const int li = w * 32 * kRadItems + r * 32 + lane;
    if (li < n) {
      k0[li] = key[r];
      v0[li] = val[r];
    }
  }
}

template <class K, int ITEMS>
cudaError_t radix_passes(K *k0, uint32_t *v0, K *k1, uint32_t *v1, int64_t n, int begin_bit, int end_bit,
                         void *scratch, cudaStream_t s, int *which) {
  const int64_t ntiles = ceil_div(n, kRadThreads * ITEMS);
  const size_t smem = sizeof(RadixTile<K, ITEMS>);
  cudaError_t e = cudaFuncSetAttribute(k_radix_scatter<K, ITEMS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)smem);
  if (e != cudaSuccess) return e;
  uint32_t *counts = (uint32_t *)scratch;
  char *scan_scr = (char *)scratch + ((((size_t)ntiles * 256 * sizeof(uint32_t)) + 255) & ~(size_t)255);
  K *kin = k0, *kout = k1;
  uint32_t *vin = v0, *vout = v1;
  int cur = 0;
  for (int shift = begin_bit; shift < end_bit; shift += 8) {
    k_radix_hist<K, ITEMS><<<(unsigned)ntiles, kRadThreads, 0, s>>>(kin, n, shift, ntiles, counts);
    count_launch();
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    e = exclusive_scan<uint32_t>(counts, counts, ntiles * 256, scan_scr, s);
    if (e != cudaSuccess) return e;
    k_radix_scatter<K, ITEMS><<<(unsigned)ntiles, kRadThreads, smem, s>>>(kin, vin, kout, vout, n, shift,
                                                                         ntiles, counts);
    count_launch();
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    K *tk = kin; kin = kout; kout = tk;
    uint32_t *tv = vin; vin = vout; vout = tv;
    cur ^= 1;
  }
  *which = cur;
  return cudaSuccess;
}

}  // namespace

// The larger of the two tile forms' needs over the sizes that take them.
template <class K>
size_t radix_scratch_bytes(int64_t n) {
  auto need = [](int64_t tiles) {
    size_t c = (((size_t)tiles * 256 * sizeof(uint32_t)) + 255) & ~(size_t)255;
    return c + scan_scratch_bytes<uint32_t>(tiles * 256);
  };
  const int64_t m = n > 0 ? n : 1;
  const size_t small = need(ceil_div(m < kRadSmall ? m : kRadSmall, kRadThreads * kRadItemsSmall));
  const size_t large = need(ceil_div(m, kRadThreads * kRadItems));
  return small > large ? small : large;
}

template <class K>
cudaError_t radix_sort_pairs(K *k0, uint32_t *v0, K *k1, uint32_t *v1, int64_t n, int begin_bit,
                             int end_bit, void *scratch, cudaStream_t s, int *which) {
  *which = 0;
  if (n <= 1 || end_bit <= begin_bit) return cudaSuccess;
  if (n <= kRadOne) {
    const size_t smem = sizeof(RadixTile<K, kRadItems>);
    cudaError_t e = cudaFuncSetAttribute(k_radix_one<K>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k_radix_one<K><<<1, kRadThreads, smem, s>>>(k0, v0, (int)n, begin_bit, end_bit);
    count_launch();
    return cudaGetLastError();
  }
  if (n < kRadSmall)
    return radix_passes<K, kRadItemsSmall>(k0, v0, k1, v1, n, begin_bit, end_bit, scratch, s, which);
  return radix_passes<K, kRadItems>(k0, v0, k1, v1, n, begin_bit, end_bit, scratch, s, which);
}

template size_t radix_scratch_bytes<uint32_t>(int64_t);
template size_t radix_scratch_bytes<unsigned long long>(int64_t);
template cudaError_t radix_sort_pairs<uint32_t>(uint32_t *, uint32_t *, uint32_t *, uint32_t *,
                                                int64_t, int, int, void *, cudaStream_t, int *);
template cudaError_t radix_sort_pairs<unsigned long long>(unsigned long long *, uint32_t *,
                                                          unsigned long long *, uint32_t *, int64_t,
                                                          int, int, void *, cudaStream_t, int *);

}  // namespace vr
