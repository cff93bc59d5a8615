// 3D friends-of-friends over a periodic lattice box (Sec. 2.1, Eq. fof3d).
//
// GB300 design:
//  1. sub-cells of side S = floor(sqrt((link_d2 - 1) / 3)) + 1, the largest side whose
//     diagonal is shorter than the linking length: all members of a sub-cell are linked
//     to each other, so each member is hooked straight below the sub-cell's first
//     particle without any distance test;
//  2. link cells of 2 sub-cells per axis (side 2S >= linking length; the last link cell
//     of each axis takes the 3 or 4 leftover sub-cells, so no link cell is thinner than
//     the linking length across the periodic edge; of 4 sub-cells for link_d2 <= 3, whose
//     S = 1 would give more link cells than the sort key has bits for): every linked pair
//     lies in the same or
//     an adjacent link cell. Particles are ordered by (Morton code of the link cell,
//     position of the sub-cell inside it) with the library's radix sort, which makes
//     every sub-cell, link cell and coarse cell (2^q link cells per axis) one contiguous
//     run;
//  3. link cells are listed in sort order (key, first sub-cell); a dense table over coarse
//     cells gives the link cells of each, so a lookup is one load and a short binary search
//     over link cells; before it, one bit per link cell (the grid folded to 2^m cells per
//     axis, 8 n bits or more, 4x4x4 cells per 64-bit word) tells most empty neighbours apart
//     in one cached load: a clear bit means an empty link cell, a set bit (the cell, or one
//     folded onto it, holds particles) goes on to the lookup;
//  4. three linking kernels over a lock-free union-find of sub-cells (atomicCAS hooks the
//     larger root under the smaller; finds halve paths):
//      - k_fof_own links the sub-cells of each link cell among themselves and marks the
//        link cells that end as one set;
//      - k_fof_neigh: a warp takes 32 consecutive link cells, screens their 13 forward
//        neighbours against the bitmap, and spreads the occupied (cell, neighbour) pairs
//        over its lanes. A pair of one-set cells that already share a root is done; a pair
//        of few members is tested by its lane; the rest go to a list;
//      - k_fof_heavy: one warp per listed pair of link cells, sub-cell pair by sub-cell
//        pair, the large ones tested by all lanes together. By then most listed pairs
//        share a root and cost two finds.
//     Pairs of sub-cells with at most 4 member pairs are tested particle by particle;
//     otherwise box distances settle most pairs (none linked / all linked), the rest are
//     skipped when A and B are already in one component, else particles are tested until a
//     linked pair is found;
//  5. labels are the minimum original index of each component (atomicMin per root).
// The grid is not a power of two per axis: the last sub-cell of each axis may be
// partial, and box tests use each cell's true extent across the periodic edge.
// Positions are gathered once into a 16-byte int4 stream in sorted order.
#include "vr_internal.cuh"
#include "vr_workspace.h"
#include "unionfind.cuh"

namespace vr {

namespace {

constexpr uint32_t kEmpty = 0xffffffffu;

struct FofGeom {
  int S;        // sub-cell side (lattice units)
  int G;        // sub-cells per axis (last one partial)
  int lw;       // a link cell is 2^lw sub-cells wide (the last one of an axis up to 4)
  int GL;       // link cells per axis
  int bl;       // bits per axis of link-cell coordinates
  int q;        // coarse cell = 2^q link cells per axis
  int64_t ncoarse;
  int om;       // occupancy bitmap: link cells folded to 2^om per axis
};

// Coarse table size: at most 8^m entries with 8^m <= max(n, 4096), m <= 9 (2^27).
int coarse_bits_per_axis(int64_t n) {
  int m = 4;
  while (m < 9 && (1LL << (3 * (m + 1))) <= n) ++m;
  return m;
}

// Occupancy bitmap: 2^(3m) bits, the smallest m >= 4 with 2^(3m) >= 8 n, m <= 11.
int occ_bits_per_axis(int64_t n) {
  int m = 4;
  while (m < 11 && (1LL << (3 * m)) < 8 * n) ++m;
  return m;
}

int64_t occ_words(int om) { return 1LL << (3 * om - 6); }

int64_t isqrt64(int64_t x) {
  int64_t r = (int64_t)sqrt((double)x);
  while (r * r > x) --r;
  while ((r + 1) * (r + 1) <= x) ++r;
  return r;
}

FofGeom fof_geom(int64_t link_d2, int64_t n) {
  FofGeom g;
  g.S = (int)isqrt64((link_d2 - 1) / 3) + 1;  // 3 (S-1)^2 <= link_d2 - 1 < link_d2
  g.G = (int)((kLattice + g.S - 1) / g.S);
  // the sort key holds 6 + 3 bl bits: 19 bits per axis at most. With S = 1 (link_d2 <= 3) link
  // cells of 2 would need 20, so they take 4, of which the 2^21 sub-cells leave no remainder
  g.lw = g.S == 1 ? 2 : 1;
  g.GL = g.S == 1 ? g.G / 4 : (g.G - 1) / 2;
  g.bl = 0;
  while ((1 << g.bl) < g.GL) ++g.bl;
  if (g.bl == 0) g.bl = 1;
  int m = coarse_bits_per_axis(n);
  g.q = g.bl - m > 0 ? g.bl - m : 0;
  g.ncoarse = 1LL << (3 * (g.bl - g.q));
  g.om = occ_bits_per_axis(n);
  return g;
}

struct FofBufs {
  u64 *k0, *k1;        // sort keys; the spare one: scan buffer, then list of heavy pairs, then
                       // minimum index per root
  uint32_t *v0, *v1;   // sort values (n + 1 each): sub-cell of each particle, and (once the
                       // positions are gathered) first sub-cell of each link cell
  int4 *posS;
  int *parent;         // union-find over sub-cells
  uint32_t *sc_start;  // first sorted index of each sub-cell
  u64 *lckey;          // key of each link cell, kOneSet in its top bit
  uint2 *ctab;         // link cells [x, y) of each coarse cell
  unsigned long long *occ;  // occupancy bitmap of the link cells
  void *scratch;       // radix sort / scan scratch, then the list's counter
};

FofBufs fof_carve(Arena &ar, int64_t n, int64_t ncoarse, int om) {
  FofBufs b;
  b.k0 = ar.take<u64>(n + 1);
  b.k1 = ar.take<u64>(n + 1);
  b.v0 = ar.take<uint32_t>(n + 1);
  b.v1 = ar.take<uint32_t>(n + 1);
  b.posS = ar.take<int4>(n);
  b.parent = ar.take<int>(n);
  b.sc_start = ar.take<uint32_t>(n + 1);
  b.lckey = ar.take<u64>(n);
  b.ctab = ar.take<uint2>(ncoarse);
  b.occ = ar.take<unsigned long long>(occ_words(om));
  size_t a = radix_scratch_bytes<u64>(n), c = scan_scratch_bytes<u64>(n + 1);
  b.scratch = ar.take<char>(a > c ? a : c);
  return b;
}

// Sub-cell c of an axis lies in link cell min(c >> lw, GL - 1) at position c - (that << lw).
__device__ __forceinline__ uint32_t link_of(uint32_t c, int lw, int GL) {
  uint32_t l = c >> lw;
  return l < (uint32_t)GL ? l : (uint32_t)GL - 1u;
}

// Word and bit of link cell (x, y, z) in the occupancy bitmap: coordinates taken modulo
// 2^om, then 4x4x4 cells per 64-bit word, words in x-fastest order.
__device__ __forceinline__ void occ_pos(uint32_t x, uint32_t y, uint32_t z, int om, u64 &word,
                                        uint32_t &bit) {
  const uint32_t M = (1u << om) - 1u;
  x &= M;
  y &= M;
  z &= M;
  const int b = om - 2;
  word = (u64)(x >> 2) | ((u64)(y >> 2) << b) | ((u64)(z >> 2) << (2 * b));
  bit = (x & 3u) | ((y & 3u) << 2) | ((z & 3u) << 4);
}

__device__ __forceinline__ uint32_t compact3(u64 x);

// Sort key: Morton code of the link cell << 6 | 2-bit sub-cell position per axis. Link
// cells (key >> 6) and coarse cells are its prefixes.
__global__ void k_fof_keys(const int32_t *__restrict__ pos, int64_t n, int S, int lw, int GL,
                           u64 *__restrict__ keys, uint32_t *__restrict__ vals) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  // masking keeps every cell index in range even for positions outside [0, 2^21)
  const uint32_t m = (uint32_t)kLattice - 1u;
  uint32_t x = ((uint32_t)pos[3 * i] & m) / (uint32_t)S,
           y = ((uint32_t)pos[3 * i + 1] & m) / (uint32_t)S,
           z = ((uint32_t)pos[3 * i + 2] & m) / (uint32_t)S;
  uint32_t lx = link_of(x, lw, GL), ly = link_of(y, lw, GL), lz = link_of(z, lw, GL);
  keys[i] = (morton3(lx, ly, lz) << 6) | ((u64)(x - (lx << lw)) << 4) | ((u64)(y - (ly << lw)) << 2) |
            (u64)(z - (lz << lw));
  vals[i] = (uint32_t)i;
}


// Positions in sorted order, and per particle the two start flags to be scanned together:
// high word 1 at the first particle of a sub-cell, low word 1 at that of a link cell.
__global__ void k_fof_prepare(const int32_t *__restrict__ pos, const u64 *__restrict__ keyS,
                              const uint32_t *__restrict__ orig, int64_t n,
                              int4 *__restrict__ posS, u64 *__restrict__ flag) {
  int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p > n) return;
  if (p == n) {
    flag[n] = 0;
    return;
  }
  int64_t i = orig[p];
  const uint32_t m = (uint32_t)kLattice - 1u;
  posS[p] = make_int4((int)((uint32_t)pos[3 * i] & m), (int)((uint32_t)pos[3 * i + 1] & m),
                      (int)((uint32_t)pos[3 * i + 2] & m), (int)i);
  const u64 d = p == 0 ? ~0ull : keyS[p - 1] ^ keyS[p];
  flag[p] = d == 0 ? 0ull : ((1ull << 32) | (d >> 6 ? 1ull : 0ull));
}

// excl = the exclusive scan of the flags. Sub-cell of every particle, start of every
// sub-cell (sc_start[nsc] = n), key and first sub-cell of every link cell (lcfirst[nlc] =
// nsc), link cells of every coarse cell, the occupancy bitmap, and one set per sub-cell:
// all its members are within the linking length of each other (3 (S-1)^2 < link_d2).
__global__ void k_fof_cells(const u64 *__restrict__ keyS, const u64 *__restrict__ excl, int64_t n,
                            int cshift, uint32_t *__restrict__ sid, uint32_t *__restrict__ sc_start,
                            uint32_t *__restrict__ lcfirst, u64 *__restrict__ lckey,
                            uint2 *__restrict__ ctab, unsigned long long *__restrict__ occ, int om,
                            int *__restrict__ parent) {
  int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= n) return;
  const u64 e = excl[p], k = keyS[p];
  const u64 d = p == 0 ? ~0ull : keyS[p - 1] ^ k;
  const uint32_t sub = (uint32_t)(e >> 32) - (d ? 0u : 1u);
  sid[p] = sub;
  if (d) {
    sc_start[sub] = (uint32_t)p;
    parent[sub] = (int)sub;
  }
  if (d >> 6) {  // first particle of its link cell
    const uint32_t c = (uint32_t)e;
    lcfirst[c] = sub;
    lckey[c] = k >> 6;
    u64 w;
    uint32_t bit;
    occ_pos(compact3(k >> 6), compact3(k >> 7), compact3(k >> 8), om, w, bit);
    atomicOr(&occ[w], 1ull << bit);
    if (p == 0 || (d >> cshift)) {  // and of its coarse cell
      ctab[k >> cshift].x = c;
      if (p > 0) ctab[keyS[p - 1] >> cshift].y = c;
    }
  }
  if (p == n - 1) {
    const u64 t = excl[n];
    sc_start[(uint32_t)(t >> 32)] = (uint32_t)n;
    lcfirst[(uint32_t)t] = (uint32_t)(t >> 32);
    ctab[k >> cshift].y = (uint32_t)t;
  }
}

__device__ __forceinline__ long long d2_periodic(int4 a, int4 b) {
  long long dx = min_image(a.x - b.x), dy = min_image(a.y - b.y), dz = min_image(a.z - b.z);
  return dx * dx + dy * dy + dz * dz;
}

// Forward half of the 26-neighbourhood: (dz > 0) or (dz == 0 and dy > 0) or
// (dz == 0, dy == 0, dx > 0). With >= 3 link cells per axis each unordered pair of
// adjacent cells is visited from exactly one side.
__constant__ signed char c_fwd[13][3] = {
    {1, 0, 0},  {-1, 1, 0}, {0, 1, 0},  {1, 1, 0},  {-1, -1, 1}, {0, -1, 1}, {1, -1, 1},
    {-1, 0, 1}, {0, 0, 1},  {1, 0, 1},  {-1, 1, 1}, {0, 1, 1},   {1, 1, 1}};

// Sub-cell extent along one axis: [c S, min((c + 1) S, 2^21) - 1].
__device__ __forceinline__ void cell_span(int c, int S, int &lo, int &hi) {
  lo = c * S;
  hi = min(lo + S, (int)kLattice) - 1;
}

// Gap and farthest separation between interval A = [alo, ahi] and interval B = [blo, bhi]
// taken in B's periodic image nearest to A. Returns B's shift into A's frame.
__device__ __forceinline__ int axis_gap(int alo, int ahi, int blo, int bhi, long long &gap,
                                        long long &far) {
  int shift = min_image(blo - alo) - (blo - alo);
  int b0 = blo + shift, b1 = bhi + shift;
  long long g = 0;
  if (b0 > ahi) g = (long long)b0 - ahi;
  else if (alo > b1) g = (long long)alo - b1;
  long long f1 = (long long)b1 - alo, f2 = (long long)ahi - b0;
  gap = g;
  far = f1 > f2 ? f1 : f2;
  return shift;
}

__device__ __forceinline__ uint32_t compact3(u64 x) {  // every third bit of x, from bit 0
  x &= 0x1249249249249249ULL;
  x = (x ^ (x >> 2)) & 0x10c30c30c30c30c3ULL;
  x = (x ^ (x >> 4)) & 0x100f00f00f00f00fULL;
  x = (x ^ (x >> 8)) & 0x1f0000ff0000ffULL;
  x = (x ^ (x >> 16)) & 0x1f00000000ffffULL;
  x = (x ^ (x >> 32)) & 0x1fffffULL;
  return (uint32_t)x;
}


// Pairs of sub-cells with at most this many member pairs are tested particle by particle,
// without the box tests; those of more than kSerialPairs by a whole warp.
constexpr uint32_t kDirectPairs = 4, kSerialPairs = 64;
// Link-cell pairs of at most this many member pairs are tested where they are found, their
// member pairs spread over the warp; larger ones are listed for a warp of their own.
constexpr uint32_t kLanePairs = 64;
constexpr u64 kOneSet = 1ull << 63;  // lckey: the link cell's sub-cells are all in one set

struct FofCells {
  const int4 *posS;
  const u64 *keyS;
  const uint32_t *sc_start, *lcfirst;
  const uint32_t *sid;
  const uint2 *ctab;
  const unsigned long long *occ;
  int om, S, lw, GL, qshift;
  long long T;
};

// Extent of sub-cell coordinates (l << lw) + (2-bit position of the sort key) per axis.
__device__ __forceinline__ void sub_box(u64 key, const int *l, int lw, int S, int *lo, int *hi) {
  cell_span((l[0] << lw) + (int)((key >> 4) & 3u), S, lo[0], hi[0]);
  cell_span((l[1] << lw) + (int)((key >> 2) & 3u), S, lo[1], hi[1]);
  cell_span((l[2] << lw) + (int)(key & 3u), S, lo[2], hi[2]);
}

// Squared distance from x (inside A's box) to box B in A's frame.
__device__ __forceinline__ long long box_gap2(int4 x, const int *bl, const int *bh) {
  const long long gx = x.x < bl[0] ? bl[0] - x.x : (x.x > bh[0] ? x.x - bh[0] : 0);
  const long long gy = x.y < bl[1] ? bl[1] - x.y : (x.y > bh[1] ? x.y - bh[1] : 0);
  const long long gz = x.z < bl[2] ? bl[2] - x.z : (x.z > bh[2] ? x.z - bh[2] : 0);
  return gx * gx + gy * gy + gz * gz;
}

// Boxes of sub-cells A and B (first particles a0, b0; link-cell coordinates la, lb), B
// shifted into A's frame: smallest and largest squared separation of their points.
__device__ __forceinline__ void pair_boxes(const FofCells &f, uint32_t a0, const int *la, uint32_t b0,
                                           const int *lb, int *bl, int *bh, long long &mind,
                                           long long &maxd) {
  int alo[3], ahi[3], lo[3], hi[3];
  sub_box(f.keyS[a0], la, f.lw, f.S, alo, ahi);
  sub_box(f.keyS[b0], lb, f.lw, f.S, lo, hi);
  mind = maxd = 0;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    long long gp, fr;
    const int sh = axis_gap(alo[k], ahi[k], lo[k], hi[k], gp, fr);
    bl[k] = lo[k] + sh;
    bh[k] = hi[k] + sh;
    mind += gp * gp;
    maxd += fr * fr;
  }
}

// All member pairs of sub-cells A and B, until one is within the linking length.
__device__ __forceinline__ bool any_pair(const FofCells &f, uint32_t a0, uint32_t a1, uint32_t b0,
                                         uint32_t b1) {
  for (uint32_t a = a0; a < a1; ++a) {
    const int4 xa = f.posS[a];
    for (uint32_t b = b0; b < b1; ++b)
      if (d2_periodic(xa, f.posS[b]) < f.T) return true;
  }
  return false;
}

// Links every sub-cell pair of link cells A = sub-cells [sa0, sa1) at la and B at lb (or
// the pairs inside A when `own`) with a whole warp: the pairs spread over the lanes, the
// large ones then tested by all lanes. `once`: A and B are one set each, so the first link
// ends it.
__device__ void link_cells_warp(const FofCells &f, int *parent, uint32_t sa0, uint32_t sa1,
                                const int *la, uint32_t sb0, uint32_t sb1, const int *lb, bool own,
                                bool once) {
  const int lane = threadIdx.x & 31;
  const unsigned FULL = 0xffffffffu;
  const uint32_t mb = sb1 - sb0, total = (sa1 - sa0) * mb;
  for (uint32_t t0 = 0; t0 < total; t0 += 32) {
    const uint32_t t = t0 + lane;
    const uint32_t i = t / mb, j = t - i * mb;
    const uint32_t sa = sa0 + i, sb = sb0 + j;
    bool linked = false, large = false;
    if (t < total && (!own || i < j)) {
      const uint32_t a0 = f.sc_start[sa], a1 = f.sc_start[sa + 1], b0 = f.sc_start[sb],
                     b1 = f.sc_start[sb + 1];
      const u64 np = (u64)(a1 - a0) * (b1 - b0);
      if (np <= kDirectPairs) {
        linked = any_pair(f, a0, a1, b0, b1);
        if (linked) uf_unite(parent, (int)sa, (int)sb);
      } else {
        int bl[3], bh[3];
        long long mind, maxd;
        pair_boxes(f, a0, la, b0, lb, bl, bh, mind, maxd);
        if (mind < f.T) {
          if (maxd < f.T) {
            uf_unite(parent, (int)sa, (int)sb);
            linked = true;
          } else if (uf_find(parent, (int)sa) == uf_find(parent, (int)sb)) {
            linked = true;
          } else if (np <= kSerialPairs) {
            for (uint32_t a = a0; a < a1 && !linked; ++a) {
              const int4 xa = f.posS[a];  // inside A's box, so no wrap in A's frame
              if (box_gap2(xa, bl, bh) >= f.T) continue;
              for (uint32_t b = b0; b < b1 && !linked; ++b) linked = d2_periodic(xa, f.posS[b]) < f.T;
            }
            if (linked) uf_unite(parent, (int)sa, (int)sb);
          } else {
            large = true;
          }
        }
      }
    }
    if (once && __any_sync(FULL, linked)) return;
    unsigned lm = __ballot_sync(FULL, large);
    while (lm) {
      const int src = __ffs(lm) - 1;
      lm &= lm - 1;
      const uint32_t ua = __shfl_sync(FULL, sa, src), ub = __shfl_sync(FULL, sb, src);
      int same = 0;
      if (lane == 0) same = uf_find(parent, (int)ua) == uf_find(parent, (int)ub);
      if (__shfl_sync(FULL, same, 0)) {
        if (once) return;
        continue;
      }
      const uint32_t a0 = f.sc_start[ua], a1 = f.sc_start[ua + 1], b0 = f.sc_start[ub],
                     b1 = f.sc_start[ub + 1];
      int bl[3], bh[3];
      long long mind, maxd;
      pair_boxes(f, a0, la, b0, lb, bl, bh, mind, maxd);
      bool found = false;
      for (uint32_t ab = a0; ab < a1 && !found; ab += 32) {  // a member of A per lane ...
        const uint32_t a = ab + lane;
        int4 xa = make_int4(0, 0, 0, 0);
        bool near = false;
        if (a < a1) {
          xa = f.posS[a];
          near = box_gap2(xa, bl, bh) < f.T;
        }
        unsigned nm = __ballot_sync(FULL, near);
        while (nm && !found) {  // ... those within reach of B's box against B's members
          const int s = __ffs(nm) - 1;
          nm &= nm - 1;
          const int4 x = make_int4(__shfl_sync(FULL, xa.x, s), __shfl_sync(FULL, xa.y, s),
                                   __shfl_sync(FULL, xa.z, s), 0);
          bool hit = false;
          for (uint32_t b = b0 + lane; b < b1 && !hit; b += 32) hit = d2_periodic(x, f.posS[b]) < f.T;
          found = __any_sync(FULL, hit);
        }
      }
      if (found) {
        if (lane == 0) uf_unite(parent, (int)ua, (int)ub);
        if (once) return;
      }
    }
  }
}

// Tests the member pairs of up to 32 pairs of particle runs, one pair of runs per lane (w =
// its member pairs, 0: none): the pairs of all lanes follow one another, and each step takes
// the next 32. Lanes that walked their own few pairs left two thirds of the warp idle
// (k_fof_neigh at 512^3, then: 23.0 ms, 17.5 so). A run paired with itself takes i < j only.
__device__ __forceinline__ void link_runs(const FofCells &f, int *parent, uint32_t a0, uint32_t b0,
                                          uint32_t nb, uint32_t w) {
  const int lane = threadIdx.x & 31;
  const unsigned FULL = 0xffffffffu;
  uint32_t incl = w;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(FULL, incl, o);
    if (lane >= o) incl += y;
  }
  const uint32_t total = __shfl_sync(FULL, incl, 31);
  for (uint32_t base = 0; base < total; base += 32) {
    const uint32_t t = base + lane;
    int o = 0;  // the lane that holds pair t: the first whose inclusive count exceeds it
#pragma unroll
    for (int s = 16; s; s >>= 1)
      if (__shfl_sync(FULL, incl, o + s - 1) <= t) o += s;
    const uint32_t at = t - __shfl_sync(FULL, incl - w, o), m = __shfl_sync(FULL, nb, o);
    const uint32_t xa = __shfl_sync(FULL, a0, o), xb = __shfl_sync(FULL, b0, o);
    if (t < total) {
      const uint32_t i = at / m, j = at - i * m;
      const uint32_t a = xa + i, b = xb + j;
      if ((xa != xb || i < j) && d2_periodic(f.posS[a], f.posS[b]) < f.T) {
        const int sa = (int)f.sid[a], sb = (int)f.sid[b];
        if (sa != sb) uf_unite(parent, sa, sb);
      }
    }
  }
}

// Pairs of sub-cells of one link cell; a warp takes `per` link cells at a time, the cells of
// more than kLanePairs member pairs go to the list (as pairs with themselves): a run of
// dense link cells is a run in sort order too, and left with the warp that holds it it was
// the kernel's last 1 ms at 256^3.
constexpr int kLW = 4;  // warps per block of the link kernels
__global__ void __launch_bounds__(32 * kLW) k_fof_own(FofCells f, const u64 *__restrict__ excl_n,
                                                      u64 *__restrict__ lckey, int *parent,
                                                      uint2 *__restrict__ heavy,
                                                      uint32_t *__restrict__ nheavy, int per) {
  const int lane = threadIdx.x & 31;
  const unsigned FULL = 0xffffffffu;
  const int64_t nlc = (uint32_t)*excl_n;
  for (int64_t c0 = ((int64_t)blockIdx.x * kLW + (threadIdx.x >> 5)) * per; c0 < nlc;
       c0 += (int64_t)gridDim.x * kLW * per) {
    const int64_t c = c0 + lane;
    uint32_t s0 = 0, s1 = 0, p0 = 0, np = 0, w = 0;
    if (lane < per && c < nlc) {
      s0 = f.lcfirst[c];
      s1 = f.lcfirst[c + 1];
      if (s1 - s0 > 1) {
        p0 = f.sc_start[s0];
        np = f.sc_start[s1] - p0;
        w = (u64)np * np > 2 * kLanePairs ? 0 : np * np;
      }
    }
    const unsigned lm = __ballot_sync(FULL, np > 0 && w == 0);
    if (lm) {
      uint32_t at = 0;
      if (lane == 0) at = atomicAdd(nheavy, (uint32_t)__popc(lm));
      at = __shfl_sync(FULL, at, 0) + (uint32_t)__popc(lm & ((1u << lane) - 1u));
      if (np > 0 && w == 0) heavy[at] = make_uint2((uint32_t)c, (uint32_t)c);  // at most one per cell
    }
    if (__any_sync(FULL, w > 0)) {
      link_runs(f, parent, p0, p0, np > 0 ? np : 1, w);
      __syncwarp();
    }
    bool one = s1 - s0 == 1;
    if (w > 0) {  // one set: every sub-cell has the first one's root
      const int r = uf_find(parent, (int)s0);
      one = true;
      for (uint32_t i = s0 + 1; i < s1 && one; ++i) one = uf_find(parent, (int)i) == r;
    }
    if (one) lckey[c] |= kOneSet;
  }
}

// The listed link cells, one warp each.
__global__ void __launch_bounds__(32 * kLW) k_fof_own_heavy(FofCells f, u64 *__restrict__ lckey,
                                                            int *parent, const uint2 *__restrict__ heavy,
                                                            const uint32_t *__restrict__ nheavy) {
  const int lane = threadIdx.x & 31;
  const unsigned FULL = 0xffffffffu;
  const uint32_t n = *nheavy;
  for (u64 k = (u64)blockIdx.x * kLW + (threadIdx.x >> 5); k < n; k += (u64)gridDim.x * kLW) {
    const uint32_t c = heavy[k].x;
    const uint32_t s0 = f.lcfirst[c], s1 = f.lcfirst[c + 1];
    const u64 key = lckey[c];
    const int l[3] = {(int)compact3(key), (int)compact3(key >> 1), (int)compact3(key >> 2)};
    link_cells_warp(f, parent, s0, s1, l, s0, s1, l, true, false);
    __syncwarp();
    bool one = true;
    const int r = uf_find(parent, (int)s0);
    for (uint32_t i = s0 + lane; i < s1; i += 32) one = one && uf_find(parent, (int)i) == r;
    if (__all_sync(FULL, one) && lane == 0) lckey[c] = key | kOneSet;
  }
}

// Link cell with key `key`, or kEmpty.
__device__ __forceinline__ uint32_t find_cell(const FofCells &f, const u64 *__restrict__ lckey, u64 key) {
  const uint2 r = __ldg(&f.ctab[key >> f.qshift]);
  if (r.x == kEmpty) return kEmpty;
  uint32_t lo = r.x, hi = r.y;
  while (lo < hi) {
    const uint32_t mid = (lo + hi) >> 1;
    if ((__ldg(&lckey[mid]) & ~kOneSet) < key) lo = mid + 1; else hi = mid;
  }
  return lo < r.y && (__ldg(&lckey[lo]) & ~kOneSet) == key ? lo : kEmpty;
}

__device__ __forceinline__ void fwd_cell(const int *l, int q, int GL, int *o) {
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const int x = l[a] + c_fwd[q][a];
    o[a] = x < 0 ? x + GL : (x >= GL ? x - GL : x);
  }
}

// Pairs of adjacent link cells, as described at the top. Each warp takes `per` consecutive
// link cells at a time: 32, fewer for a small box, whose few link cells would leave most
// warp slots empty (32^3: 197 -> 67 us).
__global__ void __launch_bounds__(32 * kLW, 12) k_fof_neigh(FofCells f, const u64 *__restrict__ excl_n,
                                                        const u64 *__restrict__ lckey, int *parent,
                                                        uint2 *__restrict__ heavy, uint32_t cap,
                                                        uint32_t *__restrict__ nheavy, int per) {
  __shared__ uint16_t s_task[kLW][32 * 13];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const unsigned FULL = 0xffffffffu;
  const int64_t nlc = (uint32_t)*excl_n;
  for (int64_t c0 = ((int64_t)blockIdx.x * kLW + w) * per; c0 < nlc; c0 += (int64_t)gridDim.x * kLW * per) {
    uint32_t bits = 0;
    int l[3] = {0, 0, 0};
    u64 k = 0;
    if (lane < per && c0 + lane < nlc) {
      k = lckey[c0 + lane];
      l[0] = (int)compact3(k);
      l[1] = (int)compact3(k >> 1);
      l[2] = (int)compact3(k >> 2);
#pragma unroll
      for (int q = 0; q < 13; ++q) {
        int o[3];
        fwd_cell(l, q, f.GL, o);
        u64 ow;
        uint32_t ob;
        occ_pos((uint32_t)o[0], (uint32_t)o[1], (uint32_t)o[2], f.om, ow, ob);
        bits |= (uint32_t)((__ldg(&f.occ[ow]) >> ob) & 1ull) << q;
      }
    }
    // the occupied (cell, neighbour) pairs of the 32 cells, one after the other
    const int mine = __popc(bits);
    int incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(FULL, incl, o);
      if (lane >= o) incl += y;
    }
    const int ntask = __shfl_sync(FULL, incl, 31);
    for (int at = incl - mine; bits; bits &= bits - 1) s_task[w][at++] = (uint16_t)(lane * 16 + __ffs(bits) - 1);
    __syncwarp();
    for (int t0 = 0; t0 < ntask; t0 += 32) {
      const int t = t0 + lane;
      uint32_t ca = 0, cb = kEmpty, p0 = 0, q0 = 0, nq = 1, wk = 0;
      bool list = false;
      const int task = t < ntask ? s_task[w][t] : 0;
      const u64 ka = __shfl_sync(FULL, k, task >> 4);
      const int la[3] = {__shfl_sync(FULL, l[0], task >> 4), __shfl_sync(FULL, l[1], task >> 4),
                         __shfl_sync(FULL, l[2], task >> 4)};
      if (t < ntask) {
        ca = (uint32_t)c0 + (uint32_t)(task >> 4);
        int o[3];
        fwd_cell(la, task & 15, f.GL, o);
        cb = find_cell(f, lckey, morton3((uint32_t)o[0], (uint32_t)o[1], (uint32_t)o[2]));
        if (cb != kEmpty) {
          const bool once = (ka & __ldg(&lckey[cb]) & kOneSet) != 0;
          const uint32_t sa0 = f.lcfirst[ca], sa1 = f.lcfirst[ca + 1], sb0 = f.lcfirst[cb],
                         sb1 = f.lcfirst[cb + 1];
          const uint32_t a0 = f.sc_start[sa0], a1 = f.sc_start[sa1], b0 = f.sc_start[sb0],
                         b1 = f.sc_start[sb1];
          if ((a1 - a0) == 1 && (b1 - b0) == 1) {
            if (d2_periodic(f.posS[a0], f.posS[b0]) < f.T) uf_unite(parent, (int)sa0, (int)sb0);
          } else if (!(once && uf_find(parent, (int)sa0) == uf_find(parent, (int)sb0))) {
            if ((u64)(a1 - a0) * (b1 - b0) <= kLanePairs) {
              p0 = a0;
              q0 = b0;
              nq = b1 - b0;
              wk = (a1 - a0) * nq;
            } else {
              list = true;
            }
          }
        }
      }
      if (__any_sync(FULL, wk > 0)) link_runs(f, parent, p0, q0, nq, wk);
      const unsigned lm = __ballot_sync(FULL, list);
      if (lm) {
        uint32_t at = 0;
        if (lane == 0) at = atomicAdd(nheavy, (uint32_t)__popc(lm));
        at = __shfl_sync(FULL, at, 0) + (uint32_t)__popc(lm & ((1u << lane) - 1u));
        if (list && at < cap) heavy[at] = make_uint2(ca, cb);
        unsigned om = __ballot_sync(FULL, list && at >= cap);  // list full: linked here
        while (om) {
          const int src = __ffs(om) - 1;
          om &= om - 1;
          const uint32_t xa = __shfl_sync(FULL, ca, src), xb = __shfl_sync(FULL, cb, src);
          const u64 k0 = lckey[xa], k1 = lckey[xb];
          const int x0[3] = {(int)compact3(k0), (int)compact3(k0 >> 1), (int)compact3(k0 >> 2)};
          const int x1[3] = {(int)compact3(k1), (int)compact3(k1 >> 1), (int)compact3(k1 >> 2)};
          link_cells_warp(f, parent, f.lcfirst[xa], f.lcfirst[xa + 1], x0, f.lcfirst[xb],
                          f.lcfirst[xb + 1], x1, false, (k0 & k1 & kOneSet) != 0);
          __syncwarp();
        }
      }
    }
    __syncwarp();  // s_task is rewritten for the next 32 cells
  }
}

// The listed pairs of link cells, one warp each.
__global__ void __launch_bounds__(32 * kLW) k_fof_heavy(FofCells f, const u64 *__restrict__ lckey,
                                                        int *parent, const uint2 *__restrict__ heavy,
                                                        uint32_t cap, const uint32_t *__restrict__ nheavy) {
  const uint32_t n = min(*nheavy, cap);
  for (u64 k = (u64)blockIdx.x * kLW + (threadIdx.x >> 5); k < n; k += (u64)gridDim.x * kLW) {
    const uint2 c = heavy[k];
    const u64 ka = lckey[c.x], kb = lckey[c.y];
    const bool once = (ka & kb & kOneSet) != 0;
    const uint32_t sa0 = f.lcfirst[c.x], sb0 = f.lcfirst[c.y];
    if (once) {
      int same = 0;
      if ((threadIdx.x & 31) == 0) same = uf_find(parent, (int)sa0) == uf_find(parent, (int)sb0);
      if (__shfl_sync(0xffffffffu, same, 0)) continue;
    }
    const int la[3] = {(int)compact3(ka), (int)compact3(ka >> 1), (int)compact3(ka >> 2)};
    const int lb[3] = {(int)compact3(kb), (int)compact3(kb >> 1), (int)compact3(kb >> 2)};
    link_cells_warp(f, parent, sa0, f.lcfirst[c.x + 1], la, sb0, f.lcfirst[c.y + 1], lb, false, once);
    __syncwarp();
  }
}

// Root of every sub-cell and the minimum original index per root. A sub-cell's particles
// follow one another in sort order: the first one in a warp finds the root for the others, and
// only the sub-cell's first particle writes it (with a find that halves paths and a store per
// particle, the 37,000 particles of each of 8 sub-cells kept one word's stores and loads waiting
// for each other: 300,000 particles in one clump 455 us, now 9.4). Neighbours in sort order mostly
// share a root too, so the lanes of a warp with the same root combine their minimum first and
// one of them updates the root (one atomic per root and warp).
__global__ void k_fof_roots(int *parent, const uint32_t *__restrict__ sid,
                            const int4 *__restrict__ posS, int64_t n, uint32_t *__restrict__ minidx) {
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int lane = threadIdx.x & 31;
  const bool valid = p < n;
  const int s = valid ? (int)sid[p] : -1;
  const int before = __shfl_up_sync(0xffffffffu, s, 1);
  const bool lead = lane == 0 || s != before;
  int r = -1 - lane;
  uint32_t w = 0xffffffffu;
  if (valid) {
    w = (uint32_t)posS[p].w;
    if (lead) {
      r = uf_root(parent, s);
      if (p == 0 || lane > 0 || (int)sid[p - 1] != s) parent[s] = r;
    }
  }
  // the run's first lane has the root (lanes beyond n follow a run of their own)
  const unsigned leads = __ballot_sync(0xffffffffu, lead) & (0xffffffffu >> (31 - lane));
  r = __shfl_sync(0xffffffffu, r, 31 - __clz(leads));
  const unsigned peers = __match_any_sync(0xffffffffu, r);
  const uint32_t m = __reduce_min_sync(peers, w);
  if (valid && lane == __ffs(peers) - 1) atomicMin(&minidx[r], m);
}

// A fresh find: parent[s] written by k_fof_roots may since have been overwritten by a
// concurrent path-halving store with an older ancestor, so it is not read directly.
__global__ void k_fof_label(int *parent, const uint32_t *__restrict__ sid,
                            const int4 *__restrict__ posS, const uint32_t *__restrict__ minidx,
                            int64_t n, int32_t *__restrict__ label) {
  int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= n) return;
  label[posS[p].w] = (int32_t)minidx[uf_find(parent, (int)sid[p])];
}

}  // namespace

size_t ws_fof3d(int64_t n) {
  Arena ar;
  fof_carve(ar, n, 1LL << (3 * coarse_bits_per_axis(n)), occ_bits_per_axis(n));
  return ar.off;
}

}  // namespace vr

using namespace vr;

extern "C" vr_status vr_fof3d(vr_ctx *ctx, const int32_t *pos, int64_t n, int64_t link_d2,
                              int32_t *label, void *ws, size_t ws_bytes, void *stream) {
  if (!ctx) return VR_ERR_INVALID_ARG;
  if (n < 0 || n >= (1LL << 31))
    return set_error(ctx, VR_ERR_INVALID_ARG, "n must be in [0, 2^31)");
  if (n == 0) return VR_OK;
  if (!pos || !label || !ws) return set_error(ctx, VR_ERR_INVALID_ARG, "NULL pointer");
  if (link_d2 < 1 || link_d2 > (1LL << 38))
    return set_error(ctx, VR_ERR_INVALID_ARG, "link_d2 must be in [1, 2^38]");
  cudaStream_t s = (cudaStream_t)stream;
  FofGeom g = fof_geom(link_d2, n);
  Arena ar(ws, ws_bytes);
  FofBufs B = fof_carve(ar, n, g.ncoarse, g.om);
  vr_status st = check_ws(ctx, ar, ws_bytes);
  if (st != VR_OK) return st;
  const int T = 256;
  k_fof_keys<<<grid_for(n, T), T, 0, s>>>(pos, n, g.S, g.lw, g.GL, B.k0, B.v0);
  VR_LAUNCHED(ctx, "k_fof_keys");
  int which = 0;
  VR_CUDA(ctx, radix_sort_pairs<u64>(B.k0, B.v0, B.k1, B.v1, n, 0, 6 + 3 * g.bl, B.scratch, s,
                                     &which));
  u64 *keyS = which ? B.k1 : B.k0;
  uint32_t *orig = which ? B.v1 : B.v0;
  VR_CUDA(ctx, cudaMemsetAsync(B.ctab, 0xff, g.ncoarse * sizeof(uint2), s));
  VR_CUDA(ctx, cudaMemsetAsync(B.occ, 0, occ_words(g.om) * sizeof(unsigned long long), s));
  const int qshift = 3 * g.q;      // link-cell key -> coarse-cell key
  const int cshift = 6 + qshift;   // sort key -> coarse-cell key
  u64 *spare = which ? B.k0 : B.k1;
  k_fof_prepare<<<grid_for(n + 1, T), T, 0, s>>>(pos, keyS, orig, n, B.posS, spare);
  VR_LAUNCHED(ctx, "k_fof_prepare");
  VR_CUDA(ctx, exclusive_scan<u64>(spare, spare, n + 1, B.scratch, s));
  uint32_t *sid = which ? B.v0 : B.v1;  // the sort's spare value buffer
  uint32_t *lcfirst = orig;             // posS holds the particle indices now
  k_fof_cells<<<grid_for(n, T), T, 0, s>>>(keyS, spare, n, cshift, sid, B.sc_start, lcfirst, B.lckey,
                                           B.ctab, B.occ, g.om, B.parent);
  VR_LAUNCHED(ctx, "k_fof_cells");
  int sms = ctx->sm_count;
  if (sms <= 0) VR_CUDA(ctx, cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, ctx->device));
  // the scanned flags stay until the link kernels have read their last entry; the list of
  // heavy pairs takes the entries before it
  uint32_t *nheavy = reinterpret_cast<uint32_t *>(B.scratch);
  uint2 *heavy = reinterpret_cast<uint2 *>(spare);
  VR_CUDA(ctx, cudaMemsetAsync(nheavy, 0, 2 * sizeof(uint32_t), s));
  FofCells f{B.posS, keyS, B.sc_start, lcfirst, sid, B.ctab, B.occ, g.om, g.S, g.lw, g.GL, qshift, (long long)link_d2};
  // link cells a warp takes at a time (n bounds their number): 32, or 64 warps per SM. Each
  // warp takes two such runs; more blocks than fit at once let the dense regions, which lie
  // together in sort order, spread over the SMs (k_fof_neigh at 512^3 with the resident
  // blocks only 17.5 ms, 13.2 so)
  int per = 4;
  while (per < 32 && n > 64LL * sms * per) per *= 2;
  const unsigned hgrid = (unsigned)grid_for(n, 32 * kLW, 64LL * sms);
  timer_begin(ctx, "fof_link", s);
  k_fof_own<<<(unsigned)grid_for(n, 2 * per * kLW), 32 * kLW, 0, s>>>(f, spare + n, B.lckey, B.parent,
                                                                           heavy, nheavy, per);
  VR_LAUNCHED(ctx, "k_fof_own");
  k_fof_own_heavy<<<hgrid, 32 * kLW, 0, s>>>(f, B.lckey, B.parent, heavy, nheavy);
  VR_LAUNCHED(ctx, "k_fof_own_heavy");
  k_fof_neigh<<<(unsigned)grid_for(n, 2 * per * kLW), 32 * kLW, 0, s>>>(
      f, spare + n, B.lckey, B.parent, heavy, (uint32_t)n, nheavy + 1, per);
  VR_LAUNCHED(ctx, "k_fof_neigh");
  k_fof_heavy<<<hgrid, 32 * kLW, 0, s>>>(f, B.lckey, B.parent, heavy, (uint32_t)n, nheavy + 1);
  VR_LAUNCHED(ctx, "k_fof_heavy");
  timer_end(ctx, "fof_link", s);
  uint32_t *minidx = reinterpret_cast<uint32_t *>(spare);  // the list is done
  VR_CUDA(ctx, cudaMemsetAsync(minidx, 0xff, n * sizeof(uint32_t), s));
  k_fof_roots<<<grid_for(n, T), T, 0, s>>>(B.parent, sid, B.posS, n, minidx);
  VR_LAUNCHED(ctx, "k_fof_roots");
  k_fof_label<<<grid_for(n, T), T, 0, s>>>(B.parent, sid, B.posS, minidx, n, label);
  VR_LAUNCHED(ctx, "k_fof_label");
  return log_call(ctx, "vr_fof3d", n, VR_OK);
}
