// Launch shapes picked by the autotuner (vr_autotune). A shape only lays the same work
// out differently over warps and registers: the arithmetic and its order are unchanged,
// so every shape gives bit-identical results.
#pragma once
#include "vr_internal.cuh"

namespace vr {

// f_l launches by halo size (members): above 65536, (4096, 65536], (N_se, 4096].
constexpr int kVBins = 3;
static_assert(sizeof(vr_ctx::vshape_last) == kVBins * sizeof(int), "one entry per bin");
constexpr uint32_t kVBinEdge0 = 65536u, kVBinEdge1 = 4096u;

// f_l kernel shapes: candidates computed side by side, register cap, warps per block.
struct VShape {
  int batch, maxreg, warps;
};
constexpr int kNVShapes = 5;
constexpr VShape kVShapes[kNVShapes] = {{4, 64, 4}, {4, 64, 8}, {4, 64, 2}, {2, 64, 4}, {8, 80, 4}};

// 6D linker shapes: warps (32-candidate tiles) per block.
constexpr int kNLShapes = 3;
constexpr int kLWarps[kNLShapes] = {4, 2, 8};

struct Tuning {
  int on = 0;                       // measure each untuned bin at its next launch
  int vshape[kVBins] = {0, 0, 0};   // chosen f_l shape per tuned bin
  int vtuned[kVBins] = {0, 0, 0};
  float vms[kVBins][kNVShapes] = {};
  int lshape = 0, ltuned = 0;       // chosen linker shape
  float lms[kNLShapes] = {};
  int force_v = -1, force_l = -1;   // every launch uses this shape (tests), -1 = off
};

// Shape index for f_l bin k / the linker under the context's tuning state. Untuned f_l
// launches of many buckets take 2 warps per block, whose places are free again sooner, of few
// buckets 4, of which more start at once. Call with 2 warps against 4, three seeds each, by
// buckets (the spread of repeated calls in brackets): 2,400 -1.2 to +0.3 % (1.5), 11,000 to
// 12,500 -2.4 to +2.0 (3), 21,000 to 28,000 -1.3 to +0.9 (4), 32,000 -0.8 to -1.0 (0.6), 38,000
// -1.0 to -1.2 (0.5), 47,000 -1.1 to -1.4 (0.2), 65,000 -1.2 to -1.5 (0.3), 187,000 (256^3 box,
// 36.9 -> 36.3 ms) -1.5 (0.1), 210,000 (catalogue, N_se 64) -1.9 (0.1).
constexpr int64_t kVManyBuckets = 32768;
constexpr int kVShapeMany = 2;
inline int vshape_for(const vr_ctx *ctx, int k, int64_t buckets = 0) {
  const Tuning *t = ctx ? ctx->tune : nullptr;
  if (t && t->force_v >= 0) return t->force_v;
  if (t && t->vtuned[k]) return t->vshape[k];
  return buckets >= kVManyBuckets ? kVShapeMany : 0;
}
// True when bin k's f_l shape follows from its launch's size: neither forced nor tuned.
inline bool vshape_by_size(const vr_ctx *ctx, int k) {
  return !ctx->tune || (ctx->tune->force_v < 0 && !ctx->tune->vtuned[k]);
}
// The f_l shape in use for bin k: forced, tuned, or what its last launch took by its size.
inline int vshape_in_use(const vr_ctx *ctx, int k) {
  return vshape_by_size(ctx, k) ? ctx->vshape_last[k] : vshape_for(ctx, k);
}
inline int lshape_for(const vr_ctx *ctx) {
  const Tuning *t = ctx ? ctx->tune : nullptr;
  if (!t) return 0;
  if (t->force_l >= 0) return t->force_l;
  return t->ltuned ? t->lshape : 0;
}
// True when the f_l bin k / the linker is to be measured at this launch.
inline bool vmeasure(const vr_ctx *ctx, int k) {
  const Tuning *t = ctx ? ctx->tune : nullptr;
  return t && t->on && t->force_v < 0 && !t->vtuned[k];
}
inline bool lmeasure(const vr_ctx *ctx) {
  const Tuning *t = ctx ? ctx->tune : nullptr;
  return t && t->on && t->force_l < 0 && !t->ltuned;
}

}  // namespace vr
