// batch_launch.cuh -- launch of one bucket of the batched evaluation kernel (shared by the minimal-form
// launchers in batch.cu and the Tersoff-form launchers in batch_gen.cu).
#pragma once
#include <algorithm>

#include "batch_kernel.cuh"

namespace tsf {

constexpr int kPT = 32;   // parameter sets per warp in FP32: one atom per warp
// FP64: four atoms x eight parameter sets per warp. The FP64 unit bounds those kernels whatever their loads, so what
// counts is that no lane works for nothing and that a 64-atom cell's stage leaves the CTA alone on its SM (77 KB
// instead of 213 KB and a cluster of two): 73 sets take 80 lanes instead of 96, one set 8 instead of 32.
constexpr int kPT64 = 8;

template <int PTV, int MMAX, bool CLUSTER, int MINB, typename R, int NW, bool GEN, bool FIT>
inline cudaError_t launch_variant(BatchParams bp, const Bucket &b, bool pdl, cudaStream_t s) {
  auto kern = batch_kernel<PTV, MMAX, CLUSTER, MINB, R, NW, GEN, FIT>;
  const size_t smem = PTV == 16 ? b.smem16 : NW != kNW ? b.smem12 : b.smem;
  int &per_sm = b.per_sm[PTV == 16 ? 4 : NW != kNW ? 5 : 2 * (GEN ? 1 : 0) + (FIT ? 1 : 0)];
  constexpr int kThr = NW * kWarp;
  bp.ntiles = (bp.P + PTV - 1) / PTV;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const int cluster = CLUSTER ? b.cluster : 1, ncta = cluster;
  // resident CTAs of this variant, rounded down to whole clusters
  int dev = 0, nsm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  if (per_sm == 0) {
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kThr, smem);
    if (e != cudaSuccess) return e;
  }
  const int slots = std::max(1, per_sm * nsm / ncta);
  const int nconf = b.nitems;
  // work items: each configuration's tiles are split into chunks. Ragged configurations: about four items per
  // CTA slot balance the dynamically claimed work. Alike ones: the chunk with the least time, waves of items x
  // (tiles + staging), staging an item costing about half a tile (FP32) or a tenth (FP64); fewer items win a tie.
  // (300 cells on 304 slots stay whole; 100 cells x 2 tiles run as 200 items, 100 cells x 10 FP64 tiles on 152
  // slots as 1000.) The autotuner's choice for this (P, mode) overrides both
  int per_conf = std::min(bp.ntiles, std::max(1, (4 * slots + nconf - 1) / nconf));
  if (b.uniform) {
    const double stage_cost = sizeof(R) == 8 ? 0.1 : 0.5;
    double best = 1e300;
    for (int ct = bp.ntiles; ct >= 1; --ct) {
      const int nch = (bp.ntiles + ct - 1) / ct;
      if ((bp.ntiles + nch - 1) / nch != ct) continue;   // the same number of chunks with fewer tiles each comes later
      const int64_t waves = ((int64_t)nconf * nch + slots - 1) / slots;
      const double cost = (double)waves * (ct + stage_cost);
      if (cost < 0.999 * best) {
        best = cost;
        per_conf = nch;
      }
    }
  }
  bp.narrow = 1;
  if (b.tune_P == bp.P && b.tune_mode == bp.mode && b.tune_per_conf > 0) {
    per_conf = std::min(bp.ntiles, b.tune_per_conf);
    bp.narrow = b.tune_narrow;
  }
  bp.nconf = nconf;
  bp.chunk_tiles = (bp.ntiles + per_conf - 1) / per_conf;
  bp.nchunks = (bp.ntiles + bp.chunk_tiles - 1) / bp.chunk_tiles;
  const int nitems = nconf * bp.nchunks;
  const int grid_clusters = std::min(nitems, slots);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(grid_clusters * ncta));
  cfg.blockDim = dim3(kThr);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  // programmatic dependent launch: the kernel may start while its predecessor (the preparation kernel
  // or the previous bucket) runs; it waits for it before reading the per-call constants
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = pdl ? 1 : 0;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if constexpr (CLUSTER) {
    if (cluster > 8) {
      e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
      if (e != cudaSuccess) return e;
    }
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = cluster;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.numAttrs = 2;
  }
  const cudaError_t el = cudaLaunchKernelEx(&cfg, kern, bp);
  if (el == cudaSuccess) count_launches(1);
  return el;
}


// One bucket of the plan in one precision and form (R, GEN), for the fitness (FIT) or for evaluation and
// gradient. Instantiated in translation units of their own (batch_*.cu), which compile side by side.
template <typename R, bool GEN, bool FIT>
cudaError_t launch_bucket(const BatchParams &bp, const Bucket &b, bool pdl, cudaStream_t s) {
  const bool cl = b.cluster > 1;
  if constexpr (sizeof(R) == 8) {
    if (!cl) return launch_variant<kPT64, 8, false, 1, R, kNW, GEN, FIT>(bp, b, pdl, s);
    return launch_variant<kPT64, 8, true, 1, R, kNW, GEN, FIT>(bp, b, pdl, s);
  } else if constexpr (GEN) {
    if (!cl && b.mmax <= 4) return launch_variant<kPT, 4, false, 2, R, kNW, GEN, FIT>(bp, b, pdl, s);
    if (!cl) return launch_variant<kPT, 8, false, 2, R, kNW, GEN, FIT>(bp, b, pdl, s);
    return launch_variant<kPT, 8, true, 2, R, kNW, GEN, FIT>(bp, b, pdl, s);
  } else {
    if constexpr (FIT) {   // schedules that only the tuner and tersoff_set_schedule choose
      const bool tuned = b.tune_P == bp.P && b.tune_mode == bp.mode && !cl && b.mmax <= 4;
      if (tuned && b.tune_pt == 16 && b.smem16 > 0)
        return launch_variant<16, 4, false, 3, R, kNW, GEN, FIT>(bp, b, pdl, s);
      if (tuned && b.tune_nw == 12 && b.smem12 > 0)
        return launch_variant<kPT, 4, false, 2, R, 12, GEN, FIT>(bp, b, pdl, s);
    }
    if (!cl && b.mmax <= 4) return launch_variant<kPT, 4, false, 2, R, kNW, GEN, FIT>(bp, b, pdl, s);
    if (!cl && b.mmax <= 6) return launch_variant<kPT, 6, false, 2, R, kNW, GEN, FIT>(bp, b, pdl, s);
    if (!cl) return launch_variant<kPT, 8, false, 2, R, kNW, GEN, FIT>(bp, b, pdl, s);
    if (b.mmax <= 4) return launch_variant<kPT, 4, true, 2, R, kNW, GEN, FIT>(bp, b, pdl, s);
    if (b.mmax <= 6) return launch_variant<kPT, 6, true, 2, R, kNW, GEN, FIT>(bp, b, pdl, s);
    return launch_variant<kPT, 8, true, 2, R, kNW, GEN, FIT>(bp, b, pdl, s);
  }
}

// Force the module loading of every kernel of one precision in the minimal form, for the fitness (FIT) or for
// evaluation and gradient (with lazy loading the driver would load each on its first launch, allocating device memory
// for its code then).
template <int PTV, int MMAX, bool CLUSTER, int MINB, typename R, int NW, bool FIT>
inline cudaError_t touch_variant() {
  cudaFuncAttributes fa;
  return cudaFuncGetAttributes(&fa, batch_kernel<PTV, MMAX, CLUSTER, MINB, R, NW, false, FIT>);
}
template <bool FIT>
inline cudaError_t touch_variants32() {
  cudaError_t e = touch_variant<kPT, 4, false, 2, float, kNW, FIT>();
  if (e == cudaSuccess) e = touch_variant<kPT, 6, false, 2, float, kNW, FIT>();
  if (e == cudaSuccess) e = touch_variant<kPT, 8, false, 2, float, kNW, FIT>();
  if (e == cudaSuccess) e = touch_variant<kPT, 4, true, 2, float, kNW, FIT>();
  if (e == cudaSuccess) e = touch_variant<kPT, 6, true, 2, float, kNW, FIT>();
  if (e == cudaSuccess) e = touch_variant<kPT, 8, true, 2, float, kNW, FIT>();
  return e;
}
template <bool FIT>
inline cudaError_t touch_variants64() {
  cudaError_t e = touch_variant<kPT64, 8, false, 1, double, kNW, FIT>();
  if (e == cudaSuccess) e = touch_variant<kPT64, 8, true, 1, double, kNW, FIT>();
  return e;
}
#ifdef TSF_DEBUG_BOUNDS
// Reads and clears a translation unit's bounds record (tersoff_debug_bounds).
#define TSF_DEBUG_TAKE(name)                                                          \
  cudaError_t name(unsigned *out4) {                                                  \
    const unsigned z[4] = {0, 0, 0, 0};                                               \
    cudaError_t e = cudaMemcpyFromSymbol(out4, tsf_dbg, 4 * sizeof(unsigned));        \
    if (e == cudaSuccess) e = cudaMemcpyToSymbol(tsf_dbg, z, sizeof(z));              \
    return e;                                                                         \
  }
cudaError_t debug_take_fit32(unsigned *), debug_take_eval32(unsigned *), debug_take_64(unsigned *),
    debug_take_gen(unsigned *), debug_take_gen64(unsigned *);
#else
#define TSF_DEBUG_TAKE(name)
#endif
cudaError_t preload_fitness32();   // batch_fit32.cu
cudaError_t preload_eval32();      // batch_eval32.cu
cudaError_t preload_batch64();     // batch_64.cu

}  // namespace tsf
