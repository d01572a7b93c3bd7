// Launches of the several-steps-per-launch kernel of small lattices (tile.cuh).
#include <cuda_runtime.h>

#include <algorithm>

#include "context.h"
#include "kernels.h"
#include "tile.cuh"

namespace lbmp {

static_assert(kTileMaxLevels <= lbmp_ctx::kMaxPerLaunch, "a graph slot for every remainder");

// Lattices that take it (us a step, before -> with it): FP32 up to some 170 000
// nodes (64 x 33: 2.0 -> 1.2, 256^2 2.7 -> 1.9, 410 x 200 2.9 -> 2.1, 400^2 3.6 -> 2.9;
// 512^2 4.1 -> 4.5), FP16 up to 70 000 (128 x 96: 2.6 -> 1.9, 256^2 2.8 -> 2.7;
// 320 x 300 2.95 -> 3.3: a rounding per node, not per pair, at every level).
bool tile_covers(int storage, int nx, int rows) {
  return (long long)nx * rows <= (storage == 0 ? 170000 : 70000);
}

// The tiles and steps per launch of the smallest estimated time per step: a
// launch and its loads take about 3.5 us and 1 ns a node of the tile, a level the
// latency of one node update for each round of the block's warps, the issue
// of its units (a unit: two rows of 32 columns) and the longer chain of a
// pressure column.  The plan is within 5% of the best of the sweeps made
// (64 x 33: 8 x 16 tiles, 12 steps; 410 x 200: 19 x 8, 6; 256^2: 12 x 12, 6).
bool tile_plan(int storage, bool dyn, int nx, int rows, bool pressure, bool walls, int nsm,
               TilePlan *out) {
  const int most = storage == 0 ? (dyn ? TileCfg<StoreF32, true>::kNodes
                                       : TileCfg<StoreF32, false>::kNodes)
                                : (dyn ? TileCfg<StoreF16, true>::kNodes
                                       : TileCfg<StoreF16, false>::kNodes);
  double best = -1.0;
  for (int levels : {4, 6, 8, 12, kTileMaxLevels}) {
    for (int tx = 1; tx == 1 || (nx / tx >= 4 && tx <= nsm); tx += 1 + tx / 32) {
      const int tw = (nx + tx - 1) / tx, w = tw + 2 * levels;
      const int most_ty = std::min(rows, nsm / tx);
      for (int part = 4; part >= 1; --part) {  // all SMs, or three, two, one in four
        const int ty = std::max(1, most_ty * part / 4);
        const int th = (rows + ty - 1) / ty, h = th + 2 * levels;
        if ((long long)w * h > most) continue;
        double us = 3.5 + 1e-3 * w * h;
        for (int l = 1; l <= levels; ++l) {
          int cw = w - 2 * l, ch = h - 2 * l;
          if (pressure) cw = std::min(cw, nx);
          if (walls) ch = std::min(ch, rows);
          const int units = (cw + 31) / 32 * ((ch + 1) / 2);
          us += 0.35 * ((units + kTileWarps - 1) / kTileWarps) + 0.04 * units +
                (pressure ? 0.3 : 0.0);
        }
        if (best < 0.0 || us / levels < best) {
          best = us / levels;
          *out = {tx, ty, levels};
        }
      }
    }
  }
  return best > 0.0;
}

// The kernel's shared-memory limit, on the current device.
template <class S, bool SR, bool DYN, bool FORCH>
static cudaError_t tile_limit() {
  return cudaFuncSetAttribute(tile_step_kernel<S, SR, DYN, FORCH>,
                              cudaFuncAttributeMaxDynamicSharedMemorySize,
                              TileCfg<S, DYN>::kSmemBytes);
}
cudaError_t prepare_tile(int storage, bool sr, bool dyn, bool forch) {
#define LBMP_TILE(S, SR, DYN) (forch ? tile_limit<S, SR, DYN, true>() : tile_limit<S, SR, DYN, false>())
  if (storage == 0) return dyn ? LBMP_TILE(StoreF32, false, true) : LBMP_TILE(StoreF32, false, false);
  if (sr) return dyn ? LBMP_TILE(StoreF16, true, true) : LBMP_TILE(StoreF16, true, false);
  return dyn ? LBMP_TILE(StoreF16, false, true) : LBMP_TILE(StoreF16, false, false);
#undef LBMP_TILE
}

template <class S, bool SR, bool DYN, bool FORCH>
static cudaError_t launch_tile_t(const StepArgs &a, int rows, const void *fin, void *fout,
                                 const float2 *med, const unsigned long long *tctr, int k,
                                 const TilePlan &p, int levels, cudaStream_t s) {
  const long long w = (a.nx + p.tx - 1) / p.tx + 2 * levels, h = (rows + p.ty - 1) / p.ty + 2 * levels;
  if (w * h > TileCfg<S, DYN>::kNodes || levels < 1 || levels > kTileMaxLevels)
    return cudaErrorInvalidValue;  // the block's shared memory holds kNodes nodes
  return launch_chained(tile_step_kernel<S, SR, DYN, FORCH>, dim3(p.tx * p.ty), dim3(kTileWarps * 32),
                        TileCfg<S, DYN>::kSmemBytes, s,
      a, (const typename S::T *)fin, (typename S::T *)fout, med, tctr, k, p, levels, rows);
}

cudaError_t launch_tile(int storage, bool sr, const StepArgs &a, int rows, const void *fin,
                        void *fout, const float2 *med, const unsigned long long *tctr, int k,
                        const TilePlan &p, int levels, cudaStream_t s) {
  const bool dyn = a.kn0 != nullptr;
#define LBMP_TILE(S, SR, DYN)                                                                   \
  (a.forch ? launch_tile_t<S, SR, DYN, true>(a, rows, fin, fout, med, tctr, k, p, levels, s)    \
           : launch_tile_t<S, SR, DYN, false>(a, rows, fin, fout, med, tctr, k, p, levels, s))
  if (storage == 0) return dyn ? LBMP_TILE(StoreF32, false, true) : LBMP_TILE(StoreF32, false, false);
  if (sr) return dyn ? LBMP_TILE(StoreF16, true, true) : LBMP_TILE(StoreF16, true, false);
  return dyn ? LBMP_TILE(StoreF16, false, true) : LBMP_TILE(StoreF16, false, false);
#undef LBMP_TILE
}

}  // namespace lbmp
