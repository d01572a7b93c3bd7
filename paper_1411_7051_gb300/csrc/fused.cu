// Launches of the two-step kernel (fused.cuh).
#include <cuda_runtime.h>

#include <algorithm>

#include "fused.cuh"
#include "kernels.h"

namespace lbmp {

// The split of the smallest cost (fused_cost), of all splits into equal segments.
// Many numbers of parts give one height: each height is looked at once (64 x 8192:
// 181 of 8192 candidates, 71 -> 2.3 us).
template <class C>
static FusedPlan split(int q, int nx, int rows, int nsm) {
  const double cap = (double)nsm * C::kBlocks * kFusedWarps;
  const FusedStrips f = fused_strips<C>(nx);
  FusedPlan best{q, rows, 0, 0};
  const int most = (int)std::max(1.0, std::min((double)rows, 8.0 * cap / (f.inner + 1)));
  double best_cost = -1.0;
  for (int parts = 1; parts <= most;) {
    const int seg = (rows + parts - 1) / parts;
    const int n = (rows + seg - 1) / seg;
    const int edges = (n + f.per - 1) / f.per;
    const int tasks = edges + f.inner * n;
    const double cost = fused_cost(seg, tasks / cap);
    if (best_cost < 0.0 || cost < best_cost) {
      best_cost = cost;
      best = {q, seg, edges, tasks};
    }
    if (seg == 1) break;
    parts = (rows + seg - 2) / (seg - 1);  // the fewest of the next lower height
  }
  return best;
}

// Two pairs a lane spend fewer instructions a node, one pair a lane spreads a small
// lattice over more warps: 768^2 FP32 7.2 / 7.0 us a step, 1024^2 9.8 / 10.1,
// 1531 x 1153 13.9 / 14.6, 4096^2 113.8 / 114.8, FP16 96.7 / 112.9.
FusedPlan fused_plan(int storage, bool dyn, int nx, int rows, int nsm) {
  const bool wide = nx >= FusedCfg<StoreF32, 2, false>::kCols && (long long)nx * rows >= 1000000;
#define LBMP_SPLIT(S, DYN)                                       \
  (wide ? split<FusedCfg<S, 2, DYN>>(2, nx, rows, nsm)           \
        : split<FusedCfg<S, 1, DYN>>(1, nx, rows, nsm))
  if (storage == 0) return dyn ? LBMP_SPLIT(StoreF32, true) : LBMP_SPLIT(StoreF32, false);
  return dyn ? LBMP_SPLIT(StoreF16, true) : LBMP_SPLIT(StoreF16, false);
#undef LBMP_SPLIT
}

// Where two steps per launch are the faster form.  FP16 storage: everywhere
// (against the staged kernel 512^2 6.4 -> 4.2 us a step, 4096^2 112 -> 97).  FP32:
// the direct kernel needs fewer rows in a row on small lattices (512^2: 3.9 us
// against 4.0; 768^2: 7.1 against 7.0; 4096^2: 190 against 114), with a dynamic Kn
// up to about 10^6 nodes (768^2: 8.3 against 8.9; 1024^2: 13.3 against 11.4).
bool fused_covers(int storage, bool dyn, int nx, int ny) {
  if (nx < FusedCfg<StoreF32, 1, false>::kCols || ny < kFusedMinNy) return false;
  return storage != 0 || (long long)nx * ny >= (dyn ? 1000000 : 500000);
}

// The kernel's shared-memory limit, on the current device, where it needs more than
// the default 48 KB (FP32 with a dynamic Kn, two pairs a lane: 54 KB).
constexpr int kDefaultSmem = 48 * 1024;
cudaError_t prepare_fused(int storage, bool dyn, bool forch) {
  using C = FusedCfg<StoreF32, 2, true>;
  static_assert(FusedCfg<StoreF32, 2, false>::kSmemBytes <= kDefaultSmem &&
                    FusedCfg<StoreF32, 1, true>::kSmemBytes <= kDefaultSmem &&
                    FusedCfg<StoreF16, 2, true>::kSmemBytes <= kDefaultSmem,
                "every other form fits the default limit");
  if (storage != 0 || !dyn) return cudaSuccess;
  return forch ? cudaFuncSetAttribute(fused_step_kernel<StoreF32, false, true, false, true, 2>,
                                      cudaFuncAttributeMaxDynamicSharedMemorySize, C::kSmemBytes)
               : cudaFuncSetAttribute(fused_step_kernel<StoreF32, false, true, false, false, 2>,
                                      cudaFuncAttributeMaxDynamicSharedMemorySize, C::kSmemBytes);
}

template <class S, bool SR, bool DYN, bool MOM, bool FORCH, int Q>
static cudaError_t launch_fused_q(const StepArgs &a, int rows, const void *fin, void *fout,
                                  const float2 *med, const unsigned long long *tctr, int k,
                                  const FusedPlan &plan, float *mom1, float *mom2, cudaStream_t s) {
  using C = FusedCfg<S, Q, DYN>;
  return launch_chained(fused_step_kernel<S, SR, DYN, MOM, FORCH, Q>,
                        dim3((plan.tasks + kFusedWarps - 1) / kFusedWarps), dim3(kFusedWarps * 32),
                        C::kSmemBytes, s,
          a, (const typename S::T *)fin, (typename S::T *)fout, med, tctr, k, rows, plan.seg,
          fused_strips<C>(a.nx), plan.edges, plan.tasks, mom1, mom2);
}

template <class S, bool SR, bool DYN, bool MOM>
static cudaError_t launch_fused_t(const StepArgs &a, int rows, const void *fin, void *fout,
                                  const float2 *med, const unsigned long long *tctr, int k,
                                  const FusedPlan &p, float *mom1, float *mom2, cudaStream_t s) {
#define LBMP_FUSED(FORCH, Q) \
  launch_fused_q<S, SR, DYN, MOM, FORCH, Q>(a, rows, fin, fout, med, tctr, k, p, mom1, mom2, s)
  if (a.forch) return p.q == 2 ? LBMP_FUSED(true, 2) : LBMP_FUSED(true, 1);
  return p.q == 2 ? LBMP_FUSED(false, 2) : LBMP_FUSED(false, 1);
#undef LBMP_FUSED
}

cudaError_t launch_fused(int storage, bool sr, const StepArgs &a, int rows, const void *fin,
                         void *fout, const float2 *med, const unsigned long long *tctr, int k,
                         const FusedPlan &plan, cudaStream_t s) {
  const bool dyn = a.kn0 != nullptr;
#define LBMP_FUSED(S, SR, DYN) \
  launch_fused_t<S, SR, DYN, false>(a, rows, fin, fout, med, tctr, k, plan, nullptr, nullptr, s)
  if (storage == 0)
    return dyn ? LBMP_FUSED(StoreF32, false, true) : LBMP_FUSED(StoreF32, false, false);
  if (sr) return dyn ? LBMP_FUSED(StoreF16, true, true) : LBMP_FUSED(StoreF16, true, false);
  return dyn ? LBMP_FUSED(StoreF16, false, true) : LBMP_FUSED(StoreF16, false, false);
#undef LBMP_FUSED
}

cudaError_t launch_fused_moments(const StepArgs &a, int rows, const float *fin, float *fout,
                                 const float2 *med, float *mom1, float *mom2,
                                 const FusedPlan &plan, cudaStream_t s) {
  return launch_fused_t<StoreF32, false, false, true>(a, rows, fin, fout, med, nullptr, 0, plan,
                                                      mom1, mom2, s);
}

}  // namespace lbmp
