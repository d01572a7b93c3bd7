// CUDA kernels of the porous lattice Boltzmann step for sm_103a
// (Chen et al., arXiv:1411.7051, Section III).
//
// The step is a stencil stream: every population is read once and written
// once per time step, so the roofline is HBM bandwidth (no dense
// contraction, no tensor cores).  One fused kernel pulls the nine
// populations of a node (periodic wrap, halfway bounce-back at plates,
// pressure-column extrapolation), solves Eq. 16-17 for the velocity, forms
// Eq. 2, Eq. 14 and Eq. 15 and writes the nine post-collision values.
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "chain.cuh"
#include "kernels.h"
#include "lattice.cuh"
#include "pairs.cuh"
#include "staged.cuh"
#include "wide.cuh"

namespace lbmp {

constexpr int kStepBX = 128;   // threads per block along x
constexpr int kStepNPT = 2;    // nodes per thread, strided by kStepBX
constexpr int kLoadBX = 256;
constexpr int kMediumBX = 256;

// ------------------------------------------------------------- step kernel
// Each thread updates kStepNPT nodes of one row, kStepBX apart, so every
// load and store instruction of a warp touches 32 consecutive elements.
// All loads of a thread are issued before its first collision.  Plate rows
// are block-uniform branches inside pull_node.  The stochastic-rounding
// bits of time level t come from *tctr + k (the counter is advanced by
// bump_kernel after a group of launches).  A chained launch (chain.cuh).
// DYN: Knudsen number per node and step from the local pressure (the
// medium holds 1/k_i, a.kn0 the Kn at p0).
// MOM: also store each node's post-stream moments (rho - rho0, m_x, m_y;
// three [ny][pitch] planes at mom, a.plane apart) -- all that the reverse
// step of the adjoint needs of the forward state.
template <class S, bool SR, bool DYN, bool MOM = false>
__global__ void __launch_bounds__(kStepBX)
    step_kernel(const StepArgs a, const typename S::T *fin,
                typename S::T *__restrict__ fout, const float2 *__restrict__ med,
                const unsigned long long *tctr, int k,
                float *__restrict__ mom) {
  const int y = a.y0 + (a.rev ? (int)gridDim.y - 1 - (int)blockIdx.y : (int)blockIdx.y);
  const int xb = blockIdx.x * (kStepBX * kStepNPT) + threadIdx.x;
  const long long row = (long long)y * a.pitch;
  chain_wait();
  float d[kStepNPT][9];
  float2 m[kStepNPT];
  float k0[kStepNPT];
#pragma unroll
  for (int j = 0; j < kStepNPT; ++j) {
    const int x = xb + j * kStepBX;
    k0[j] = 0.0f;
    if (x < a.nx) {
      pull_node<S>(fin, a, x, y, d[j]);
      m[j] = med[row + x];
      if (DYN) k0[j] = a.kn0[row + x];
    }
  }
  uint32_t ts = 0;
  if (SR) {
    const unsigned long long t = *tctr + (unsigned long long)k;
    ts = mix32((uint32_t)t * 0x9e3779b9u ^ a.seed_lo ^ mix32((uint32_t)(t >> 32) ^ a.seed_hi));
  }
#pragma unroll
  for (int j = 0; j < kStepNPT; ++j) {
    const int x = xb + j * kStepBX;
    if (x >= a.nx) continue;
    if (a.pressure && (x == 0 || x == a.nx - 1))
      pressure_node<S, DYN>(fin, med, a, x, y, m[j].x, d[j]);
    const NodeState s = node_state<DYN>(d[j], m[j].x, m[j].y, a, k0[j]);
    if (MOM) {
      float *mo = mom + row + x;
      mo[0] = s.drho_s;
      mo[a.plane] = s.mx;
      mo[2 * a.plane] = s.my;
    }
    collide<S::kHiLo>(d[j], s, a);
    typename S::T *o = fout + row + x;
    const uint32_t h = SR ? mix32((uint32_t)(row + x) ^ ts) : 0u;
#pragma unroll
    for (int i = 0; i < 9; ++i) S::template st1r<SR>(o + i * a.plane, d[j][i], h, i);
  }
}

// Advance the time-level counter of the stochastic rounding by n.
__global__ void bump_kernel(unsigned long long *tctr, int n) { *tctr += (unsigned long long)n; }

cudaError_t launch_step(int storage, bool sr, const StepArgs &a, int rows, const void *fin,
                        void *fout, const float2 *med, const unsigned long long *tctr, int k,
                        cudaStream_t s) {
  if (rows <= 0 || a.nx <= 0) return cudaSuccess;
  dim3 block(kStepBX);
  dim3 grid((a.nx + kStepBX * kStepNPT - 1) / (kStepBX * kStepNPT), rows);
  const bool dyn = a.kn0 != nullptr;
  const float *f32i = (const float *)fin;
  float *f32o = (float *)fout;
  const __half *f16i = (const __half *)fin;
  __half *f16o = (__half *)fout;
  if (storage == 0) {
    if (dyn)
      return launch_chained(step_kernel<StoreF32, false, true>, grid, block, 0, s, a, f32i, f32o, med, tctr, k, nullptr);
    else
      return launch_chained(step_kernel<StoreF32, false, false>, grid, block, 0, s, a, f32i, f32o, med, tctr, k, nullptr);
  } else if (sr) {
    if (dyn)
      return launch_chained(step_kernel<StoreF16, true, true>, grid, block, 0, s, a, f16i, f16o, med, tctr, k, nullptr);
    else
      return launch_chained(step_kernel<StoreF16, true, false>, grid, block, 0, s, a, f16i, f16o, med, tctr, k, nullptr);
  } else {
    if (dyn)
      return launch_chained(step_kernel<StoreF16, false, true>, grid, block, 0, s, a, f16i, f16o, med, tctr, k, nullptr);
    else
      return launch_chained(step_kernel<StoreF16, false, false>, grid, block, 0, s, a, f16i, f16o, med, tctr, k, nullptr);
  }
}

cudaError_t launch_step_moments(const StepArgs &a, int rows, const float *fin, float *fout,
                                const float2 *med, float *mom, cudaStream_t s) {
  if (rows <= 0 || a.nx <= 0) return cudaSuccess;
  dim3 block(kStepBX);
  dim3 grid((a.nx + kStepBX * kStepNPT - 1) / (kStepBX * kStepNPT), rows);
  return launch_chained(step_kernel<StoreF32, false, false, true>, grid, block, 0, s, a, fin, fout,
                        med, nullptr, 0, mom);
}

// -------------------------------------------------------- wide variant
cudaError_t launch_wide(bool sr, const StepArgs &a, int rows, const void *fin, void *fout,
                        const float2 *med, const unsigned long long *tctr, int k,
                        cudaStream_t s) {
  if (rows <= 0 || a.nx <= 0) return cudaSuccess;
  dim3 block(kWideBX);
  dim3 grid((a.nx + kWideBX * kWideV - 1) / (kWideBX * kWideV), rows);
  const __half *i = (const __half *)fin;
  __half *o = (__half *)fout;
  const bool dyn = a.kn0 != nullptr;
  if (sr) {
    if (dyn) wide_step_kernel<true, true><<<grid, block, 0, s>>>(a, i, o, med, tctr, k);
    else wide_step_kernel<true, false><<<grid, block, 0, s>>>(a, i, o, med, tctr, k);
  } else {
    if (dyn) wide_step_kernel<false, true><<<grid, block, 0, s>>>(a, i, o, med, tctr, k);
    else wide_step_kernel<false, false><<<grid, block, 0, s>>>(a, i, o, med, tctr, k);
  }
  return cudaGetLastError();
}

// ------------------------------------------------------ staged variant
template <class S, bool SR, bool DYN>
static cudaError_t launch_staged_t(const StepArgs &a, int rows, const void *fin, void *fout,
                                   const float2 *med, const unsigned long long *tctr, int k,
                                   unsigned *err, int nsm, cudaStream_t s) {
  using C = StageCfgFor<S, DYN>;
  using L = StageLayout<S, C>;
  const long long span = (long long)rows * a.pitch;  // flat nodes of the launch rows
  const int ntiles = (int)((span + C::W - 1) / C::W);
  const int grid = ntiles < nsm ? ntiles : nsm;
  staged_step_kernel<S, SR, DYN><<<grid, kStagedThreads, L::kSmemBytes, s>>>(
      a, (const typename S::T *)fin, (typename S::T *)fout, med, tctr, k, rows, err);
  return cudaGetLastError();
}

template <class S, bool SR, bool DYN>
static cudaError_t staged_smem_attr() {
  return cudaFuncSetAttribute(staged_step_kernel<S, SR, DYN>,
                              cudaFuncAttributeMaxDynamicSharedMemorySize,
                              StageLayout<S, StageCfgFor<S, DYN>>::kSmemBytes);
}

cudaError_t prepare_staged() {
  cudaError_t e;
  if ((e = staged_smem_attr<StoreF32, false, false>()) != cudaSuccess) return e;
  if ((e = staged_smem_attr<StoreF16, false, false>()) != cudaSuccess) return e;
  if ((e = staged_smem_attr<StoreF16, true, false>()) != cudaSuccess) return e;
  if ((e = staged_smem_attr<StoreF16, false, true>()) != cudaSuccess) return e;
  return staged_smem_attr<StoreF16, true, true>();
}

// A dynamic Kn (a.kn0 set) takes the FP16 kernel that also stages the Kn
// plane; with FP32 storage the direct kernel serves it (the context never
// selects the staged one).
cudaError_t launch_staged(int storage, bool sr, const StepArgs &a, int rows, const void *fin,
                          void *fout, const float2 *med, const unsigned long long *tctr, int k,
                          unsigned *err, int nsm, cudaStream_t s) {
  if (rows <= 0 || a.nx <= 0) return cudaSuccess;
  const bool dyn = a.kn0 != nullptr;
  if (storage == 0) {
    if (dyn) return cudaErrorInvalidValue;
    return launch_staged_t<StoreF32, false, false>(a, rows, fin, fout, med, tctr, k, err, nsm, s);
  }
  if (dyn) {
    if (sr) return launch_staged_t<StoreF16, true, true>(a, rows, fin, fout, med, tctr, k, err, nsm, s);
    return launch_staged_t<StoreF16, false, true>(a, rows, fin, fout, med, tctr, k, err, nsm, s);
  }
  if (sr) return launch_staged_t<StoreF16, true, false>(a, rows, fin, fout, med, tctr, k, err, nsm, s);
  return launch_staged_t<StoreF16, false, false>(a, rows, fin, fout, med, tctr, k, err, nsm, s);
}

cudaError_t launch_bump(unsigned long long *tctr, int n, cudaStream_t s) {
  bump_kernel<<<1, 1, 0, s>>>(tctr, n);
  return cudaGetLastError();
}

// ------------------------------------------------- block reduction helper
// Sums kNQ doubles over the block in a fixed order and writes them to
// partials[blockLinear * kNQ + q] (deterministic for a fixed launch shape).
// Quantities whose bit is set in max_mask are reduced by max (values >= 0).
template <int BX>
__device__ __forceinline__ void block_reduce_store(double v[kNQ], double *partials,
                                                   unsigned max_mask = 0u) {
  __shared__ double red[BX / 32][kNQ];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int q = 0; q < kNQ; ++q) {
    const bool mx = (max_mask >> q) & 1u;
    double t = v[q];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      const double o = __shfl_down_sync(0xffffffffu, t, off);
      t = mx ? fmax(t, o) : t + o;
    }
    if (lane == 0) red[warp][q] = t;
  }
  __syncthreads();
  if (threadIdx.x < kNQ) {
    const bool mx = (max_mask >> threadIdx.x) & 1u;
    double t = 0.0;
    for (int w = 0; w < BX / 32; ++w) t = mx ? fmax(t, red[w][threadIdx.x]) : t + red[w][threadIdx.x];
    const long long b = (long long)blockIdx.y * gridDim.x + blockIdx.x;
    partials[b * kNQ + threadIdx.x] = t;
  }
}

// ------------------------------------------------------------- finalize
constexpr int kFinBX = 256;

__global__ void __launch_bounds__(kFinBX)
    finalize_kernel(const double *__restrict__ partials, int nblocks, int nq,
                    double *__restrict__ out, unsigned max_mask) {
  __shared__ double sh[kFinBX];
  for (int q = 0; q < nq; ++q) {
    const bool mx = (max_mask >> q) & 1u;
    double t = 0.0;
    for (int b = threadIdx.x; b < nblocks; b += kFinBX) {
      const double v = partials[(long long)b * nq + q];
      t = mx ? fmax(t, v) : t + v;
    }
    sh[threadIdx.x] = t;
    __syncthreads();
    for (int w = kFinBX / 2; w > 0; w >>= 1) {
      if (threadIdx.x < w)
        sh[threadIdx.x] = mx ? fmax(sh[threadIdx.x], sh[threadIdx.x + w])
                             : sh[threadIdx.x] + sh[threadIdx.x + w];
      __syncthreads();
    }
    if (threadIdx.x == 0) out[q] = sh[0];
    __syncthreads();
  }
}

cudaError_t launch_finalize(const double *partials, int nblocks, int nq, double *out,
                            cudaStream_t s, unsigned max_mask) {
  finalize_kernel<<<1, kFinBX, 0, s>>>(partials, nblocks, nq, out, max_mask);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- medium
// The largest k_a of a dynamic-Kn medium (it only sets the FP16 scale) takes
// fc_f32 of the lattice header.

// 1 / k_a = 1 / (k_i f_c(Kn)) of Eq. 3 in FP64 with a single division.
// Eq. 6-7 (b = -1) as one fraction: with t = Kn^-0.4348 and a = 1 + 0.17 t,
//   1 + alpha Kn = (a + 1.358 Kn) / a,   1 + 4 Kn / (1 + Kn) = (1 + 5 Kn) / (1 + Kn),
//   1 / k_a = a (1 + Kn) / (k_i (a + 1.358 Kn) (1 + 5 Kn)).
// Only t comes from FP32 (log2f, exp2f: ~3e-7 relative); it enters through
// a in both numerator and denominator, whose sensitivities nearly cancel:
// d ln(1/k_a) / d ln t = 0.17 t 1.358 Kn / (a (a + 1.358 Kn)) <= 0.08, so
// the FP32 1/k_a stored is within ~0.1 ulp of the FP64 value before its
// final rounding.  FP64 runs at a small fraction of the FP32 rate on this
// GPU: the FP64 power of Kn made the precompute 50 times slower than its
// memory traffic.  Kn = 0 gives f_c = 1 exactly.
__device__ __forceinline__ double inv_ka(double k, double K, int model) {
  if (model == 1) return 1.0 / (k * fma(4.0, K, 1.0));
  if (K == 0.0) return 1.0 / k;
  const double t = (double)exp2f(-0.4348f * log2f((float)K));
  const double a = fma(0.17, t, 1.0);
  return (a * (1.0 + K)) / (k * fma(1.358, K, a) * fma(5.0, K, 1.0));
}

// ---- the same fraction in FP32-pair arithmetic (the F2 helpers above) ----
// FP64 instructions are the bottleneck of the precompute on this GPU, so
// for the usual ranges of k_i and Kn the fraction is evaluated with FP32
// pairs.  Beside the FP32 power of Kn (as in inv_ka) the result differs from
// the FP64 one by ~2^-40 before its final rounding to FP32.
// A double in [2^-60, 2^60] (not 0) as hi + lo with integer operations only: hi
// keeps the leading 24 bits, lo the next 29 (rounded to 24; the pair then
// carries d to a relative 2^-48).
__device__ __forceinline__ F2 f2_from_double(double d) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(d);
  const int e = (int)((b >> 52) & 0x7ff) - 1023;             // unbiased exponent
  const unsigned hib = (unsigned)((b >> 32) & 0x80000000u) |  // sign
                       ((unsigned)(e + 127) << 23) | (unsigned)((b >> 29) & 0x7fffffu);
  const float lo_int = (float)(unsigned)(b & 0x1fffffffull);  // the low 29 mantissa bits
  const float scale = __uint_as_float((unsigned)(e - 52 + 127) << 23);  // 2^(e - 52)
  return {__uint_as_float(hib), (b >> 63) ? -lo_int * scale : lo_int * scale};
}

// 1 / k_a of inv_ka() for k_i and Kn in the ranges FP32 pairs hold
// comfortably (k_i in [1e-16, 1e12], Kn in [1e-12, 1e6] or 0; the others
// take the FP64 fraction): FP32 to within the FP32 power's error.  k > 0
// and K >= 0 (or -0) on entry, so the range tests compare bit patterns: the
// bits of non-negative doubles order as their values (FP64 compares are
// as slow as the rest of FP64 on this GPU).
__device__ __forceinline__ float inv_ka_pair(double k, double K, int model) {
  const unsigned long long kb = (unsigned long long)__double_as_longlong(k);
  const unsigned long long Kb = (unsigned long long)__double_as_longlong(K) << 1;  // sign dropped
  const bool K0 = Kb == 0;
  const bool k_ok = kb >= 0x3c9cd2b297d889bcull && kb <= 0x426d1a94a2000000ull;  // [1e-16, 1e12]
  const bool K_ok = K0 || (Kb >= (0x3d719799812dea11ull << 1) &&
                           Kb <= (0x412e848000000000ull << 1));                  // [1e-12, 1e6]
  if (!k_ok || !K_ok) return (float)inv_ka(k, K, model);
  const F2 kk = f2_from_double(k);
  const F2 one = {1.0f, 0.0f};
  if (K0) {  // f_c = 1 in both models
    const F2 q = f2_div(one, kk);
    return __fadd_rn(q.hi, q.lo);
  }
  if (model == 1) {  // 1 / (k (1 + 4 Kn))
    const F2 KK = f2_from_double(K);
    const F2 den = f2_mul(kk, f2_add(one, f2_mul({4.0f, 0.0f}, KK)));
    const F2 q = f2_div(one, den);
    return __fadd_rn(q.hi, q.lo);
  }
  const F2 KK = f2_from_double(K);
  const float t = kn_power(KK.hi);  // Kn^-0.4348
  const F2 c017 = {0.17f, (float)(0.17 - (double)0.17f)};
  const F2 c1358 = {1.358f, (float)(1.358 - (double)1.358f)};
  const F2 a = f2_add(one, f2_mul(c017, {t, 0.0f}));  // 1 + 0.17 t
  const F2 num = f2_mul(a, f2_add(one, KK));
  const F2 den = f2_mul(f2_mul(kk, f2_add(a, f2_mul(c1358, KK))),
                        f2_add(one, f2_mul({5.0f, 0.0f}, KK)));
  const F2 q = f2_div(num, den);
  return __fadd_rn(q.hi, q.lo);
}

// A double in [2^-126, 1] rounded to the nearest FP32 (ties to even) with
// integer operations; the rest (0, and values too small for a normal FP32)
// by the FP64 conversion.
__device__ __forceinline__ float unit_to_float(double d) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(d);
  const int e = (int)((b >> 52) & 0x7ff) - 1023;
  if (e < -126) return (float)d;
  const unsigned rest = (unsigned)(b & 0x1fffffffull);  // the 29 bits dropped
  unsigned f = ((unsigned)(e + 127) << 23) | (unsigned)((b >> 29) & 0x7fffffu);
  if (rest > 0x10000000u || (rest == 0x10000000u && (f & 1u))) ++f;  // carries into the exponent
  return __uint_as_float(f);
}

// Range checks on the bits of an FP64 value (integer comparisons; NaN
// fails all of them).  0 <= e <= 1: the bits of a non-negative double order
// as the value; -0 counts as 0.
__device__ __forceinline__ bool in_unit_interval(double e) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(e);
  return b <= 0x3ff0000000000000ull || b == 0x8000000000000000ull;
}
// k > 0 (finite or +inf)
__device__ __forceinline__ bool positive_or_inf(double k) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(k);
  return b >= 1ull && b <= 0x7ff0000000000000ull;
}
// K >= 0 and finite
__device__ __forceinline__ bool nonneg_finite(double K) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(K);
  return b < 0x7ff0000000000000ull || b == 0x8000000000000000ull;
}

// One block per row up to 5 resident blocks of 256 threads on each of 152
// SMs (the launch bound keeps all of them resident); wider grids only add
// partials.
constexpr int kMediumMaxBlocks = 5 * 152;

// Grid-stride over rows: block b takes rows b, b + gridDim.x, ..., its
// threads x, x + 256, ...  Each thread accumulates its nodes' partial sums
// (one FP64 add per node: sum eps) and reduces them once at the end.
__global__ void __launch_bounds__(kMediumBX, kMediumMaxBlocks / 152)
    medium_kernel(const double *__restrict__ eps, const double *__restrict__ k_i,
                  const double *__restrict__ kn, int nx, int ny, int pitch, int y_lo,
                  int y_hi, int kn_model, float *__restrict__ kn0, float kn_scale_max,
                  float2 *__restrict__ med, unsigned *bad, double *__restrict__ partials) {
  F2 se = {0.0f, 0.0f};  // sum of eps: FP32 pairs (~44 bits) without FP64 arithmetic
  double se_small = 0.0;  // and the few eps below 2^-60
  unsigned nodes = 0, open = 0, flags = 0;
  float ka_max = 0.0f;         // dynamic Kn: the largest finite k_a
  float inv_min = INFINITY;    // static Kn: the smallest positive 1/k_a
  for (int y = blockIdx.x; y < ny; y += gridDim.x) {
    const bool fluid_row = y >= y_lo && y < y_hi;
    for (int x = threadIdx.x; x < nx; x += kMediumBX) {
      const long long j = (long long)y * nx + x;
      const long long jp = (long long)y * pitch + x;
      float2 out = make_float2(0.0f, 0.0f);
      float kn_out = 0.0f;
      if (fluid_row) {
        const double e = eps[j], k = k_i[j], K = kn[j];
        unsigned f = 0;
        if (!in_unit_interval(e)) f |= 1u;
        if (!positive_or_inf(k)) f |= 2u;
        if (!nonneg_finite(K)) f |= 4u;
        const float ef = unit_to_float(e);
        float inv_k = 0.0f, ka = 0.0f;
        if (!f) {
          if (kn0) {  // dynamic Kn: 1/k_i stored, k_a formed at every step
            const float kf = (float)k, Kf = (float)K;
            if (!(kf >= 1e-15f)) f |= 8u;
            inv_k = 1.0f / kf;                                    // 0 for k_i = inf
            ka = kf * fc_f32(Kf * kn_scale_max, kn_model);     // at the lowest pressure
            kn_out = Kf;
          } else {
            inv_k = inv_ka_pair(k, K, kn_model);                 // Eq. 3 with Eq. 6-7 or 4-5
            if (!(inv_k <= 1e15f)) f |= 8u;                       // k_a >= 1e-15 (FP32 math)
          }
        }
        flags |= f;
        out = make_float2(ef, inv_k);
        const unsigned long long eb = (unsigned long long)__double_as_longlong(e);
        if (eb >= (963ull << 52) && eb <= 0x3ff0000000000000ull)  // 2^-60 <= e <= 1
          se = f2_add(se, f2_from_double(e));
        else
          se_small += e;  // below 2^-60, -0, and values the flags reject
        ++nodes;
        if (!f && ef > 0.0f) {
          if (inv_k > 0.0f) {  // finite k_a
            if (kn0) ka_max = fmaxf(ka_max, ka);
            else inv_min = fminf(inv_min, inv_k);
          } else {
            ++open;  // open pores (k_a = inf)
          }
        }
      }
      med[jp] = out;
      if (kn0) kn0[jp] = kn_out;
    }
  }
  if (flags) atomicOr(bad, flags);
  // the correctly rounded 1 / x does not increase with x: the largest of the
  // nodes' 1 / inv_k is 1 / (their smallest inv_k)
  if (inv_min < INFINITY) ka_max = fmaxf(ka_max, 1.0f / inv_min);
  double v[kNQ] = {(double)se.hi + (double)se.lo + se_small, (double)nodes, (double)ka_max,
                   (double)open, 0.0, 0.0};
  block_reduce_store<kMediumBX>(v, partials, kMediumMaxMask);
}

int medium_blocks(int nx, int ny) {
  (void)nx;
  return ny < kMediumMaxBlocks ? ny : kMediumMaxBlocks;
}

cudaError_t launch_medium(const double *eps, const double *k_i, const double *kn,
                          int nx, int ny, int pitch, int y_lo, int y_hi, int kn_model,
                          float *kn0, double kn_scale_max, float2 *med, unsigned *bad,
                          double *partials, cudaStream_t s) {
  medium_kernel<<<medium_blocks(nx, ny), kMediumBX, 0, s>>>(
      eps, k_i, kn, nx, ny, pitch, y_lo, y_hi, kn_model, kn0, (float)kn_scale_max, med, bad,
      partials);
  return cudaGetLastError();
}

// ----------------------------------------------------- population loading
// B_j(z) = f_j(z + e_j) when z + e_j is a fluid node (wrapped), f_opp(j)(z)
// when it lies in a plate row, and 0 (unused) beyond a pressure column.
template <class S>
__global__ void __launch_bounds__(kLoadBX)
    load_pops_kernel(const StepArgs a, const double *__restrict__ f,
                     typename S::T *__restrict__ buf) {
  const int y = a.y0 + blockIdx.y;
  const int x = blockIdx.x * kLoadBX + threadIdx.x;
  if (x >= a.nx) return;
  const int ex[9] = {0, 1, 0, -1, 0, 1, -1, -1, 1};
  const int ey[9] = {0, 0, 1, 0, -1, 1, 1, -1, -1};
  const int opp[9] = {0, 3, 4, 1, 2, 7, 8, 5, 6};
  const double w[9] = {4.0 / 9.0,  1.0 / 9.0,  1.0 / 9.0,  1.0 / 9.0, 1.0 / 9.0,
                       1.0 / 36.0, 1.0 / 36.0, 1.0 / 36.0, 1.0 / 36.0};
  const long long n = (long long)a.nx * a.ny;
  const double r0 = (double)a.rho0;
  for (int j = 0; j < 9; ++j) {
    int tx = x + ex[j], ty = y + ey[j];
    double val;
    if (a.walls && (ty == 0 || ty == a.ny - 1)) {
      val = f[opp[j] * n + (long long)y * a.nx + x];
    } else {
      ty = (ty + a.ny) % a.ny;
      if (tx < 0 || tx >= a.nx) {
        if (a.pressure) {
          val = w[j] * r0;
        } else {
          tx = (tx + a.nx) % a.nx;
          val = f[j * n + (long long)ty * a.nx + tx];
        }
      } else {
        val = f[j * n + (long long)ty * a.nx + tx];
      }
    }
    S::st1(buf + j * a.plane + (long long)y * a.pitch + x,
           (float)((val - w[j] * r0) * (double)a.scale));
  }
}

cudaError_t launch_load_pops(int storage, const StepArgs &a, int rows, const double *f,
                             void *buf, cudaStream_t s) {
  dim3 block(kLoadBX);
  dim3 grid((a.nx + kLoadBX - 1) / kLoadBX, rows);
  if (storage == 0)
    load_pops_kernel<StoreF32><<<grid, block, 0, s>>>(a, f, (float *)buf);
  else
    load_pops_kernel<StoreF16><<<grid, block, 0, s>>>(a, f, (__half *)buf);
  return cudaGetLastError();
}

}  // namespace lbmp
