// Read-outs of the current time level: macroscopic fields and populations in
// FP64, the sums behind k_g, mass and residual, the normalised-velocity
// histogram (Eq. 16-17 per node; Section IV.A and Fig. 6).
//
// Each kernel reads every node once (44 B with FP32 storage), so HBM bounds it
// as long as enough loads are in flight and FP64 arithmetic stays rare (~1/64
// of the FP32 rate here): a thread holds the loads of two nodes at a time, and
// FP64 values are formed with integer operations.
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "kernels.h"
#include "lattice.cuh"
#include "pairs.cuh"
#include "readout.cuh"

namespace lbmp {

constexpr int kReadPerSM = 4;  // resident blocks: 64 registers a thread

// Columns in blocks of kReadBX, rows dealt out to the blocks of a column:
// one wave of blocks, up to four (whose ends and starts overlap) while a thread
// keeps at least 16 rows, which the block's own reduction needs to pay.  k_g, FP32:
// 1024^2 37 us with one wave, 55 with four; 4096^2 210 and 186.  Less than half a wave
// beyond the first is left out, since the few blocks of it take as long as a whole
// one: 40 x 65535 fields 282 us with 640 blocks, 168 with 608, populations 447 and
// 262; 257 x 12000 fields 134 with 753 blocks, 108 with 608.
static dim3 read_grid(const StepArgs &a) {
  const long long wave = (long long)kReadPerSM * 152;
  long long blocks = std::min(4 * wave, (long long)a.nx * a.ny / (16 * kReadBX));
  if (blocks < wave + wave / 2) blocks = wave;
  const int gx = (a.nx + kReadBX - 1) / kReadBX;
  return dim3(gx, (unsigned)std::max(1LL, std::min((long long)a.ny, blocks / gx)));
}

int macro_blocks(const StepArgs &a) {
  const dim3 g = read_grid(a);
  return (int)(g.x * g.y);
}

// Calls use(s, y, z, both) with the states of the fluid rows of the thread's
// column among blockIdx.y, blockIdx.y + gridDim.y, ..., two at a time (both =
// false: z = y, a lone row).
template <bool DYN, class P, class Use>
__device__ __forceinline__ void walk_column(const P &p, Use use) {
  if (p.x >= p.a.nx) return;
  const int gy = (int)gridDim.y, ny = p.a.ny;
#pragma unroll 1
  for (int y = blockIdx.y; y < ny; y += 2 * gy) {
    const int z = y + gy;
    const bool fy = p.fluid(y), fz = p.fluid(z);
    if (!fy && !fz) continue;
    typename P::Raw r;
    p.template load<DYN>(fy ? y : z, fz ? z : y, r);
    const NodeStateT<float2> s = p.template state<DYN>(r);
    use(s, r.y, r.z, fy && fz);
  }
}
// Zeros in the plate rows of the thread's column.
__device__ __forceinline__ void zero_plates(const StepArgs &a, int x, double *__restrict__ f) {
  if (!a.walls || x >= a.nx || !f) return;
  if (blockIdx.y == 0) f[x] = 0.0;
  if ((a.ny - 1) % (int)gridDim.y == (int)blockIdx.y) f[(long long)(a.ny - 1) * a.nx + x] = 0.0;
}

// ------------------------------------------------------------------ fields
template <class S, bool DYN>
__global__ void __launch_bounds__(kReadBX, kReadPerSM)
    fields_kernel(const StepArgs a, const typename S::T *__restrict__ fin,
                  const float2 *__restrict__ med, double *__restrict__ rho,
                  double *__restrict__ ux, double *__restrict__ uy) {
  const PairIn<S> p(fin, med, a, blockIdx.x * kReadBX + threadIdx.x);
  zero_plates(a, p.x, rho);
  zero_plates(a, p.x, ux);
  zero_plates(a, p.x, uy);
  walk_column<DYN>(p, [&](const NodeStateT<float2> &s, int y, int z, bool both) {
    const long long j = (long long)y * a.nx + p.x, k = (long long)z * a.nx + p.x;
    if (rho) rho[j] = wide_value(s.rho.x);
    if (ux) ux[j] = wide_value(s.ux.x);
    if (uy) uy[j] = wide_value(s.uy.x);
    if (both) {
      if (rho) rho[k] = wide_value(s.rho.y);
      if (ux) ux[k] = wide_value(s.ux.y);
      if (uy) uy[k] = wide_value(s.uy.y);
    }
  });
}

// ------------------------------------------------------------- populations
// f_i = w_i rho0 + d_i / S: one FP64 operation per value, which bounds it (9 a
// node at ~1/64 of the FP32 rate, 260 us at 4096^2; 1062 -> 435 us a call).  shift: log2(1 / S).
template <class S, bool DYN>
__global__ void __launch_bounds__(kReadBX, kReadPerSM)
    pops_kernel(const StepArgs a, const typename S::T *__restrict__ fin,
                const float2 *__restrict__ med, int shift, double *__restrict__ pops) {
  const PairIn<S> p(fin, med, a, blockIdx.x * kReadBX + threadIdx.x);
  if (p.x >= a.nx) return;
  const long long n = (long long)a.nx * a.ny;
  const double r0 = (double)a.rho0;
  const double c0 = 4.0 / 9.0 * r0, c1 = 1.0 / 9.0 * r0, c2 = 1.0 / 36.0 * r0;
#pragma unroll 1
  for (int y = blockIdx.y; y < a.ny; y += gridDim.y) {
    double *o = pops + (long long)y * a.nx + p.x;
    if (!p.fluid(y)) {
      for (int i = 0; i < 9; ++i) o[i * n] = 0.0;
      continue;
    }
    float d[9];
    p.pull(y, d);
    if (p.column)
      pressure_node<S, DYN>(fin, med, a, p.x, y, med[(long long)y * a.pitch + p.x].x, d);
#pragma unroll
    for (int i = 0; i < 9; ++i)
      o[i * n] = __dadd_rn(i == 0 ? c0 : (i < 5 ? c1 : c2), wide_value(d[i], shift));
  }
}

// ------------------------------------------------------------------- sums
// True in the last block of the launch to arrive, whose threads then see
// the partials of all others.  *done returns to 0.
__device__ __forceinline__ bool last_block(unsigned *done) {
  __shared__ bool last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    const unsigned blocks = gridDim.x * gridDim.y;
    last = atomicInc(done, blocks - 1) == blocks - 1;
  }
  __syncthreads();
  __threadfence();
  return last;
}

// RES = false: sum u_x and sum (rho - rho0) into out[0], out[2]; RES = true:
// sum |u|^2 and sum |u - u_prev|^2 into out[3], out[4], and u_prev = u.  out[5]:
// nodes whose velocity or density is not finite.  A thread adds the terms of its
// nodes one by one in FP32 pairs (squares as exact products, differences as exact
// sums; ~2^-44 relative), the blocks and the last block add them up in FP64, in a
// fixed order.  out is pinned host memory.
// 4096^2 FP32, a whole call: k_g 279 -> 186 us, residual 346 -> 234 (scalar nodes,
// six FP64 block sums and a second launch over the partials before); the 738 MB
// take 109 us at the copy bandwidth, the rest is the issue of the loads' addresses.
template <class S, bool DYN, bool RES>
__global__ void __launch_bounds__(kReadBX, kReadPerSM)
    sums_kernel(const StepArgs a, const typename S::T *__restrict__ fin,
                const float2 *__restrict__ med, float2 *__restrict__ uprev,
                double *__restrict__ partials, unsigned *done, double *__restrict__ out) {
  const PairIn<S> p(fin, med, a, blockIdx.x * kReadBX + threadIdx.x);
  F2 sa = {0.0f, 0.0f}, sb = {0.0f, 0.0f};
  unsigned bad = 0;
  // The sums take scalar operations: the packed ones may be fused with the
  // products that they add, which the error-free sums do not survive.
  auto add = [&](float ux, float uy, float rho, float drho_s, float2 up) {
    if (!finite_node(ux, uy, rho)) {
      ++bad;
    } else if (RES) {
      sa = f2_add(sa, f2_add(two_prod(ux, ux), two_prod(uy, uy)));
      const F2 dx = two_sum(ux, -up.x), dy = two_sum(uy, -up.y);
      sb = f2_add(sb, f2_add(f2_mul(dx, dx), f2_mul(dy, dy)));
    } else {
      f2_acc(sa, ux);
      f2_acc(sb, drho_s);
    }
  };
  walk_column<DYN>(p, [&](const NodeStateT<float2> &s, int y, int z, bool both) {
    float2 vy = make_float2(0.0f, 0.0f), vz = vy;
    const long long jy = (long long)y * a.pitch + p.x, jz = (long long)z * a.pitch + p.x;
    if (RES) {
      vy = uprev[jy];
      vz = uprev[jz];
    }
    add(s.ux.x, s.uy.x, s.rho.x, s.drho_s.x, vy);
    if (RES) uprev[jy] = make_float2(s.ux.x, s.uy.x);
    if (both) {
      add(s.ux.y, s.uy.y, s.rho.y, s.drho_s.y, vz);
      if (RES) uprev[jz] = make_float2(s.ux.y, s.uy.y);
    }
  });
  Sums v = {(double)sa.hi + (double)sa.lo, (double)sb.hi + (double)sb.lo, bad};
  if (!RES) v.b *= (double)a.inv_scale;
  v = block_sums(v);
  const int blocks = (int)(gridDim.x * gridDim.y);
  if (threadIdx.x == 0) {
    double *p = partials + 3 * ((long long)blockIdx.y * gridDim.x + blockIdx.x);
    p[0] = v.a;
    p[1] = v.b;
    p[2] = (double)v.bad;
  }
  if (!last_block(done)) return;
  v = {0.0, 0.0, 0u};
  Sums nbad = {0.0, 0.0, 0u};
  for (int b = threadIdx.x; b < blocks; b += kReadBX) {
    v.a += __ldcg(partials + 3 * b);
    v.b += __ldcg(partials + 3 * b + 1);
    nbad.a += __ldcg(partials + 3 * b + 2);
  }
  v = block_sums(v);
  nbad = block_sums(nbad);
  if (threadIdx.x == 0) {
    out[RES ? 3 : 0] = v.a;
    out[RES ? 4 : 2] = v.b;
    out[5] = nbad.a;
  }
}

// ------------------------------------------- normalised-velocity histogram
// |u|^2 of a node in FP64 from the FP32 velocity of node_state (as the
// fields kernel reports it), every operation rounded separately so that the bin
// decisions can be replayed exactly on the host: |u| = sqrt(|u|^2), bin
// min(floor(|u| / max|u| nbins), nbins - 1).
__device__ __forceinline__ double speed2(float vx, float vy) {
  const double ux = vx, uy = vy;
  return __dadd_rn(__dmul_rn(ux, ux), __dmul_rn(uy, uy));
}
// The FP32 estimate of |u|^2 2^60 that decides whether the FP64 value is
// needed: relative error < 2^-21 between kTiny and the largest FP32 number.
constexpr float kTiny = 1e-30f;
__device__ __forceinline__ float speed2_estimate(float ux, float uy) {
  const float vx = ux * 0x1p30f, vy = uy * 0x1p30f;
  return fmaf(vx, vx, vy * vy);
}

// Pass 1: max |u| into out[0] (pinned host memory) and *umax.  The square
// root is monotonic, so the largest |u|^2 gives it; a node's FP64 square is
// formed only when its estimate can reach the thread's maximum (the two passes
// at 4096^2: 2041 us with FP64 squares, roots and quotients per node, now 348).  Non-negative
// doubles order as their bits; a non-finite speed counts as infinite.
template <class S, bool DYN>
__global__ void __launch_bounds__(kReadBX, kReadPerSM)
    speed_max_kernel(const StepArgs a, const typename S::T *__restrict__ fin,
                     const float2 *__restrict__ med, double *__restrict__ partials, unsigned *done,
                     double *__restrict__ umax, double *__restrict__ out) {
  const PairIn<S> p(fin, med, a, blockIdx.x * kReadBX + threadIdx.x);
  constexpr unsigned long long kInf = 0x7ff0000000000000ull;
  unsigned long long best = 0;
  float reach = 0.0f;  // estimates below it cannot be the maximum
  auto see = [&](float ux, float uy) {
    const float e = speed2_estimate(ux, uy);
    if (e < reach && e >= kTiny) return;
    if (ux == 0.0f && uy == 0.0f) return;
    const double q = speed2(ux, uy);
    const unsigned long long b = q >= 0.0 ? (unsigned long long)__double_as_longlong(q) : kInf;
    best = b > best ? b : best;
    reach = fmaxf(reach, e * 0.99999f);  // 1 - 1e-5 > both estimates' errors
  };
  walk_column<DYN>(p, [&](const NodeStateT<float2> &s, int, int, bool both) {
    see(s.ux.x, s.uy.x);
    if (both) see(s.ux.y, s.uy.y);
  });
  __shared__ unsigned long long red[kReadBX / 32];
  auto block_max = [&](unsigned long long v) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      const unsigned long long o = __shfl_down_sync(0xffffffffu, v, off);
      v = o > v ? o : v;
    }
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    for (int w = 0; w < kReadBX / 32; ++w) v = red[w] > v ? red[w] : v;
    return v;
  };
  best = block_max(best);
  const int blocks = (int)(gridDim.x * gridDim.y);
  if (threadIdx.x == 0)
    partials[(long long)blockIdx.y * gridDim.x + blockIdx.x] = __longlong_as_double((long long)best);
  if (!last_block(done)) return;
  best = 0;
  for (int b = threadIdx.x; b < blocks; b += kReadBX) {
    const unsigned long long v = (unsigned long long)__double_as_longlong(__ldcg(partials + b));
    best = v > best ? v : best;
  }
  best = block_max(best);
  if (threadIdx.x == 0) {
    const double u = __dsqrt_rn(__longlong_as_double((long long)best));
    *umax = u;
    *out = u;
  }
}

// Pass 2: the bins, counted per block in shared memory (a thread adds up
// runs of equal bins first: neighbouring nodes mostly share one), then added to
// counts.  A node whose FP32 estimate of |u| / max|u| nbins is clear of the bin
// edges (2^-19 relative, over four times its error) takes its bin from that; the
// others, and fields beyond the estimate's range, form the FP64 quotient.
template <class S, bool DYN>
__global__ void __launch_bounds__(kReadBX, kReadPerSM)
    histogram_kernel(const StepArgs a, const typename S::T *__restrict__ fin,
                     const float2 *__restrict__ med, const double *__restrict__ umax_p, int nbins,
                     unsigned long long *__restrict__ counts) {
  __shared__ unsigned sh[kMaxHistBins];
  for (int k = threadIdx.x; k < nbins; k += kReadBX) sh[k] = 0u;
  __syncthreads();
  const PairIn<S> p(fin, med, a, blockIdx.x * kReadBX + threadIdx.x);
  const double umax = *umax_p;
  // A non-finite velocity makes the maximum infinite and has no bin (its quotient is
  // NaN, no index): nothing is counted, the caller reports the lattice.
  if (!isfinite(umax)) return;
  const bool in_range = umax > 1e-20 && umax < 1e8;
  const float per = in_range ? (float)nbins / ((float)umax * 0x1p30f) : 0.0f;
  int run_bin = 0;
  unsigned run = 0;
  auto count = [&](float ux, float uy) {
    const float t = in_range ? sqrt_approx(speed2_estimate(ux, uy)) * per : 0.0f;
    int k;
    if (in_range && (t < 0.5f || fabsf(t - rintf(t)) > t * 0x1p-19f)) {
      k = t >= (float)(nbins - 1) ? nbins - 1 : (int)t;
    } else {
      const double u0 = __ddiv_rn(__dsqrt_rn(speed2(ux, uy)), umax);
      const double f = floor(__dmul_rn(u0, (double)nbins));
      k = f >= (double)(nbins - 1) ? nbins - 1 : (int)f;
    }
    if (k != run_bin) {
      if (run) atomicAdd(&sh[run_bin], run);
      run_bin = k;
      run = 0;
    }
    ++run;
  };
  walk_column<DYN>(p, [&](const NodeStateT<float2> &s, int, int, bool both) {
    if (!(umax > 0.0)) {  // no flow: every node in the first bin
      run += both ? 2u : 1u;
      return;
    }
    count(s.ux.x, s.uy.x);
    if (both) count(s.ux.y, s.uy.y);
  });
  if (run) atomicAdd(&sh[run_bin], run);
  __syncthreads();
  for (int k = threadIdx.x; k < nbins; k += kReadBX)
    if (sh[k]) atomicAdd(counts + k, (unsigned long long)sh[k]);
}

// ------------------------------------------------- apparent permeability
// 1 / (double)v, correctly rounded, for a positive normal v, by long division
// in 32-bit integers: with v = m 2^(E - 150), m of 24 bits, the 53-bit quotient
// 2^76 / m is formed 26 bits at a time from an FP32 reciprocal and exact
// remainders.  (An FP64 division per node took 196 us at 4096^2, this 88.)
static __device__ __noinline__ double wide_reciprocal_any(float v) { return 1.0 / (double)v; }
__device__ __forceinline__ double wide_reciprocal(float v) {
  const uint32_t u = __float_as_uint(v), E = u >> 23;
  if (u - 0x00800000u >= 0x7f000000u) return wide_reciprocal_any(v);  // 0, subnormal, inf, NaN, < 0
  const uint32_t m = (u & 0x7fffffu) | 0x800000u;
  if (m == 0x800000u) return wide_reciprocal_any(v);  // a power of two: a 54-bit quotient
  const float r = rcp_approx((float)m);
  // quotient and remainder of n = 2^50 (32-bit arithmetic: the remainder of a
  // near quotient is small), then of the remainder times 2^26
  auto digits = [&](uint32_t n_low, float estimate, uint32_t &rem) {
    uint32_t q = (uint32_t)estimate;
    int t = (int)(n_low - q * m);
    const int c = (int)floorf((float)t * r);
    q += (uint32_t)c;
    t -= c * (int)m;
    if (t < 0) {
      --q;
      t += (int)m;
    } else if (t >= (int)m) {
      ++q;
      t -= (int)m;
    }
    rem = (uint32_t)t;
    return q;
  };
  uint32_t rem;
  const uint32_t hi = digits(0u, r * 0x1p50f, rem);
  const uint32_t lo = digits(rem << 26, (float)rem * r * 0x1p26f, rem);
  unsigned long long q = ((unsigned long long)hi << 26) + lo;
  if (2u * rem > m) ++q;  // to nearest (no ties: m is no power of two)
  return __longlong_as_double(
      (long long)(((unsigned long long)(1149u - E) << 52) + (q - (1ull << 52))));
}

// k_a of every node of the fluid rows as the step sees it: 1 / (stored
// 1/k_a), or with a dynamic Kn 1 / ((1/k_i) / f_c(Kn0)) at the pressure
// p0 (q = 1) with the step's own FP32 f_c.  Plate rows read 0, open pores inf.
__global__ void __launch_bounds__(kReadBX)
    ka_kernel(const float2 *__restrict__ med, const float *__restrict__ kn0, int nx, int ny,
              int pitch, int y_lo, int y_hi, int kn_model, double *__restrict__ ka) {
  const int y = blockIdx.y;
  const int x = blockIdx.x * kReadBX + threadIdx.x;
  if (x >= nx) return;
  double v = 0.0;
  if (y >= y_lo && y < y_hi) {
    const long long jp = (long long)y * pitch + x;
    float inv = med[jp].y;
    if (kn0) inv = inv_ka_dynamic(inv, kn0[jp], kn_model);  // the step's form at p = p0
    v = wide_reciprocal(inv);  // inf for an open pore (1/k_a = 0)
  }
  ka[(long long)y * nx + x] = v;
}

cudaError_t launch_ka(const float2 *med, const float *kn0, int nx, int ny, int pitch, int y_lo,
                      int y_hi, int kn_model, double *ka, cudaStream_t s) {
  dim3 grid((nx + kReadBX - 1) / kReadBX, ny);
  ka_kernel<<<grid, kReadBX, 0, s>>>(med, kn0, nx, ny, pitch, y_lo, y_hi, kn_model, ka);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- launches
#define LBMP_READ(KERNEL, ...)                                                              \
  do {                                                                                      \
    const dim3 grid = read_grid(a);                                                         \
    if (storage == 0) {                                                                     \
      if (a.kn0)                                                                            \
        KERNEL(StoreF32, true)<<<grid, kReadBX, 0, s>>>(a, (const float *)fin, med, __VA_ARGS__);   \
      else                                                                                  \
        KERNEL(StoreF32, false)<<<grid, kReadBX, 0, s>>>(a, (const float *)fin, med, __VA_ARGS__);  \
    } else {                                                                                \
      if (a.kn0)                                                                            \
        KERNEL(StoreF16, true)<<<grid, kReadBX, 0, s>>>(a, (const __half *)fin, med, __VA_ARGS__);  \
      else                                                                                  \
        KERNEL(StoreF16, false)<<<grid, kReadBX, 0, s>>>(a, (const __half *)fin, med, __VA_ARGS__); \
    }                                                                                       \
    return cudaGetLastError();                                                              \
  } while (0)

cudaError_t launch_fields(int storage, const StepArgs &a, const void *fin, const float2 *med,
                          double *rho, double *ux, double *uy, cudaStream_t s) {
#define K(S, D) fields_kernel<S, D>
  LBMP_READ(K, rho, ux, uy);
#undef K
}

cudaError_t launch_pops(int storage, const StepArgs &a, const void *fin, const float2 *med,
                        double *pops, cudaStream_t s) {
  int shift = 0;
  frexpf(a.inv_scale, &shift);
  --shift;  // inv_scale = 2^shift
#define K(S, D) pops_kernel<S, D>
  LBMP_READ(K, shift, pops);
#undef K
}

cudaError_t launch_sums(int storage, const StepArgs &a, const void *fin, const float2 *med,
                        double *partials, unsigned *done, double *out, cudaStream_t s) {
#define K(S, D) sums_kernel<S, D, false>
  LBMP_READ(K, nullptr, partials, done, out);
#undef K
}

cudaError_t launch_residual_sums(int storage, const StepArgs &a, const void *fin,
                                 const float2 *med, float2 *uprev, double *partials,
                                 unsigned *done, double *out, cudaStream_t s) {
#define K(S, D) sums_kernel<S, D, true>
  LBMP_READ(K, uprev, partials, done, out);
#undef K
}

cudaError_t launch_speed_max(int storage, const StepArgs &a, const void *fin, const float2 *med,
                             double *partials, unsigned *done, double *umax, double *out,
                             cudaStream_t s) {
#define K(S, D) speed_max_kernel<S, D>
  LBMP_READ(K, partials, done, umax, out);
#undef K
}

cudaError_t launch_histogram(int storage, const StepArgs &a, const void *fin, const float2 *med,
                             const double *umax, int nbins, unsigned long long *counts,
                             cudaStream_t s) {
#define K(S, D) histogram_kernel<S, D>
  LBMP_READ(K, umax, nbins, counts);
#undef K
}

}  // namespace lbmp
