// Device building blocks of the read-outs: nodes of the current time level,
// two at a time, and exact FP64 values of FP32 results without FP64 arithmetic.
#pragma once

#include <stdint.h>

#include "lattice.cuh"

namespace lbmp {

// Two nodes of one column (rows y and z) in the lanes of float2 values: their
// loads are in flight together and the packed arithmetic serves both (each lane
// gives the bits of one node).  Addresses are cheap: the rows' bases are uniform
// over the block and the neighbours' columns are the thread's own constants.
template <class S>
struct PairIn {
  using T = typename S::T;
  const T *fin;
  const float2 *med;
  const StepArgs &a;
  int x, xl, xr;   // the column, and the sources' columns for e_x = +1, -1
  bool column;     // a pressure column

  __device__ __forceinline__ PairIn(const T *f, const float2 *m, const StepArgs &args, int col)
      : fin(f), med(m), a(args), x(col) {
    xl = x == 0 ? a.nx - 1 : x - 1;
    xr = x == a.nx - 1 ? 0 : x + 1;
    column = a.pressure && (x == 0 || x == a.nx - 1);
  }
  __device__ __forceinline__ bool fluid(int y) const {
    return y < a.ny && !(a.walls && (y == 0 || y == a.ny - 1));
  }
  // Post-stream values of node (x, y) (y a fluid row).  At a plate the
  // directions that would come from it are the node's own opposite ones: planes
  // 4, 7, 8 in the place of 2, 5, 6 (two planes up), or the reverse.
  __device__ __forceinline__ void pull(int y, float d[9]) const {
    const long long P = a.plane;
    const T *c = fin + (long long)y * a.pitch;
    const bool pb = a.walls && y == 1, pt = a.walls && y == a.ny - 2;
    const T *u = pb ? c + 2 * P : fin + (long long)(y == 0 ? a.ny - 1 : y - 1) * a.pitch;
    const T *w = pt ? c - 2 * P : fin + (long long)(y == a.ny - 1 ? 0 : y + 1) * a.pitch;
    const int ul = pb ? x : xl, ur = pb ? x : xr, wl = pt ? x : xl, wr = pt ? x : xr;
    d[0] = S::ld1(c + x);
    d[1] = S::ld1(c + P + xl);
    d[3] = S::ld1(c + 3 * P + xr);
    d[2] = S::ld1(u + 2 * P + x);
    d[5] = S::ld1(u + 5 * P + ul);
    d[6] = S::ld1(u + 6 * P + ur);
    d[4] = S::ld1(w + 4 * P + x);
    d[7] = S::ld1(w + 7 * P + wr);
    d[8] = S::ld1(w + 8 * P + wl);
  }
  // What the states of rows y and z (both fluid, z = y for a lone row) are
  // formed from; loads and arithmetic apart, so that the loads of the next two
  // rows are in flight meanwhile.
  struct Raw {
    float dy[9], dz[9];
    float2 my, mz, k0;
    int y, z;
  };
  template <bool DYN>
  __device__ __forceinline__ void load(int y, int z, Raw &r) const {
    pull(y, r.dy);
    pull(z, r.dz);
    const long long jy = (long long)y * a.pitch + x, jz = (long long)z * a.pitch + x;
    r.my = med[jy];
    r.mz = med[jz];
    r.k0 = DYN ? make_float2(a.kn0[jy], a.kn0[jz]) : make_float2(0.0f, 0.0f);
    r.y = y;
    r.z = z;
  }
  template <bool DYN>
  __device__ __forceinline__ NodeStateT<float2> state(Raw &r) const {
    if (column) {
      pressure_node<S, DYN>(fin, med, a, x, r.y, r.my.x, r.dy);
      pressure_node<S, DYN>(fin, med, a, x, r.z, r.mz.x, r.dz);
    }
    float2 d[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) d[i] = make_float2(r.dy[i], r.dz[i]);
    return node_state_t<float2, DYN>(d, make_float2(r.my.x, r.mz.x), make_float2(r.my.y, r.mz.y),
                                     a, r.k0);
  }
};
__device__ __forceinline__ bool finite_node(float ux, float uy, float rho) {
  return isfinite(ux) && isfinite(uy) && isfinite(rho);
}

// (double)v * 2^shift, exact, with integer operations: FP64 instructions,
// conversions included, run at ~1/64 of the FP32 rate on this GPU.
// (Out of line: the compiler would otherwise run the FP64 form beside the other.)
static __device__ __noinline__ double wide_subnormal(float v, int shift) {
  return (double)v * __hiloint2double((1023 + shift) << 20, 0);
}
__device__ __forceinline__ double wide_value(float v, int shift = 0) {
  const uint32_t u = __float_as_uint(v), mag = u & 0x7fffffffu;
  if (mag - 0x00800000u < 0x7f000000u)  // a normal number
    return __hiloint2double((int)((u & 0x80000000u) | ((mag >> 3) + ((uint32_t)(896 + shift) << 20))),
                            (int)(u << 29));
  if (mag == 0u) return __hiloint2double((int)u, 0);
  return wide_subnormal(v, shift);  // or not finite
}

constexpr int kReadBX = 256;  // threads of a read-out block

// Block sums of two FP64 values and a count, in a fixed order (thread 0).
struct Sums {
  double a, b;
  unsigned bad;
};
__device__ __forceinline__ Sums block_sums(Sums v) {
  __shared__ Sums red[kReadBX / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    v.a += __shfl_down_sync(0xffffffffu, v.a, off);
    v.b += __shfl_down_sync(0xffffffffu, v.b, off);
    v.bad += __shfl_down_sync(0xffffffffu, v.bad, off);
  }
  __syncthreads();
  if (lane == 0) red[warp] = v;
  __syncthreads();
  v = red[0];
  for (int w = 1; w < kReadBX / 32; ++w) {
    v.a += red[w].a;
    v.b += red[w].b;
    v.bad += red[w].bad;
  }
  return v;
}

}  // namespace lbmp
