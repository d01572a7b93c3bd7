// Several time steps per launch for small lattices (Chen et al.,
// arXiv:1411.7051, Section III, Eq. 12-17).
//
// A lattice of some 10^3 - 10^5 nodes spends a step's time on the launch and on
// the latency of one node update, not on bandwidth or issue.  Here a block
// takes a tile of the lattice with a halo of L nodes into shared memory, runs
// L time steps on it -- the region shrinks by one node on every side per step, so
// no block waits for another -- and writes the tile back.  The redundant halo
// updates cost issue slots that such a lattice leaves idle.  410 x 200: 6 steps a
// launch of 12 us (launch and loads 4 - 5, a level 1.2: the issue of some 330
// instructions a unit and the chain of a node update), 2.9 -> 2.1 us a step.
//
// A thread updates two rows of one column at a time in the lanes of the packed
// arithmetic, with the operations, the order and the rounding bits of the
// single-step kernels: the populations are the same to the last bit.
#pragma once

#include <cuda_fp16.h>
#include <stdint.h>

#include "fused.cuh"
#include "kernels.h"
#include "lattice.cuh"

namespace lbmp {

constexpr int kTileWarps = 16;   // 128 registers a thread
constexpr int kTileMaxLevels = 16;

// Shared memory of a block: two copies of the populations and the medium, in
// planes of a constant number of nodes (so that plane offsets are immediates).
template <class S, bool DYN>
struct TileCfg {
  using T = typename S::T;
  static constexpr int kNodeBytes = 18 * (int)sizeof(T) + 8 + (DYN ? 4 : 0);
  static constexpr int kNodes = 226 * 1024 / kNodeBytes / 32 * 32;
  static constexpr int kSmemBytes = kNodes * kNodeBytes;
};

template <class S, bool SR, bool DYN, bool FORCH>
__global__ void __launch_bounds__(kTileWarps * 32, 1)
    tile_step_kernel(const StepArgs a0, const typename S::T *fin,
                     typename S::T *__restrict__ fout, const float2 *__restrict__ med,
                     const unsigned long long *tctr, int k, const TilePlan p,
                     int levels, int rows) {
  using T = typename S::T;
  using L = LaneRaw<S, float>;
  constexpr int PL = TileCfg<S, DYN>::kNodes;
  extern __shared__ __align__(16) unsigned char smem[];
  StepArgs a = a0;
  a.forch = FORCH;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int i = blockIdx.x % p.tx, j = blockIdx.x / p.tx;
  const int y_end = a.y0 + rows;
  // the tile, and the region that it is computed from
  const int cx0 = (int)((long long)i * a.nx / p.tx), cx1 = (int)((long long)(i + 1) * a.nx / p.tx);
  const int cy0 = a.y0 + (int)((long long)j * rows / p.ty),
            cy1 = a.y0 + (int)((long long)(j + 1) * rows / p.ty);
  const int gx0 = cx0 - levels, gy0 = cy0 - levels;
  const int w = cx1 - cx0 + 2 * levels, h = cy1 - cy0 + 2 * levels;
  float2 *const sm = reinterpret_cast<float2 *>(smem);
  float *const sk = reinterpret_cast<float *>(sm + PL);
  T *const buf = reinterpret_cast<T *>(sk + (DYN ? PL : 0));  // the two copies
  auto wrap = [](int v, int n) {
    while (v < 0) v += n;
    while (v >= n) v -= n;
    return v;
  };
  chain_wait();
  // Beyond a pressure column or a fluid row next to a plate nothing is read.
  const bool inside = gx0 >= 0 && gx0 + w <= a.nx && gy0 >= a.y0 && gy0 + h <= y_end;
  for (int q = threadIdx.x; q < w * h; q += kTileWarps * 32) {
    const int r = q / w;
    int gx = gx0 + (q - r * w), gy = gy0 + r;
    if (!inside) {
      if (a.pressure && (gx < 0 || gx >= a.nx)) continue;
      if (a.walls && (gy < a.y0 || gy >= y_end)) continue;
      gx = wrap(gx, a.nx);
      gy = wrap(gy, a.ny);
    }
    const long long o = (long long)gy * a.pitch + gx;
    const T *const g = fin + o;
    const float2 m = med[o];
    const float k0 = DYN ? a.kn0[o] : 0.0f;
    T v[9];
#pragma unroll
    for (int d = 0; d < 9; ++d) v[d] = g[d * a.plane];
#pragma unroll
    for (int d = 0; d < 9; ++d) buf[d * PL + q] = v[d];
    sm[q] = m;
    if (DYN) sk[q] = k0;
  }
  // columns and rows of the region that lie inside the lattice, where it ends
  const int c_min = a.pressure ? -gx0 : 0, c_max = a.pressure ? a.nx - gx0 : w;
  const int r_min = a.walls ? a.y0 - gy0 : 0, r_max = a.walls ? y_end - gy0 : h;
  unsigned long long t0 = 0;
  if (SR) t0 = *tctr + (unsigned long long)k;
  __syncthreads();
#pragma unroll 1
  for (int l = 1; l <= levels; ++l) {
    const int src = (l & 1) ? 0 : 9 * PL, dst = 9 * PL - src;  // in buf
    const bool last = l == levels;
    // the region of this level
    const int c_lo = max(l, c_min), c_hi = min(w - l, c_max);
    const int r_lo = max(l, r_min), r_hi = min(h - l, r_max);
    const uint32_t ts = SR ? level_hash(a, t0 + (unsigned long long)(l - 1)) : 0u;
    // post-stream values of node (c, r); at a plate the node's own opposite ones
    auto pull = [&](int c, int r, float d[9]) {
      const int q = src + r * w + c;
      int u = q - w, b = q + w, u5 = u - 1, u6 = u + 1, b7 = b + 1, b8 = b - 1;
      if (a.walls) {
        if (gy0 + r == a.y0) u = u5 = u6 = q + 2 * PL;
        if (gy0 + r == y_end - 1) b = b7 = b8 = q - 2 * PL;
      }
      d[0] = S::ld1(buf + q);
      d[1] = S::ld1(buf + q + (PL - 1));
      d[3] = S::ld1(buf + q + (3 * PL + 1));
      d[2] = S::ld1(buf + u + 2 * PL);
      d[5] = S::ld1(buf + u5 + 5 * PL);
      d[6] = S::ld1(buf + u6 + 6 * PL);
      d[4] = S::ld1(buf + b + 4 * PL);
      d[7] = S::ld1(buf + b7 + 7 * PL);
      d[8] = S::ld1(buf + b8 + 8 * PL);
    };
    auto put = [&](int c, int r, const float d[9]) {
      long long o = 0;
      uint32_t hash = 0;
      if (SR || last) {
        const int x = gx0 + c, y = gy0 + r;  // inside the lattice at the last level
        o = last ? (long long)y * a.pitch + x
                 : (long long)wrap(y, a.ny) * a.pitch + wrap(x, a.nx);
        if (SR) hash = mix32((uint32_t)(o >> 1) ^ ts);
      }
      typename L::R v[9];
#pragma unroll
      for (int q = 0; q < 9; ++q)
        v[q] = L::template round<SR>(d[q], SR ? pair_bits(hash, q) : 0u, (int)(o & 1));
      if (last) {
#pragma unroll
        for (int q = 0; q < 9; ++q) L::store(fout + o + q * a.plane, v[q]);
      } else {
        const int g = dst + r * w + c;
#pragma unroll
        for (int q = 0; q < 9; ++q) L::keep(buf + g + q * PL, v[q]);
      }
    };
    // Units of two rows x 32 columns; then, one per 32 rows, the pressure columns
    // inside the region (a lane per row), whose chain of operations is twice as
    // long: they go to the first warps, the others follow.
    const int left = a.pressure && c_lo == c_min, right = a.pressure && c_hi == c_max;
    const int i_lo = c_lo + left, i_hi = c_hi - right;
    const int per_col = (r_hi - r_lo + 31) >> 5, cols = (left + right) * per_col;
    const int pairs = (r_hi - r_lo + 1) >> 1;
    const int units = cols + ((i_hi - i_lo + 31) >> 5) * pairs;
    for (int u = warp; u < units; u += kTileWarps) {
      if (u < cols) {
        const bool lo = left && u < per_col;
        const int r = r_lo + ((lo || !left ? u : u - per_col) << 5) + lane;
        const int c = lo ? c_lo : c_hi - 1, cn = lo ? c + 1 : c - 1;
        if (r >= r_hi) continue;
        float dn[9], d[9];
        pull(cn, r, dn);
        const int s = r * w + c, sn = r * w + cn;
        const float2 m = sm[s], mn = sm[sn];
        const NodeState n = node_state<DYN>(dn, mn.x, mn.y, a, DYN ? sk[sn] : 0.0f);
        column_from_neighbour(a, dn, n, mn.x, gx0 + c, m.x, d);
        const NodeState b = node_state<DYN>(d, m.x, m.y, a, DYN ? sk[s] : 0.0f);
        collide<S::kHiLo>(d, b, a);
        put(c, r, d);
        continue;
      }
      int rp = u - cols, c = i_lo + lane;
      while (rp >= pairs) {  // the next 32 columns
        rp -= pairs;
        c += 32;
      }
      if (c >= i_hi) continue;
      const int ra = r_lo + 2 * rp;
      const bool both = ra + 1 < r_hi;
      const int rb = both ? ra + 1 : ra;
      const int sa = ra * w + c, sb = rb * w + c;
      float da[9], db[9];
      pull(c, ra, da);
      pull(c, rb, db);
      const float2 ma = sm[sa], mb = sm[sb];
      const float2 k0 = DYN ? make_float2(sk[sa], sk[sb]) : make_float2(0.0f, 0.0f);
      float2 d[9];
#pragma unroll
      for (int q = 0; q < 9; ++q) d[q] = make_float2(da[q], db[q]);
      const NodeStateT<float2> s = node_state_t<float2, DYN>(
          d, make_float2(ma.x, mb.x), make_float2(ma.y, mb.y), a, k0);
      collide_t<S::kHiLo>(d, s, a);
#pragma unroll
      for (int q = 0; q < 9; ++q) {
        da[q] = d[q].x;
        db[q] = d[q].y;
      }
      put(c, ra, da);
      if (both) put(c, rb, db);
    }
    __syncthreads();
  }
}

}  // namespace lbmp
