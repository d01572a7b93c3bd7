// Two time steps in one pass over the lattice (Chen et al., arXiv:1411.7051,
// Section III, Eq. 12-17): the populations of level t are read from HBM, those
// of level t + 1 live in registers only, and level t + 2 is written back.
//
// Work split.  A warp owns a strip of 64 columns (a node pair per lane) and
// walks the rows of a segment upwards.  At row r it pulls and collides row r
// of level t (shifted sources come from the neighbouring lanes by shuffles),
// then row r - 1 of level t + 1, whose sources are the results of rows r - 2,
// r - 1 and r of the first level: the directions with e_y = -1 are used at
// once, those with e_y = 0 wait one row and those with e_y = +1 two rows, in
// registers, already shifted in x.  No shared memory, no barrier, no wait on
// another warp: warps recompute the two columns at each side of their strip
// (64 loaded, 60 stored; 128 and 124 with two pairs per lane) and two rows per
// segment.
//
// The columns that an interior strip cannot produce -- the first and the
// last ones of a row, with the periodic wrap or the pressure extrapolation --
// belong to edge warps, which run the same walk over the last and the first 16
// (or 8) columns of a row, for two (four) segments at a time: a node pair per
// lane where nx is even, one node (half the segments) where it is odd.
//
// Bound: FP32 by HBM (40 B an update, 4096^2: 190 us a step with one step per
// pass, 114 now, 0.87 of the copy bandwidth), FP16 by the issue of some
// 300 instructions a pair and step and too few warps to cover their latency
// (12 an SM; 112 -> 97 us).
//
// Every node is updated with the operations of the single-step kernels, in
// their order and with their stochastic-rounding bits, so the populations
// are the same to the last bit.
#pragma once

#include <cuda_fp16.h>
#include <stdint.h>

#include <cmath>

#include "chain.cuh"
#include "lattice.cuh"
#include "staged.cuh"

namespace lbmp {

constexpr int kFusedWarps = 4;     // warps (strips) per block
constexpr int kFusedMinNy = 6;     // a segment and its halo rows stay apart under the wrap

// Configuration of the interior strips: Q node pairs per lane, so a strip
// loads 64 Q columns and stores all but two at each side.  Each lane copies its
// own columns of the rows ahead into its part of a shared-memory FIFO
// (cp.async), kStages - 1 rows ahead of the row in use; the medium stays one
// row longer, for the second level.
template <class S, int Q, bool DYN>
struct FusedCfg {
  using T = typename S::T;
  static constexpr int kCols = 64 * Q;
  // Columns a strip stores: all but two at each side, or for FP32 with two
  // pairs per lane those of lanes 1 .. 30, whose rows start on 32-byte sectors
  // (4096^2: 114 us a step against 120 with 124 columns).
  static constexpr int kOut = sizeof(T) == 4 && Q == 2 ? 120 : kCols - 4;
  static constexpr int kLead = (kCols - kOut) / 2;
  static constexpr int kAlign = sizeof(T) == 4 && Q == 2 ? 8 : 4;  // of first columns
  static constexpr int kBlocks = Q == 1 ? 4 : 3;  // resident blocks per SM
  static constexpr int kStages = Q == 1 ? 3 : 2;
  static constexpr int kMedSlots = kStages + 1;
  static constexpr int kPlaneBytes = kCols * (int)sizeof(T);
  static constexpr int kPopBytes = 9 * kPlaneBytes;
  static constexpr int kMedBytes = kCols * 8;
  static constexpr int kKnBytes = DYN ? kCols * 4 : 0;
  static constexpr int kWarpBytes = kStages * kPopBytes + kMedSlots * (kMedBytes + kKnBytes);
  static constexpr int kSmemBytes = kFusedWarps * kWarpBytes;
  static constexpr int kLaneBytes = 2 * Q * (int)sizeof(T);  // of one direction
  static_assert(kBlocks * (kSmemBytes + 1024) <= 228 * 1024, "shared memory of the blocks of an SM");
};

// Global -> shared copy of BYTES (4, 8 or 16) by one thread.
template <int BYTES>
__device__ __forceinline__ void lane_copy(uint32_t dst, const void *src) {
  if constexpr (BYTES == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(dst), "l"(src), "n"(BYTES)
                 : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void copy_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Stores to global memory: the batched kernel reads its buffer pointers from
// memory, where the compiler cannot see their address space.
__device__ __forceinline__ void put_global(float *p, float v) {
  asm volatile("st.global.f32 [%0], %1;" ::"l"(p), "f"(v) : "memory");
}
__device__ __forceinline__ void put_global(float *p, float2 v) {
  asm volatile("st.global.v2.f32 [%0], {%1, %2};" ::"l"(p), "f"(v.x), "f"(v.y) : "memory");
}
__device__ __forceinline__ void put_global(float *p, float2 a, float2 b) {
  asm volatile("st.global.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(a.x), "f"(a.y), "f"(b.x),
               "f"(b.y)
               : "memory");
}
__device__ __forceinline__ void put_global(__half *p, uint32_t v) {
  asm volatile("st.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ void put_global(__half *p, uint32_t a, uint32_t b) {
  asm volatile("st.global.v2.u32 [%0], {%1, %2};" ::"l"(p), "r"(a), "r"(b) : "memory");
}
__device__ __forceinline__ void put_global(__half *p, unsigned short v) {
  asm volatile("st.global.u16 [%0], %1;" ::"l"(p), "h"(v) : "memory");
}

// What a lane holds of one direction, in the precision of the storage: the
// node pair (x, x + 1) for V = float2, one node for V = float.
template <class S, class V>
struct LaneRaw;

template <>
struct LaneRaw<StoreF32, float2> {
  using R = float2;
  static __device__ __forceinline__ R load(const float *p) {
    return *reinterpret_cast<const float2 *>(p);
  }
  static __device__ __forceinline__ R from_left(R v) {  // sources at x - 1
    return make_float2(__shfl_up_sync(0xffffffffu, v.y, 1), v.x);
  }
  static __device__ __forceinline__ R from_right(R v) {  // sources at x + 1
    return make_float2(v.y, __shfl_down_sync(0xffffffffu, v.x, 1));
  }
  static __device__ __forceinline__ float2 value(R v) { return v; }
  template <bool SR>
  static __device__ __forceinline__ R round(float2 v, uint32_t, int) { return v; }
  static __device__ __forceinline__ void store(float *p, R v) { put_global(p, v); }
};

template <>
struct LaneRaw<StoreF32, float> {
  using R = float;
  static __device__ __forceinline__ R load(const float *p) { return *p; }
  static __device__ __forceinline__ R from_left(R v) { return __shfl_up_sync(0xffffffffu, v, 1); }
  static __device__ __forceinline__ R from_right(R v) {
    return __shfl_down_sync(0xffffffffu, v, 1);
  }
  static __device__ __forceinline__ float value(R v) { return v; }
  template <bool SR>
  static __device__ __forceinline__ R round(float v, uint32_t, int) { return v; }
  static __device__ __forceinline__ void store(float *p, R v) { put_global(p, v); }
  static __device__ __forceinline__ void keep(float *p, R v) { *p = v; }  // any memory
};

template <>
struct LaneRaw<StoreF16, float2> {
  using R = uint32_t;  // half of node x in the low 16 bits, of node x + 1 in the high ones
  static __device__ __forceinline__ R load(const __half *p) {
    return *reinterpret_cast<const uint32_t *>(p);
  }
  static __device__ __forceinline__ R from_left(R v) {
    return __byte_perm(__shfl_up_sync(0xffffffffu, v, 1), v, 0x5432);
  }
  static __device__ __forceinline__ R from_right(R v) {
    return __byte_perm(v, __shfl_down_sync(0xffffffffu, v, 1), 0x5432);
  }
  static __device__ __forceinline__ float2 value(R v) {
    return __half22float2(*reinterpret_cast<const __half2 *>(&v));
  }
  // The rounding of StoreF16::st2 (bits: those of the pair and direction).
  template <bool SR>
  static __device__ __forceinline__ R round(float2 v, uint32_t bits, int) {
    uint32_t packed;
    if (SR) {
      asm("cvt.rs.f16x2.f32 %0, %1, %2, %3;" : "=r"(packed) : "f"(v.y), "f"(v.x), "r"(bits));
    } else {
      const __half2 h = __floats2half2_rn(v.x, v.y);
      packed = *reinterpret_cast<const uint32_t *>(&h);
    }
    return packed;
  }
  static __device__ __forceinline__ void store(__half *p, R v) {
    put_global(p, v);
  }
};

template <>
struct LaneRaw<StoreF16, float> {
  using R = uint32_t;  // in the low 16 bits
  static __device__ __forceinline__ R load(const __half *p) {
    return *reinterpret_cast<const unsigned short *>(p);
  }
  static __device__ __forceinline__ R from_left(R v) { return __shfl_up_sync(0xffffffffu, v, 1); }
  static __device__ __forceinline__ R from_right(R v) {
    return __shfl_down_sync(0xffffffffu, v, 1);
  }
  static __device__ __forceinline__ float value(R v) {
    return __half2float(__ushort_as_half((unsigned short)v));
  }
  // One node of a pair: rounded in its half of the pair's word (odd = node
  // x + 1 of the pair).
  template <bool SR>
  static __device__ __forceinline__ R round(float v, uint32_t bits, int odd) {
    if (SR) {
      uint32_t packed;
      asm("cvt.rs.f16x2.f32 %0, %1, %1, %2;" : "=r"(packed) : "f"(v), "r"(bits));
      return odd ? packed >> 16 : packed & 0xffffu;
    }
    return __half_as_ushort(__float2half_rn(v));
  }
  static __device__ __forceinline__ void store(__half *p, R v) {
    put_global(p, (unsigned short)v);
  }
  static __device__ __forceinline__ void keep(__half *p, R v) {
    *reinterpret_cast<unsigned short *>(p) = (unsigned short)v;
  }
};

// Medium of a lane: porosity, 1/k_a (1/k_i with a dynamic Kn), Kn at p0.
template <class V>
struct LaneMed {
  V eps, inv_k, kn0;
};
template <bool DYN>
__device__ __forceinline__ void load_med(const StepArgs &a, const float2 *__restrict__ med,
                                         long long j, LaneMed<float2> &m) {
  const float4 v = __ldg(reinterpret_cast<const float4 *>(med + j));
  m.eps = make_float2(v.x, v.z);
  m.inv_k = make_float2(v.y, v.w);
  m.kn0 = DYN ? __ldg(reinterpret_cast<const float2 *>(a.kn0 + j)) : make_float2(0.0f, 0.0f);
}
template <bool DYN>
__device__ __forceinline__ void load_med(const StepArgs &a, const float2 *__restrict__ med,
                                         long long j, LaneMed<float> &m) {
  const float2 v = __ldg(med + j);
  m.eps = v.x;
  m.inv_k = v.y;
  m.kn0 = DYN ? __ldg(a.kn0 + j) : 0.0f;
}

// Moments and state of the node(s) of an edge lane from the pulled values d.
// The pressure columns take their populations from the interior neighbour
// first (non-equilibrium extrapolation): the other node of the pair, or with
// one node per lane the neighbouring lane's.
template <bool DYN>
__device__ __forceinline__ NodeStateT<float2> lane_state(float2 d[9], const LaneMed<float2> &m,
                                                         const StepArgs &a, int x) {
  NodeStateT<float2> s = node_state_t<float2, DYN>(d, m.eps, m.inv_k, a, m.kn0);
  if (!a.pressure) return s;
  const bool lo = x == 0, hi = x + 2 == a.nx;
  if (lo || hi) {
    float dn[9], db[9];
    NodeState sn;
#pragma unroll
    for (int i = 0; i < 9; ++i) dn[i] = lo ? d[i].y : d[i].x;
    sn.drho_s = lo ? s.drho_s.y : s.drho_s.x;
    sn.rho = lo ? s.rho.y : s.rho.x;
    sn.ux = lo ? s.ux.y : s.ux.x;
    sn.uy = lo ? s.uy.y : s.uy.x;
    column_from_neighbour(a, dn, sn, lo ? m.eps.y : m.eps.x, lo ? 0 : a.nx - 1,
                          lo ? m.eps.x : m.eps.y, db);
#pragma unroll
    for (int i = 0; i < 9; ++i) d[i] = lo ? make_float2(db[i], dn[i]) : make_float2(dn[i], db[i]);
    s = node_state_t<float2, DYN>(d, m.eps, m.inv_k, a, m.kn0);
  }
  return s;
}
template <bool DYN>
__device__ __forceinline__ NodeState lane_state(float d[9], const LaneMed<float> &m,
                                                const StepArgs &a, int x) {
  NodeState s = node_state<DYN>(d, m.eps, m.inv_k, a, m.kn0);
  if (!a.pressure) return s;
  const bool lo = x == 0, hi = x == a.nx - 1;
  const int lane = threadIdx.x & 31;
  const int src = lo ? lane + 1 : (hi ? lane - 1 : lane);
  float dn[9];
#pragma unroll
  for (int i = 0; i < 9; ++i) dn[i] = __shfl_sync(0xffffffffu, d[i], src);
  NodeState sn = s;
  sn.drho_s = __shfl_sync(0xffffffffu, s.drho_s, src);
  sn.rho = __shfl_sync(0xffffffffu, s.rho, src);
  sn.ux = __shfl_sync(0xffffffffu, s.ux, src);
  sn.uy = __shfl_sync(0xffffffffu, s.uy, src);
  const float eps_n = __shfl_sync(0xffffffffu, m.eps, src);
  if (lo || hi) {
    column_from_neighbour(a, dn, sn, eps_n, x, m.eps, d);
    s = node_state<DYN>(d, m.eps, m.inv_k, a, m.kn0);
  }
  return s;
}

__device__ __forceinline__ void store_moments(float *__restrict__ mom, long long plane,
                                              const NodeStateT<float2> &s) {
  *reinterpret_cast<float2 *>(mom) = s.drho_s;
  *reinterpret_cast<float2 *>(mom + plane) = s.mx;
  *reinterpret_cast<float2 *>(mom + 2 * plane) = s.my;
}
__device__ __forceinline__ void store_moments(float *__restrict__ mom, long long plane,
                                              const NodeState &s) {
  mom[0] = s.drho_s;
  mom[plane] = s.mx;
  mom[2 * plane] = s.my;
}

// Collision of the lane's node(s) of flat index o, rounded to the storage.
template <class S, bool SR, class V>
__device__ __forceinline__ void lane_collide(V d[9], const NodeStateT<V> &s, const StepArgs &a,
                                             long long o, uint32_t ts,
                                             typename LaneRaw<S, V>::R p[9]) {
  using L = LaneRaw<S, V>;
  collide_t<S::kHiLo>(d, s, a);
  const uint32_t h = SR ? mix32((uint32_t)(o >> 1) ^ ts) : 0u;
#pragma unroll
  for (int i = 0; i < 9; ++i)
    p[i] = L::template round<SR>(d[i], SR ? pair_bits(h, i) : 0u, (int)(o & 1));
}

// The walk of the edge warp: the same two levels for groups of lanes, each of
// which covers the last and the first win / 2 columns of the rows of its own
// segment (win = 16 or 32; of the window all columns but two at each end come
// out right), with a node pair per lane (V = float2, nx even) or one node.
// Rows [s0, s1) are the group's segment, seg >= s1 - s0 the rows every group
// walks: conditions on rows are per lane, and rows outside the segment and its
// halo are computed on clamped addresses and not used.  x_lo, x_hi: columns
// below x_lo or from x_hi on are stored.  MOM: the moments of levels t and t + 1
// go to mom1 and mom2.
template <class S, bool SR, bool DYN, bool MOM, class V>
__device__ __forceinline__ void fused_edges(const StepArgs &a, const typename S::T *fin,
                                            typename S::T *__restrict__ fout,
                                            const float2 *__restrict__ med, int win, int x_lo,
                                            int x_hi, int s0, int s1, int seg, int y_end,
                                            uint32_t ts1, uint32_t ts2, float *__restrict__ mom1,
                                            float *__restrict__ mom2) {
  using L = LaneRaw<S, V>;
  using R = typename L::R;
  using T = typename S::T;
  constexpr int kNodes = (int)(sizeof(V) / sizeof(float));  // per lane
  const long long P = a.plane;
  const int c = ((threadIdx.x * kNodes) & (win - 1)) - win / 2;  // column, from the row's end on
  const int x = c < 0 ? a.nx + c : c;
  const bool out = x < x_lo || x >= x_hi;
  auto wrap = [&](int y) { return y < 0 ? y + a.ny : (y >= a.ny ? y - a.ny : y); };
  // the row whose first level is computed in the place of row r
  auto row_of = [&](int r) {
    r = r < s1 ? r : s1;
    if (a.walls) r = r < a.y0 ? a.y0 : (r < y_end ? r : y_end - 1);
    return wrap(r);
  };
  R raw[9];
  LaneMed<V> m;
  // Sources of a row.  At a plate the directions that would come from it
  // are the node's own opposite ones, unshifted: planes 4, 7, 8 in the
  // place of 2, 5, 6 (two planes up), or the reverse.
  auto load_row = [&](int y) {
    const T *e = fin + (long long)y * a.pitch + x;
    const T *u = (a.walls && y == a.y0) ? e + 2 * P : fin + (long long)wrap(y - 1) * a.pitch + x;
    const T *d = (a.walls && y == y_end - 1) ? e - 2 * P
                                             : fin + (long long)wrap(y + 1) * a.pitch + x;
    raw[0] = L::load(e);
    raw[1] = L::load(e + P);
    raw[3] = L::load(e + 3 * P);
    raw[2] = L::load(u + 2 * P);
    raw[5] = L::load(u + 5 * P);
    raw[6] = L::load(u + 6 * P);
    raw[4] = L::load(d + 4 * P);
    raw[7] = L::load(d + 7 * P);
    raw[8] = L::load(d + 8 * P);
    load_med<DYN>(a, med, (long long)y * a.pitch + x, m);
  };
  load_row(row_of(s0 - 1));
  R h0 = R(), h1 = R(), h3 = R();   // e_y = 0 of row r - 1, shifted
  R b2 = R(), b5 = R(), b6 = R();   // e_y = +1 of row r - 2, shifted
  R c2 = R(), c5 = R(), c6 = R();   // e_y = +1 of row r - 1, shifted
  LaneMed<V> m1 = m;            // medium of row r - 1
#pragma unroll 1
  for (int n = 0; n <= seg + 1; ++n) {
    const int r = s0 - 1 + n, y = row_of(r);
    const LaneMed<V> m0 = m;
    V d[9];
    R p[9];
    R t5 = L::from_left(raw[5]), t6 = L::from_right(raw[6]);
    R t7 = L::from_right(raw[7]), t8 = L::from_left(raw[8]);
    d[0] = L::value(raw[0]);
    d[2] = L::value(raw[2]);
    d[4] = L::value(raw[4]);
    d[1] = L::value(L::from_left(raw[1]));
    d[3] = L::value(L::from_right(raw[3]));
    if (a.walls && y == a.y0) {
      t5 = raw[5];
      t6 = raw[6];
    }
    if (a.walls && y == y_end - 1) {
      t7 = raw[7];
      t8 = raw[8];
    }
    d[5] = L::value(t5);
    d[6] = L::value(t6);
    d[7] = L::value(t7);
    d[8] = L::value(t8);
    if (n <= seg) load_row(row_of(r + 1));
    {
      const NodeStateT<V> s = lane_state<DYN>(d, m0, a, x);
      const long long o = (long long)y * a.pitch + x;
      if (MOM && out && r >= s0 && r < s1) store_moments(mom1 + o, P, s);
      lane_collide<S, SR>(d, s, a, o, ts1, p);
    }
    R f4 = p[4], f7 = L::from_right(p[7]), f8 = L::from_left(p[8]);  // e_y = -1 of row r
    // beyond the last row below a plate: that row's own e_y = +1 values
    const R g7 = L::from_right(c5), g8 = L::from_left(c6);  // undo the shifts
    if (a.walls && r == y_end) {
      f4 = c2;
      f7 = g7;
      f8 = g8;
    }
    if (n >= 2) {  // second level at row r - 1
      d[0] = L::value(h0);
      d[1] = L::value(h1);
      d[3] = L::value(h3);
      d[2] = L::value(b2);
      d[5] = L::value(b5);
      d[6] = L::value(b6);
      d[4] = L::value(f4);
      d[7] = L::value(f7);
      d[8] = L::value(f8);
      const NodeStateT<V> s = lane_state<DYN>(d, m1, a, x);
      const long long o = (long long)(r - 1) * a.pitch + x;
      R q[9];
      lane_collide<S, SR>(d, s, a, o, ts2, q);
      if (out && r - 1 < s1) {
        if (MOM) store_moments(mom2 + o, P, s);
        T *g = fout + o;
#pragma unroll
        for (int i = 0; i < 9; ++i) L::store(g + i * P, q[i]);
      }
    }
    // row a.y0 bounces its e_y = -1 values off the plate below
    const bool plate = a.walls && r == a.y0;
    b2 = plate ? p[4] : c2;
    b5 = plate ? p[7] : c5;
    b6 = plate ? p[8] : c6;
    c2 = p[2];
    c5 = L::from_left(p[5]);
    c6 = L::from_right(p[6]);
    h0 = p[0];
    h1 = L::from_left(p[1]);
    h3 = L::from_right(p[3]);
    m1 = m0;
  }
}

// ---------------------------------------------------------- interior strips
// A lane's Q consecutive pairs of one direction, from a row in shared memory.
template <int Q>
__device__ __forceinline__ void lane_row(const float *row, int lane, float2 v[Q]) {
  if constexpr (Q == 2) {
    const float4 w = reinterpret_cast<const float4 *>(row)[lane];
    v[0] = make_float2(w.x, w.y);
    v[1] = make_float2(w.z, w.w);
  } else {
    v[0] = reinterpret_cast<const float2 *>(row)[lane];
  }
}
template <int Q>
__device__ __forceinline__ void lane_row(const __half *row, int lane, uint32_t v[Q]) {
  if constexpr (Q == 2) {
    const uint2 w = reinterpret_cast<const uint2 *>(row)[lane];
    v[0] = w.x;
    v[1] = w.y;
  } else {
    v[0] = reinterpret_cast<const uint32_t *>(row)[lane];
  }
}
template <int Q>
__device__ __forceinline__ void store_row(float *p, const float2 v[Q]) {
  if constexpr (Q == 2)
    put_global(p, v[0], v[1]);
  else
    put_global(p, v[0]);
}
template <int Q>
__device__ __forceinline__ void store_row(__half *p, const uint32_t v[Q]) {
  if constexpr (Q == 2)
    put_global(p, v[0], v[1]);
  else
    put_global(p, v[0]);
}

// Values one column to the left (right) of the lane's pairs.
__device__ __forceinline__ float2 pair_join(float2 a, float2 b) { return make_float2(a.y, b.x); }
__device__ __forceinline__ uint32_t pair_join(uint32_t a, uint32_t b) {
  return __byte_perm(a, b, 0x5432);
}
__device__ __forceinline__ float2 pair_up(float2 v) {
  return make_float2(0.0f, __shfl_up_sync(0xffffffffu, v.y, 1));
}
__device__ __forceinline__ uint32_t pair_up(uint32_t v) { return __shfl_up_sync(0xffffffffu, v, 1); }
__device__ __forceinline__ float2 pair_down(float2 v) {
  return make_float2(__shfl_down_sync(0xffffffffu, v.x, 1), 0.0f);
}
__device__ __forceinline__ uint32_t pair_down(uint32_t v) {
  return __shfl_down_sync(0xffffffffu, v, 1);
}
template <int Q, class R>
__device__ __forceinline__ void from_left(const R v[Q], R o[Q]) {
  const R e = pair_up(v[Q - 1]);
#pragma unroll
  for (int q = Q - 1; q > 0; --q) o[q] = pair_join(v[q - 1], v[q]);
  o[0] = pair_join(e, v[0]);
}
template <int Q, class R>
__device__ __forceinline__ void from_right(const R v[Q], R o[Q]) {
  const R e = pair_down(v[0]);
#pragma unroll
  for (int q = 0; q < Q - 1; ++q) o[q] = pair_join(v[q], v[q + 1]);
  o[Q - 1] = pair_join(v[Q - 1], e);
}
template <int Q, class R>
__device__ __forceinline__ void copy_row(const R v[Q], R o[Q]) {
#pragma unroll
  for (int q = 0; q < Q; ++q) o[q] = v[q];
}

// One level of a row: the lane's pairs from their pulled values t (stored
// precision) to the rounded post-collision ones, in place.  When every node
// of the warp is permeable (and, with a dynamic Kn, in the range of the
// fraction), the pairs run as straight-line code that the scheduler
// interleaves; otherwise pair by pair through the general form.
template <class S, bool SR, bool DYN, bool MOM, int Q>
__device__ __forceinline__ void level_row(typename LaneRaw<S, float2>::R t[9][Q],
                                          const unsigned char *ms, const StepArgs &a,
                                          long long o, uint32_t ts, bool mom_rows,
                                          float *__restrict__ mom) {
  using L = LaneRaw<S, float2>;
  using C = FusedCfg<S, Q, DYN>;
  const int lane = threadIdx.x & 31;
  float2 d[Q][9], eps[Q], inv_k[Q], kn[Q], c[Q];
  NodeStateT<float2> s[Q];
  bool fast = true;
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    const float4 m = reinterpret_cast<const float4 *>(ms)[lane * Q + q];
    eps[q] = make_float2(m.x, m.z);
    inv_k[q] = make_float2(m.y, m.w);
    fast = fast && eps[q].x > 0.0f && eps[q].y > 0.0f;
#pragma unroll
    for (int i = 0; i < 9; ++i) d[q][i] = L::value(t[i][q]);
    c[q] = node_moments<!S::kHiLo>(d[q], a, s[q]);
    if (DYN) {
      kn[q] = dynamic_kn(s[q].drho_s,
                         reinterpret_cast<const float2 *>(ms + C::kMedBytes)[lane * Q + q], a);
      fast = fast && kn_common(kn[q], a);
    }
  }
  if (__all_sync(0xffffffffu, fast)) {
#pragma unroll
    for (int q = 0; q < Q; ++q)
      porous_state<!S::kHiLo>(s[q], eps[q], DYN ? inv_ka_common(inv_k[q], kn[q]) : inv_k[q], c[q], a);
  } else {
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      const float2 k0 = DYN ? reinterpret_cast<const float2 *>(ms + C::kMedBytes)[lane * Q + q]
                            : make_float2(0.0f, 0.0f);
      s[q] = node_state_t<float2, DYN>(d[q], eps[q], inv_k[q], a, k0);
    }
  }
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    if (MOM && mom_rows && (C::kLead == 2 && Q == 2 ? (q == 0 ? lane > 0 : lane < 31) : lane > 0 && lane < 31))
      store_moments(mom + o + 2 * q, a.plane, s[q]);
    typename L::R p[9];
    lane_collide<S, SR, float2>(d[q], s[q], a, o + 2 * q, ts, p);
#pragma unroll
    for (int i = 0; i < 9; ++i) t[i][q] = p[i];
  }
}

// The walk of an interior strip (first column c0) over rows [s0, s1), as
// fused_edges, with the rows of level t copied ahead.
template <class S, bool SR, bool DYN, bool MOM, int Q>
__device__ __forceinline__ void fused_strip(const StepArgs &a, const typename S::T *fin,
                                            typename S::T *__restrict__ fout,
                                            const float2 *__restrict__ med, int c0, int s0, int s1,
                                            int y_end, uint32_t ts1, uint32_t ts2,
                                            float *__restrict__ mom1, float *__restrict__ mom2,
                                            unsigned char *ring) {
  using C = FusedCfg<S, Q, DYN>;
  using T = typename S::T;
  using R = typename LaneRaw<S, float2>::R;
  constexpr int NS = C::kStages, NM = C::kMedSlots;
  const int lane = threadIdx.x & 31;
  const long long P = a.plane;
  // the kLead columns at each side are not right: those of lanes 0 and 31, or
  // (kLead = 2 with two pairs a lane) half of theirs
  const bool out = lane >= 1 && lane <= 30;
  const int x = c0 + 2 * Q * lane;
  const int r0 = a.walls && s0 == a.y0 ? s0 : s0 - 1;
  const int r_last = a.walls && s1 == y_end ? s1 - 1 : s1;
  unsigned char *const meds = ring + NS * C::kPopBytes;
  const uint32_t pops_u = smem_u32(ring) + (uint32_t)(lane * C::kLaneBytes);
  const uint32_t meds_u = smem_u32(meds);
  auto wrap = [&](int y) { return y < 0 ? y + a.ny : (y >= a.ny ? y - a.ny : y); };
  // Copy row r into stage s and medium slot ms (one commit group per row).
  // At a plate the directions that would come from it are the node's own
  // opposite ones, unshifted: planes 4, 7, 8 in the place of 2, 5, 6 (two
  // planes up), or the reverse.
  auto copy = [&](int r, int s, int ms) {
    if (r <= r_last) {
      const int y = wrap(r);
      const T *m = fin + (long long)y * a.pitch + x;
      const T *u = (a.walls && y == a.y0) ? m + 2 * P : fin + (long long)wrap(r - 1) * a.pitch + x;
      const T *d = (a.walls && y == y_end - 1) ? m - 2 * P
                                               : fin + (long long)wrap(r + 1) * a.pitch + x;
      const uint32_t dst = pops_u + (uint32_t)(s * C::kPopBytes);
      auto put = [&](int i, const T *row) {
        lane_copy<C::kLaneBytes>(dst + (uint32_t)(i * C::kPlaneBytes), row + i * P);
      };
      put(0, m);
      put(1, m);
      put(3, m);
      put(2, u);
      put(5, u);
      put(6, u);
      put(4, d);
      put(7, d);
      put(8, d);
      const uint32_t md = meds_u + (uint32_t)(ms * (C::kMedBytes + C::kKnBytes));
      const long long j = (long long)y * a.pitch + x;
#pragma unroll
      for (int q = 0; q < Q; ++q)
        lane_copy<16>(md + (uint32_t)((lane * Q + q) * 16), med + j + 2 * q);
      if (DYN)
        lane_copy<8 * Q>(md + (uint32_t)(C::kMedBytes + lane * 8 * Q), a.kn0 + j);
    }
    copy_commit();
  };
#pragma unroll
  for (int n = 0; n < NS - 1; ++n) copy(r0 + n, n, n);
  R h0[Q], h1[Q], h3[Q];   // e_y = 0 of row r - 1, shifted
  R b2[Q], b5[Q], b6[Q];   // e_y = +1 of row r - 2, shifted
  R c2[Q], c5[Q], c6[Q];   // e_y = +1 of row r - 1, shifted
#pragma unroll
  for (int q = 0; q < Q; ++q)
    h0[q] = h1[q] = h3[q] = b2[q] = b5[q] = b6[q] = c2[q] = c5[q] = c6[q] = R();
  int st = 0, ms = 0;      // stage and medium slot of row r
#pragma unroll 1
  for (int r = r0; r <= s1; ++r) {
    R t[9][Q];
    R f4[Q], f7[Q], f8[Q];
    // row r + NS - 1 takes the stage that row r - 1 has left
    copy(r + NS - 1, st == 0 ? NS - 1 : st - 1, ms + NS - 1 < NM ? ms + NS - 1 : ms + NS - 1 - NM);
    const unsigned char *m_now = meds + ms * (C::kMedBytes + C::kKnBytes);
    const unsigned char *m_was = meds + (ms == 0 ? NM - 1 : ms - 1) * (C::kMedBytes + C::kKnBytes);
    if (r <= r_last) {
      const int y = wrap(r);
      copy_wait<NS - 1>();  // row r has landed
      const T *sp = reinterpret_cast<const T *>(ring + st * C::kPopBytes);
      R w[Q];
      lane_row<Q>(sp, lane, t[0]);
      lane_row<Q>(sp + 2 * C::kCols, lane, t[2]);
      lane_row<Q>(sp + 4 * C::kCols, lane, t[4]);
      lane_row<Q>(sp + 1 * C::kCols, lane, w);
      from_left<Q>(w, t[1]);
      lane_row<Q>(sp + 3 * C::kCols, lane, w);
      from_right<Q>(w, t[3]);
      lane_row<Q>(sp + 5 * C::kCols, lane, t[5]);
      lane_row<Q>(sp + 6 * C::kCols, lane, t[6]);
      lane_row<Q>(sp + 7 * C::kCols, lane, t[7]);
      lane_row<Q>(sp + 8 * C::kCols, lane, t[8]);
      if (!(a.walls && y == a.y0)) {
        copy_row<Q>(t[5], w);
        from_left<Q>(w, t[5]);
        copy_row<Q>(t[6], w);
        from_right<Q>(w, t[6]);
      }
      if (!(a.walls && y == y_end - 1)) {
        copy_row<Q>(t[7], w);
        from_right<Q>(w, t[7]);
        copy_row<Q>(t[8], w);
        from_left<Q>(w, t[8]);
      }
      level_row<S, SR, DYN, MOM, Q>(t, m_now, a, (long long)y * a.pitch + x, ts1,
                                    MOM && r >= s0 && r < s1, mom1);
      copy_row<Q>(t[4], f4);
      from_right<Q>(t[7], f7);
      from_left<Q>(t[8], f8);
    } else {
      // row r is a plate: row r - 1 gets its own e_y = +1 values back
      copy_row<Q>(c2, f4);
      from_right<Q>(c5, f7);  // undoes the shift of c5 (from the left)
      from_left<Q>(c6, f8);
    }
    if (r > s0) {
      R u[9][Q];
#pragma unroll
      for (int q = 0; q < Q; ++q) {
        u[0][q] = h0[q];
        u[1][q] = h1[q];
        u[2][q] = b2[q];
        u[3][q] = h3[q];
        u[4][q] = f4[q];
        u[5][q] = b5[q];
        u[6][q] = b6[q];
        u[7][q] = f7[q];
        u[8][q] = f8[q];
      }
      const long long o = (long long)(r - 1) * a.pitch + x;
      level_row<S, SR, DYN, MOM, Q>(u, m_was, a, o, ts2, MOM, mom2);
      T *g = fout + o;
      if (out) {
#pragma unroll
        for (int i = 0; i < 9; ++i) store_row<Q>(g + i * P, u[i]);
      } else if (C::kLead == 2 && Q == 2) {
        const int q = lane == 0 ? Q - 1 : 0;
#pragma unroll
        for (int i = 0; i < 9; ++i)
          LaneRaw<S, float2>::store(g + i * P + 2 * q, lane == 0 ? u[i][Q - 1] : u[i][0]);
      }
    }
    if (r <= r_last) {
      if (a.walls && r == a.y0) {  // its e_y = -1 values bounce off the plate below
        copy_row<Q>(t[4], b2);
        copy_row<Q>(t[7], b5);
        copy_row<Q>(t[8], b6);
      } else {
        copy_row<Q>(c2, b2);
        copy_row<Q>(c5, b5);
        copy_row<Q>(c6, b6);
      }
      copy_row<Q>(t[2], c2);
      from_left<Q>(t[5], c5);
      from_right<Q>(t[6], c6);
      copy_row<Q>(t[0], h0);
      from_left<Q>(t[1], h1);
      from_right<Q>(t[3], h3);
    }
    st = st + 1 < NS ? st + 1 : 0;
    ms = ms + 1 < NM ? ms + 1 : 0;
  }
}

// Strips of a lattice nx wide: `inner` interior ones, the first at column
// c0 and the others kOut apart (the last one moved left if it would leave the
// row; it then stores some columns again, with the same values), and the edge
// warp's columns below x_lo and from x_hi on, in windows of `win` columns.  A
// window of 16 covers 6 columns at each end of a row, one of 32 covers 14: the
// wider one where it saves a strip.  An edge warp holds `per` windows, of
// consecutive segments.
struct FusedStrips {
  int inner, c0, last, win, per, x_lo, x_hi;
};
template <class C>
__host__ __device__ inline FusedStrips fused_strips(int nx) {
  FusedStrips f{};
  for (int win = 32; win >= 16; win -= 16) {
    const int edge = win / 2 - 2;
    const int last = (nx - C::kCols) & ~3;
    int c0 = (edge - C::kLead) / C::kAlign * C::kAlign;
    c0 = c0 < last ? c0 : last;
    const int left = nx - edge - c0 - C::kLead;
    const int n = left > C::kOut ? (left + C::kOut - 1) / C::kOut : 1;
    const int end = c0 + (n - 1) * C::kOut < last ? c0 + (n - 1) * C::kOut : last;
    if (win == 32 || (n <= f.inner && nx - (end + C::kCols - C::kLead) <= edge)) {
      f = {n, c0, last, win, (nx & 1 ? 32 : 64) / win, c0 + C::kLead, end + C::kCols - C::kLead};
    }
  }
  return f;
}

// Relative time of a launch in segments of seg rows and w waves of resident
// warps, one warp per strip and segment.  A warp's time is that of its seg + 2
// rows (the two halo rows run the first level only), so small segments cost
// redundant rows and large ones leave the last wave uneven: up to one wave
// 0.7 + w / 2 (a partly filled chip runs each row faster), 2.2 up to two, w + 0.25
// beyond and a little more where the last wave is nearly empty.  Fitted to
// sweeps of seg at 512^2 .. 4096^2 (1024^2: 6 rows 9.8 us a step, 5 rows 11.4;
// 4096^2 FP32: 20 and 28 rows 111, 26 rows 114, one wave of 82 rows 121).
inline double fused_cost(int seg, double w) {
  if (w <= 1.0) return (seg + 2) * (0.7 + 0.5 * w);
  if (w <= 2.0) return (seg + 2) * 2.2;
  return (seg + 2) * (w + 0.25 + 0.15 * (std::ceil(w) - w));
}

// One warp's task: strip `strip` of the segment that starts at row s0, seg
// rows high at most; strip < 0: the edges of that segment and the next per - 1.
template <class S, bool SR, bool DYN, bool MOM, int Q>
__device__ __forceinline__ void fused_task(const StepArgs &a, const typename S::T *fin,
                                           typename S::T *__restrict__ fout,
                                           const float2 *__restrict__ med, const FusedStrips &f,
                                           int strip, int s0, int seg, int y_end, uint32_t ts1,
                                           uint32_t ts2, float *__restrict__ mom1,
                                           float *__restrict__ mom2, unsigned char *ring) {
  using C = FusedCfg<S, Q, DYN>;
  if (strip >= 0) {
    const int c0 = f.c0 + strip * C::kOut < f.last ? f.c0 + strip * C::kOut : f.last;
    const int s1 = s0 + seg < y_end ? s0 + seg : y_end;
    fused_strip<S, SR, DYN, MOM, Q>(a, fin, fout, med, c0, s0, s1, y_end, ts1, ts2, mom1, mom2,
                                    ring);
  } else {
    s0 += (int)((threadIdx.x & 31) / (32 / f.per)) * seg;
    // a window past the last row repeats the first segment, without storing
    const bool none = s0 >= y_end;
    s0 = none ? a.y0 : s0;
    const int s1 = s0 + seg < y_end ? s0 + seg : y_end;
    const int x_lo = none ? 0 : f.x_lo, x_hi = none ? a.nx : f.x_hi;
    if (a.nx & 1)
      fused_edges<S, SR, DYN, MOM, float>(a, fin, fout, med, f.win, x_lo, x_hi, s0, s1, seg, y_end,
                                          ts1, ts2, mom1, mom2);
    else
      fused_edges<S, SR, DYN, MOM, float2>(a, fin, fout, med, f.win, x_lo, x_hi, s0, s1, seg, y_end,
                                           ts1, ts2, mom1, mom2);
  }
}

// Time levels t, t + 1 of the stochastic rounding (t = *tctr + k).
__device__ __forceinline__ uint32_t level_hash(const StepArgs &a, unsigned long long t) {
  return mix32((uint32_t)t * 0x9e3779b9u ^ a.seed_lo ^ mix32((uint32_t)(t >> 32) ^ a.seed_hi));
}

// Task w of the launch: the edge warps first (they take longest per row),
// then strip by strip of segment after segment, seg rows high (the last one
// shorter).  FORCH = a0.forch, as a constant: no branch inside a row.
template <class S, bool SR, bool DYN, bool MOM, bool FORCH, int Q>
__global__ void __launch_bounds__(kFusedWarps * 32, FusedCfg<S, Q, DYN>::kBlocks)
    fused_step_kernel(const StepArgs a0, const typename S::T *fin,
                      typename S::T *__restrict__ fout, const float2 *__restrict__ med,
                      const unsigned long long *tctr, int k, int rows, int seg,
                      const FusedStrips f, int edges, int tasks, float *__restrict__ mom1,
                      float *__restrict__ mom2) {
  extern __shared__ __align__(128) unsigned char smem[];
  StepArgs a = a0;
  a.forch = FORCH;
  const int warp = threadIdx.x >> 5;
  const int w = blockIdx.x * kFusedWarps + warp;
  if (w >= tasks) return;
  const int strip = w < edges ? -1 : (w - edges) % f.inner;
  const int part = w < edges ? w * f.per : (w - edges) / f.inner;
  chain_wait();
  uint32_t ts1 = 0, ts2 = 0;
  if (SR) {
    const unsigned long long t = *tctr + (unsigned long long)k;
    ts1 = level_hash(a, t);
    ts2 = level_hash(a, t + 1);
  }
  fused_task<S, SR, DYN, MOM, Q>(a, fin, fout, med, f, strip, a.y0 + part * seg, seg, a.y0 + rows,
                                 ts1, ts2, mom1, mom2, smem + warp * FusedCfg<S, Q, DYN>::kWarpBytes);
}

}  // namespace lbmp
