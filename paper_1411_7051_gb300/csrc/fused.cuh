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
// (64 loaded, 60 stored) and two rows per segment.
//
// The columns that an interior strip cannot produce -- the first two and
// the last two or three of a row, with the periodic wrap or the pressure
// extrapolation -- belong to one more warp per segment, which runs the same
// walk with one node per lane over columns nx - 16 .. nx - 1, 0 .. 15.
//
// Every node is updated with the operations of the single-step kernels, in
// their order and with their stochastic-rounding bits, so the populations
// are the same to the last bit.
#pragma once

#include <cuda_fp16.h>
#include <stdint.h>

#include "lattice.cuh"
#include "staged.cuh"

namespace lbmp {

constexpr int kFusedWarps = 4;     // warps (strips) per block
constexpr int kFusedMinNy = 6;     // a segment and its halo rows stay apart under the wrap

// Configuration of the interior strips: Q node pairs per lane, so a strip
// loads 64 Q columns and stores those of lanes 1 .. 30.  Each lane copies its
// own columns of the rows ahead into its part of a shared-memory FIFO
// (cp.async), kStages - 1 rows ahead of the row in use; the medium stays one
// row longer, for the second level.
template <class S, int Q, bool DYN>
struct FusedCfg {
  using T = typename S::T;
  static constexpr int kCols = 64 * Q, kHalo = 2 * Q;
  static constexpr int kOut = 60 * Q;             // from one strip to the next
  static constexpr int kBlocks = Q == 1 ? 5 : 3;  // resident blocks per SM
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

// What a lane holds of one direction, in the precision of the storage: the
// node pair (x, x + 1) for V = float2, one node for V = float.
template <class S, class V>
struct LaneRaw;

template <>
struct LaneRaw<StoreF32, float2> {
  using R = float2;
  static __device__ __forceinline__ R load(const float *p) {
    return __ldg(reinterpret_cast<const float2 *>(p));
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
  static __device__ __forceinline__ void store(float *p, R v) {
    *reinterpret_cast<float2 *>(p) = v;
  }
};

template <>
struct LaneRaw<StoreF32, float> {
  using R = float;
  static __device__ __forceinline__ R load(const float *p) { return __ldg(p); }
  static __device__ __forceinline__ R from_left(R v) { return __shfl_up_sync(0xffffffffu, v, 1); }
  static __device__ __forceinline__ R from_right(R v) {
    return __shfl_down_sync(0xffffffffu, v, 1);
  }
  static __device__ __forceinline__ float value(R v) { return v; }
  template <bool SR>
  static __device__ __forceinline__ R round(float v, uint32_t, int) { return v; }
  static __device__ __forceinline__ void store(float *p, R v) { *p = v; }
};

template <>
struct LaneRaw<StoreF16, float2> {
  using R = uint32_t;  // half of node x in the low 16 bits, of node x + 1 in the high ones
  static __device__ __forceinline__ R load(const __half *p) {
    return __ldg(reinterpret_cast<const uint32_t *>(p));
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
    *reinterpret_cast<uint32_t *>(p) = v;
  }
};

template <>
struct LaneRaw<StoreF16, float> {
  using R = uint32_t;  // in the low 16 bits
  static __device__ __forceinline__ R load(const __half *p) {
    return __ldg(reinterpret_cast<const unsigned short *>(p));
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

// Moments and state of the lane's node(s) from the pulled values d.  With
// one node per lane the pressure columns take their populations from the
// neighbouring lane first (non-equilibrium extrapolation, as
// column_from_neighbour).
template <bool DYN>
__device__ __forceinline__ NodeStateT<float2> lane_state(float2 d[9], const LaneMed<float2> &m,
                                                         const StepArgs &a, int) {
  return node_state_t<float2, DYN>(d, m.eps, m.inv_k, a, m.kn0);
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

// The walk of one warp: rows [s0, s1) of level t + 2 over the lane's
// column(s) x (the pair x, x + 1 for V = float2; x even).  Fluid rows are
// [a.y0, y_end); with walls those are 1 .. ny - 2.  out: this lane stores.
// MOM: the moments of levels t and t + 1 go to mom1 and mom2.
template <class S, bool SR, bool DYN, bool MOM, class V>
__device__ __forceinline__ void fused_walk(const StepArgs &a, const typename S::T *__restrict__ fin,
                                           typename S::T *__restrict__ fout,
                                           const float2 *__restrict__ med, int x, bool out, int s0,
                                           int s1, int y_end, uint32_t ts1, uint32_t ts2,
                                           float *__restrict__ mom1, float *__restrict__ mom2) {
  using L = LaneRaw<S, V>;
  using R = typename L::R;
  using T = typename S::T;
  const long long P = a.plane;
  auto wrap = [&](int y) { return y < 0 ? y + a.ny : (y >= a.ny ? y - a.ny : y); };
  R raw[9];
  LaneMed<V> m;
  // Sources of row r.  At a plate the directions that would come from it
  // are the node's own opposite ones, unshifted: planes 4, 7, 8 in the
  // place of 2, 5, 6 (two planes up), or the reverse.
  auto load_row = [&](int r) {
    const int y = wrap(r);
    const T *c = fin + (long long)y * a.pitch + x;
    const T *u = (a.walls && y == a.y0) ? c + 2 * P : fin + (long long)wrap(r - 1) * a.pitch + x;
    const T *d = (a.walls && y == y_end - 1) ? c - 2 * P
                                             : fin + (long long)wrap(r + 1) * a.pitch + x;
    raw[0] = L::load(c);
    raw[1] = L::load(c + P);
    raw[3] = L::load(c + 3 * P);
    raw[2] = L::load(u + 2 * P);
    raw[5] = L::load(u + 5 * P);
    raw[6] = L::load(u + 6 * P);
    raw[4] = L::load(d + 4 * P);
    raw[7] = L::load(d + 7 * P);
    raw[8] = L::load(d + 8 * P);
    load_med<DYN>(a, med, (long long)y * a.pitch + x, m);
  };
  // first level: rows s0 - 1 .. s1, without the plates
  const int r0 = a.walls && s0 == a.y0 ? s0 : s0 - 1;
  const int r_last = a.walls && s1 == y_end ? s1 - 1 : s1;
  load_row(r0);
  R h0 = R(), h1 = R(), h3 = R();   // e_y = 0 of row r - 1, shifted
  R b2 = R(), b5 = R(), b6 = R();   // e_y = +1 of row r - 2, shifted
  R c2 = R(), c5 = R(), c6 = R();   // e_y = +1 of row r - 1, shifted
  LaneMed<V> m1 = m;                // medium of row r - 1
#pragma unroll 1
  for (int r = r0; r <= s1; ++r) {
    R p[9];
    R f4, f7, f8;                   // e_y = -1 of row r, shifted
    LaneMed<V> m0 = m;
    if (r <= r_last) {
      const int y = wrap(r);
      V d[9];
      d[0] = L::value(raw[0]);
      d[2] = L::value(raw[2]);
      d[4] = L::value(raw[4]);
      d[1] = L::value(L::from_left(raw[1]));
      d[3] = L::value(L::from_right(raw[3]));
      R t5 = L::from_left(raw[5]), t6 = L::from_right(raw[6]);
      R t7 = L::from_right(raw[7]), t8 = L::from_left(raw[8]);
      if (a.walls) {
        if (y == a.y0) {
          t5 = raw[5];
          t6 = raw[6];
        }
        if (y == y_end - 1) {
          t7 = raw[7];
          t8 = raw[8];
        }
      }
      d[5] = L::value(t5);
      d[6] = L::value(t6);
      d[7] = L::value(t7);
      d[8] = L::value(t8);
      if (r < r_last) load_row(r + 1);
      const NodeStateT<V> s = lane_state<DYN>(d, m0, a, x);
      const long long o = (long long)y * a.pitch + x;
      if (MOM && out && r >= s0 && r < s1) store_moments(mom1 + o, P, s);
      lane_collide<S, SR>(d, s, a, o, ts1, p);
      f4 = p[4];
      f7 = L::from_right(p[7]);
      f8 = L::from_left(p[8]);
    } else {
      // row r is a plate: row r - 1 gets its own e_y = +1 values back
      f4 = c2;
      f7 = L::from_right(c5);  // undoes the shift of c5 (from the left)
      f8 = L::from_left(c6);
    }
    if (r > s0) {
      // second level at row r - 1 (inside the segment: no wrap)
      V d[9];
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
      if (out) {
        if (MOM) store_moments(mom2 + o, P, s);
        T *g = fout + o;
#pragma unroll
        for (int i = 0; i < 9; ++i) L::store(g + i * P, q[i]);
      }
    }
    if (r <= r_last) {
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
    *reinterpret_cast<float4 *>(p) = make_float4(v[0].x, v[0].y, v[1].x, v[1].y);
  else
    *reinterpret_cast<float2 *>(p) = v[0];
}
template <int Q>
__device__ __forceinline__ void store_row(__half *p, const uint32_t v[Q]) {
  if constexpr (Q == 2)
    *reinterpret_cast<uint2 *>(p) = make_uint2(v[0], v[1]);
  else
    *reinterpret_cast<uint32_t *>(p) = v[0];
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
                                          long long o, uint32_t ts, bool mom_out,
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
    if (MOM && mom_out) store_moments(mom + o + 2 * q, a.plane, s[q]);
    typename L::R p[9];
    lane_collide<S, SR, float2>(d[q], s[q], a, o + 2 * q, ts, p);
#pragma unroll
    for (int i = 0; i < 9; ++i) t[i][q] = p[i];
  }
}

// The walk of an interior strip (first column c0) over rows [s0, s1), as
// fused_walk, with the rows of level t copied ahead.
template <class S, bool SR, bool DYN, bool MOM, int Q>
__device__ __forceinline__ void fused_strip(const StepArgs &a, const typename S::T *__restrict__ fin,
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
                                    MOM && out && r >= s0 && r < s1, mom1);
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
      level_row<S, SR, DYN, MOM, Q>(u, m_was, a, o, ts2, MOM && out, mom2);
      if (out) {
        T *g = fout + o;
#pragma unroll
        for (int i = 0; i < 9; ++i) store_row<Q>(g + i * P, u[i]);
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

// Interior strips of a lattice nx wide: they store columns kHalo .., kOut a
// strip, the last one moved left to end inside the row (it stores some columns
// again, with the same values).
template <class C>
__host__ __device__ inline int fused_last_column(int nx) { return (nx - C::kCols) & ~3; }
template <class C>
__host__ __device__ inline int fused_interior_strips(int nx) {
  return (fused_last_column<C>(nx) + C::kOut - 1) / C::kOut + 1;
}

// One warp's task: strip `strip` (the last is the edge strip) of rows [s0, s1).
template <class S, bool SR, bool DYN, bool MOM, int Q>
__device__ __forceinline__ void fused_task(const StepArgs &a, const typename S::T *__restrict__ fin,
                                           typename S::T *__restrict__ fout,
                                           const float2 *__restrict__ med, int strip, int s0,
                                           int s1, int y_end, uint32_t ts1, uint32_t ts2,
                                           float *__restrict__ mom1, float *__restrict__ mom2,
                                           unsigned char *ring) {
  using C = FusedCfg<S, Q, DYN>;
  const int lane = threadIdx.x & 31;
  const int last = fused_last_column<C>(a.nx);
  if (strip < fused_interior_strips<C>(a.nx)) {
    const int c0 = strip * C::kOut < last ? strip * C::kOut : last;
    fused_strip<S, SR, DYN, MOM, Q>(a, fin, fout, med, c0, s0, s1, y_end, ts1, ts2, mom1, mom2,
                                    ring);
  } else {
    // at most kHalo columns on the left and kHalo + 3 on the right
    const int x = lane < 16 ? a.nx - 16 + lane : lane - 16;
    const bool out = x < C::kHalo || x >= last + C::kCols - C::kHalo;
    fused_walk<S, SR, DYN, MOM, float>(a, fin, fout, med, x, out, s0, s1, y_end, ts1, ts2, mom1,
                                       mom2);
  }
}

// Time levels t, t + 1 of the stochastic rounding (t = *tctr + k).
__device__ __forceinline__ uint32_t level_hash(const StepArgs &a, unsigned long long t) {
  return mix32((uint32_t)t * 0x9e3779b9u ^ a.seed_lo ^ mix32((uint32_t)(t >> 32) ^ a.seed_hi));
}

// Task w of the launch: strip w % strips of segment w / strips, the
// segments being `seg` rows high (the last one shorter).  FORCH = a0.forch, as
// a constant: no branch inside a row.
template <class S, bool SR, bool DYN, bool MOM, bool FORCH, int Q>
__global__ void __launch_bounds__(kFusedWarps * 32, FusedCfg<S, Q, DYN>::kBlocks)
    fused_step_kernel(const StepArgs a0, const typename S::T *__restrict__ fin,
                      typename S::T *__restrict__ fout, const float2 *__restrict__ med,
                      const unsigned long long *__restrict__ tctr, int k, int rows, int seg,
                      int strips, int tasks, float *__restrict__ mom1, float *__restrict__ mom2) {
  extern __shared__ __align__(128) unsigned char smem[];
  StepArgs a = a0;
  a.forch = FORCH;
  const int warp = threadIdx.x >> 5;
  const int w = blockIdx.x * kFusedWarps + warp;
  if (w >= tasks) return;
  const int strip = w % strips, part = w / strips;
  const int y_end = a.y0 + rows;
  const int s0 = a.y0 + part * seg;
  const int s1 = s0 + seg < y_end ? s0 + seg : y_end;
  uint32_t ts1 = 0, ts2 = 0;
  if (SR) {
    const unsigned long long t = *tctr + (unsigned long long)k;
    ts1 = level_hash(a, t);
    ts2 = level_hash(a, t + 1);
  }
  fused_task<S, SR, DYN, MOM, Q>(a, fin, fout, med, strip, s0, s1, y_end, ts1, ts2, mom1, mom2,
                                 smem + warp * FusedCfg<S, Q, DYN>::kWarpBytes);
}

}  // namespace lbmp
