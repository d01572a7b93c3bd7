// Discrete adjoint of the time loop (Section III, Eq. 12-17) for the global
// permeability k_g = nu <u_x> / G_eff of the final time level (Darcy's law
// over the domain, Section IV.A): gradients with respect to ln k_a and eps
// of every node.
//
// Forward: B_{t+1} = C(E(P(B_t))), B the post-collision buffer (B_0 = rest),
// P the pull (streaming with plates and periodic edges), E the pressure
// column extrapolation (non-equilibrium, from the adjacent interior node),
// C the collision of every fluid node; J depends on f^N = E(P(B_N)).
// Reverse: mu^N = dJ/df^N, then for t = N-1 .. 0
//   lambda*(z) = mu^{t+1}(z + e_i) for each direction (P transposed: a
//                plate returns it to the opposite direction of the same
//                node, a pressure column or the outside returns nothing),
//   mu^t       = C_t^T lambda* at the state f^t, with E^T folded in: a
//                column's adjoint is pushed into its interior neighbour by
//                the thread of that neighbour, which also forms it.
// C_t^T: post_i = (1 - 1/tau) f_i + g_i(rho, m; eps, k_a) with g_i = f_eq_i /
// tau + F_i (Eq. 14, 15), so mu_j = (1 - 1/tau) lambda*_j + dG/drho +
// e_j . dG/dm, G = sum_i lambda*_i g_i.  G is written through the weighted
// moments L0 = sum w lambda, L1 = sum w lambda e, L2 = sum w lambda e e of
// lambda* and differentiated by hand, back through the velocity solve of
// Eq. 16b-17 (with the Forchheimer drag of Eq. 2, the quadratic form).
// States f^t are recomputed segment by segment from checkpoints taken every
// `every` steps (sqrt(N) by default).  Each reverse step adds its parameter
// derivatives to FP32 accumulators, folded into the FP64 gradients every
// kFold steps (a schedule independent of `every`).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdarg>
#include <cstdio>

#include "chain.cuh"
#include "context.h"
#include "device_scope.h"
#include "kernels.h"
#include "lattice.cuh"
#include "lbmp.h"

namespace lbmp {

struct AdjArgs {
  StepArgs a;            // forward parameters (FP32 storage, scale 1)
  const float *lam_in;   // mu^{t+1}, [9][ny][pitch] (pressure columns unused)
  float *lam_out;        // mu^t
  const float *fin;      // forward buffer whose pull gives f^t (seed step)
  const float *mom;      // moments of f^t (rho - rho0, m_x, m_y planes; reverse steps)
  const float2 *med;     // (eps, 1/k_a)
  float2 *acc;           // [ny][pitch] (dJ/d eps, dJ/d ln k_a) of the last few steps, FP32
  double *g_eps;         // [ny][pitch] dJ/d eps, FP64 (acc folded in every kFold steps)
  double *g_lk;          // [ny][pitch] dJ/d ln k_a, FP64
  float coef;            // dJ/du_x of one node: nu / (G_eff * fluid nodes)
};

constexpr int kAdjBX = 128;
constexpr int kAdjBlocks = 5;   // blocks of the reverse step on an SM
constexpr int kAdjRows = 16;    // and the most rows that one of its warps takes
constexpr int kFold = 32;  // reverse steps summed in FP32 before the FP64 fold

// The arithmetic of the reverse step rounds where it says so (fmaf, mul; a plain
// sum is one addition), so that a kernel's form does not move its results: left to the
// compiler, products contract one way here and another there.
__device__ __forceinline__ float mul(float a, float b) { return __fmul_rn(a, b); }
// a b + c d, a b - c d: the second product rounded first.
__device__ __forceinline__ float sum2(float a, float b, float c, float d) {
  return fmaf(a, b, mul(c, d));
}
__device__ __forceinline__ float dif2(float a, float b, float c, float d) {
  return fmaf(a, b, -mul(c, d));
}

// Weighted moments of an adjoint population vector.  A node's own, a pressure
// column's and the seed's differ in the order of a few roundings.
struct LamMom {
  float L0, Lx, Ly, Lxx, Lxy, Lyy;
};
template <bool SEED>
__device__ __forceinline__ LamMom lam_moments(const float l[9], bool column) {
  const float s1 = l[1] + l[3], s2 = l[2] + l[4];
  const float a57 = l[5] + l[7], a68 = l[6] + l[8];
  const float d57 = l[5] - l[7], d86 = l[8] - l[6];
  const float diag = a57 + a68, ex = l[1] - l[3], ey = l[2] - l[4];
  LamMom M;
  const float axes = sum2(kW1, s1 + s2, kW0, l[0]);
  M.L0 = column ? fmaf(kW2, diag, axes) : __fadd_rn(axes, mul(kW2, diag));
  if (SEED) {
    M.Lx = sum2(kW1, ex, kW2, d57 + d86);
    M.Ly = sum2(kW1, ey, kW2, d57 - d86);
  } else {
    M.Lx = sum2(kW2, d57 + d86, kW1, ex);
    M.Ly = sum2(kW2, d57 - d86, kW1, ey);
  }
  M.Lxx = sum2(kW1, s1, kW2, diag);
  M.Lyy = sum2(kW1, s2, kW2, diag);
  M.Lxy = mul(kW2, a57 - a68);
  return M;
}

// Velocity solve of a node with eps > 0, kept for its adjoint:
// v = m / rho + eps G / 2, u = v / den, F = eps G - drag u, with
// den = c0 + s, s = sqrt(c0^2 + c1 |v|), drag = eps nu / k_a + 2 c1 |v| / den
// (Forchheimer), or den = 2 c0, drag = eps nu / k_a (Darcy only);
// c0 = 1/2 + eps nu / (4 k_a), c1 = (eps F_eps / 2) / sqrt(k_a).
struct Vel {
  float vx, vy, vmag, c0, c1, s, den, id, drag, ux, uy, Fx, Fy;  // id = 1 / den
};
__device__ __forceinline__ Vel vel_forward(float rho, float mx, float my, float eps, float kap,
                                           const StepArgs &a) {
  Vel V;
  const float ir = rcp_approx(rho);
  V.vx = fmaf(mx, ir, 0.5f * eps * a.Gx);
  V.vy = fmaf(my, ir, 0.5f * eps * a.Gy);
  const float darcy = a.nu * eps * kap;
  V.c0 = fmaf(0.25f, darcy, 0.5f);
  if (a.forch) {
    V.c1 = a.fe_half * sqrt_approx(kap * rcp_approx(eps));
    V.vmag = sqrt_approx(fmaf(V.vx, V.vx, V.vy * V.vy));
    V.s = sqrt_approx(fmaf(V.c0, V.c0, V.c1 * V.vmag));
    V.den = V.c0 + V.s;
    V.id = rcp_approx(V.den);
    V.drag = fmaf(2.0f * V.c1, V.vmag * V.id, darcy);
  } else {
    V.c1 = 0.0f;
    V.vmag = 0.0f;
    V.s = 0.0f;
    V.den = 2.0f * V.c0;
    V.id = rcp_approx(V.den);
    V.drag = darcy;
  }
  V.ux = V.vx * V.id;
  V.uy = V.vy * V.id;
  V.Fx = dif2(eps, a.Gx, V.drag, V.ux);
  V.Fy = dif2(eps, a.Gy, V.drag, V.uy);
  return V;
}

// Sensitivities of a node: d/drho and d/dm of its post-stream moments, and
// the parameter derivatives d/d eps and d/d ln k_a.
struct Bar {
  float rho, mx, my, eps, lk;
};

// Reverse of vel_forward: adds to b the derivatives of ub . u + Fb . F, ub
// already without the part that F = eps G - drag u takes (- drag Fb).  FORCE: Fb is
// not zero.
template <bool SEED, bool FORCE>
__device__ __forceinline__ void vel_adjoint(const Vel &V, float rho, float mx, float my,
                                            float eps, float kap, float ubx, float uby, float Fbx,
                                            float Fby, const StepArgs &a, Bar &b) {
  const float dragb = FORCE ? -sum2(Fbx, V.ux, Fby, V.uy) : 0.0f;
  if (FORCE) b.eps += sum2(Fbx, a.Gx, Fby, a.Gy);
  // u = v / den
  const float id = V.id;
  float vbx = mul(ubx, id), vby = mul(uby, id);
  float denb = mul(-sum2(ubx, V.ux, uby, V.uy), id);
  const float darcy = mul(mul(a.nu, eps), kap);
  float c0b;
  if (a.forch) {
    // drag = darcy + 2 c1 |v| / den
    const float dragb_v = mul(2.0f * dragb, V.vmag), dragb_c = mul(2.0f * dragb, V.c1);
    denb = fmaf(-mul(mul(dragb_c, V.vmag), id), id, denb);
    // den = c0 + s, s = sqrt(c0^2 + c1 |v|) >= c0 >= 1/2
    const float is = rcp_approx(V.s);
    c0b = mul(denb, fmaf(V.c0, is, 1.0f));
    const float c1b = sum2(dragb_v, id, mul(0.5f * denb, V.vmag), is);
    const float vmagb = sum2(dragb_c, id, mul(0.5f * denb, V.c1), is);
    // |v|: at v = 0 the terms it enters vanish with u, so its derivative is
    // not needed there
    if (V.vmag > 0.0f) {
      const float iv = rcp_approx(V.vmag);
      vbx = fmaf(mul(vmagb, V.vx), iv, vbx);
      vby = fmaf(mul(vmagb, V.vy), iv, vby);
    }
    // c1 = fe_half sqrt(kap / eps): dc1/d ln k_a = -c1 / 2, dc1/d eps = -c1 / (2 eps)
    const float h = 0.5f * V.c1;
    b.lk = SEED ? __fadd_rn(b.lk, -mul(h, c1b)) : fmaf(-h, c1b, b.lk);
    b.eps = fmaf(-mul(h, c1b), rcp_approx(eps), b.eps);
  } else {
    c0b = 2.0f * denb;
  }
  // darcy = nu eps kap: d/d ln k_a = -darcy, d/d eps = nu kap
  const float darcyb = fmaf(0.25f, c0b, dragb);
  b.lk = fmaf(-darcy, darcyb, b.lk);
  b.eps = fmaf(mul(a.nu, kap), darcyb, b.eps);
  // v = m / rho + eps G / 2
  const float ir = rcp_approx(rho);
  b.mx = fmaf(vbx, ir, b.mx);
  b.my = fmaf(vby, ir, b.my);
  b.rho = fmaf(-mul(sum2(vbx, mx, vby, my), ir), ir, b.rho);
  b.eps = fmaf(0.5f, sum2(vbx, a.Gx, vby, a.Gy), b.eps);
}

// Adds to b the derivatives of G = sum_i lam_i g_i(rho, m; eps, k_a) of one
// node.  sum_i lam_i f_eq_i = rho [L0 + 3 u.L1 + (9/2 u.L2.u - 3/2 u^2 L0) /
// eps] (Eq. 14) and sum_i lam_i F_i = (1 - 1/2tau) rho [3 F.L1 + (9 u.L2.F -
// 3 (u.F) L0) / eps] (Eq. 15); eps = 0 keeps f_eq = w rho, u = 0 and
// F = -2 m / rho.
__device__ __forceinline__ void collide_adjoint(const float lam[9], bool column, float rho,
                                                float mx, float my, float eps, float kap,
                                                const StepArgs &a, Bar &b) {
  const LamMom M = lam_moments<false>(lam, column);
  const float om = a.omega, cf = a.cforce;
  if (!(eps > 0.0f)) {
    b.rho += mul(om, M.L0);
    b.mx -= mul(6.0f * cf, M.Lx);
    b.my -= mul(6.0f * cf, M.Ly);
    return;
  }
  const Vel V = vel_forward(rho, mx, my, eps, kap, a);
  const float ie = rcp_approx(eps);
  const float ux = V.ux, uy = V.uy, Fx = V.Fx, Fy = V.Fy;
  const float L2ux = sum2(M.Lxx, ux, M.Lxy, uy), L2uy = sum2(M.Lxy, ux, M.Lyy, uy);
  const float L2Fx = sum2(M.Lxx, Fx, M.Lxy, Fy), L2Fy = sum2(M.Lxy, Fx, M.Lyy, Fy);
  const float qe = dif2(4.5f, sum2(ux, L2ux, uy, L2uy), mul(1.5f, sum2(ux, ux, uy, uy)), M.L0);
  const float qf = dif2(9.0f, sum2(ux, L2Fx, uy, L2Fy), mul(3.0f, sum2(ux, Fx, uy, Fy)), M.L0);
  const float Seq = fmaf(qe, ie, fmaf(3.0f, sum2(ux, M.Lx, uy, M.Ly), M.L0));
  const float SF = sum2(3.0f, sum2(Fx, M.Lx, Fy, M.Ly), qf, ie);
  b.rho += sum2(om, Seq, cf, SF);
  // dSeq/du = dSF/dF
  const float ax = sum2(3.0f, M.Lx, dif2(9.0f, L2ux, mul(3.0f, ux), M.L0), ie);
  const float ay = sum2(3.0f, M.Ly, dif2(9.0f, L2uy, mul(3.0f, uy), M.L0), ie);
  const float ubx = sum2(om, ax, mul(cf, dif2(9.0f, L2Fx, mul(3.0f, Fx), M.L0)), ie);
  const float uby = sum2(om, ay, mul(cf, dif2(9.0f, L2Fy, mul(3.0f, Fy), M.L0)), ie);
  b.eps -= mul(mul(mul(rho, sum2(om, qe, cf, qf)), ie), ie);
  const float rcf = mul(rho, cf), Fbx = mul(rcf, ax), Fby = mul(rcf, ay);
  vel_adjoint<false, true>(V, rho, mx, my, eps, kap, dif2(rho, ubx, V.drag, Fbx),
                         dif2(rho, uby, V.drag, Fby), Fbx, Fby, a, b);
}

// Pressure column b next to interior node n: f_b = f_n + f_eq(rho_b, u_n;
// eps_b) - f_eq(rho_n, u_n; eps_n).  Adds to bn the derivatives of
// sum_i lb_i f_b,i with respect to n's moments and parameters (the identity
// part, lb itself, is added by the caller) and to eb the one of eps_b.
template <bool SEED>
__device__ __forceinline__ void neep_adjoint(const float lb[9], float rho_n, float mx, float my,
                                             float eps_n, float kap_n, float eps_b, float rho_b,
                                             const StepArgs &a, Bar &bn, float &eb) {
  const LamMom M = lam_moments<SEED>(lb, true);
  if (!(eps_n > 0.0f)) {  // u_n = 0: f_b = f_n + w (rho_b - rho_n)
    bn.rho -= M.L0;
    return;
  }
  const Vel V = vel_forward(rho_n, mx, my, eps_n, kap_n, a);
  const float ux = V.ux, uy = V.uy;
  const float L2ux = sum2(M.Lxx, ux, M.Lxy, uy), L2uy = sum2(M.Lxy, ux, M.Lyy, uy);
  const float q = dif2(4.5f, sum2(ux, L2ux, uy, L2uy), mul(1.5f, sum2(ux, ux, uy, uy)), M.L0);
  const float cx = mul(3.0f, M.Lx), cy = mul(3.0f, M.Ly);
  const float qx = dif2(9.0f, L2ux, mul(3.0f, ux), M.L0);
  const float qy = dif2(9.0f, L2uy, mul(3.0f, uy), M.L0);
  // d/du of sum_i lb_i f_eq_i / rho at porosity eps: c + q / eps
  const float ien = rcp_approx(eps_n);
  const bool open = !SEED && eps_b > 0.0f;
  bn.rho -= fmaf(q, ien, __fadd_rn(M.L0, sum2(ux, cx, uy, cy)));
  const float dux = open ? sum2(3.0f, M.Lx, qx, ien) : fmaf(qx, ien, cx);
  const float duy = open ? sum2(3.0f, M.Ly, qy, ien) : fmaf(qy, ien, cy);
  float ubx = mul(-rho_n, dux), uby = mul(-rho_n, duy);
  bn.eps = fmaf(mul(mul(rho_n, q), ien), ien, bn.eps);
  if (eps_b > 0.0f) {
    const float ieb = rcp_approx(eps_b);
    ubx = sum2(-rho_n, dux, rho_b,
               open ? sum2(3.0f, M.Lx, qx, ieb) : fmaf(qx, ieb, cx));
    uby = sum2(-rho_n, duy, rho_b,
               open ? sum2(3.0f, M.Ly, qy, ieb) : fmaf(qy, ieb, cy));
    eb -= mul(mul(mul(rho_b, q), ieb), ieb);
  }
  vel_adjoint<SEED, false>(V, rho_n, mx, my, eps_n, kap_n, ubx, uby, 0.0f, 0.0f, a, bn);
}

__device__ __forceinline__ float lam_at(const AdjArgs &A, int i, int x, int y) {
  return A.lam_in[i * A.a.plane + (long long)y * A.a.pitch + x];
}

// Reverse streaming for node (x, y): the adjoint of its post-collision
// values, read where each of them streams to.
__device__ __forceinline__ void reverse_pull(const AdjArgs &A, int x, int y, float lp[9]) {
  const StepArgs &a = A.a;
  const int ex[9] = {0, 1, 0, -1, 0, 1, -1, -1, 1};
  const int ey[9] = {0, 0, 1, 0, -1, 1, 1, -1, -1};
  const int opp[9] = {0, 3, 4, 1, 2, 7, 8, 5, 6};
  // the pulls of a pressure column are discarded (replaced by the
  // extrapolation), so whatever streams into one carries no adjoint
  const bool col = a.pressure && (x == 0 || x == a.nx - 1);
#pragma unroll
  for (int i = 0; i < 9; ++i) {
    int xd = x + ex[i], yd = y + ey[i];
    if (a.walls && ey[i] != 0 && (yd == 0 || yd == a.ny - 1)) {
      lp[i] = col ? 0.0f : lam_at(A, opp[i], x, y);  // bounced back into the same node
      continue;
    }
    yd = (yd < 0) ? yd + a.ny : (yd >= a.ny ? yd - a.ny : yd);
    if (a.pressure) {
      if (xd <= 0 || xd >= a.nx - 1) {  // lost at the edge or received by a pressure column
        lp[i] = 0.0f;
        continue;
      }
    } else {
      xd = (xd < 0) ? xd + a.nx : (xd >= a.nx ? xd - a.nx : xd);
    }
    lp[i] = lam_at(A, i, xd, yd);
  }
}

__device__ __forceinline__ void moments(const float d[9], float rho0, float &rho, float &mx,
                                        float &my) {
  const float drho = ((d[0] + (d[1] + d[3])) + (d[2] + d[4])) + ((d[5] + d[7]) + (d[6] + d[8]));
  rho = rho0 + drho;
  mx = (d[1] - d[3]) + ((d[5] - d[7]) + (d[8] - d[6]));
  my = (d[2] - d[4]) + ((d[5] - d[7]) + (d[6] - d[8]));
}

// The objective's adjoint of the pressure column beside interior node (x, y),
// formed and pushed into the node by the node's own thread (E^T): adds it to mu and
// the node's moment and parameter sensitivities to bn; writes the column's
// parameter gradients.
__device__ __forceinline__ void column_seed(const AdjArgs &A, int x, int y, float rho, float mx,
                                            float my, float2 mn, float mu[9], Bar &bn) {
  const StepArgs &a = A.a;
  const int ex[9] = {0, 1, 0, -1, 0, 1, -1, -1, 1};
  const int ey[9] = {0, 0, 1, 0, -1, 1, 1, -1, -1};
#pragma unroll 1
  for (int side = 0; side < 2; ++side) {
    const int xn = side ? a.nx - 2 : 1;
    if (x != xn) continue;
    const int xb = side ? a.nx - 1 : 0;
    const long long jb = (long long)y * a.pitch + xb;
    const float2 mb = A.med[jb];
    float rb, mbx, mby, fb[9];
    pressure_node<StoreF32>(A.fin, A.med, a, xb, y, mb.x, fb);
    moments(fb, a.rho0, rb, mbx, mby);
    Bar bb = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
    if (mb.x > 0.0f) {
      const Vel V = vel_forward(rb, mbx, mby, mb.x, mb.y, a);
      vel_adjoint<true, false>(V, rb, mbx, mby, mb.x, mb.y, A.coef, 0.0f, 0.0f, 0.0f, a, bb);
    }
    float lb[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) lb[i] = bb.rho + ex[i] * bb.mx + ey[i] * bb.my;
    float eb = 0.0f;
    const float rho_b = a.rho0 + (side ? a.drho_out : a.drho_in);
    neep_adjoint<true>(lb, rho, mx, my, mn.x, mn.y, mb.x, rho_b, a, bn, eb);
#pragma unroll
    for (int i = 0; i < 9; ++i) mu[i] += lb[i];
    const float2 g = A.acc[jb];  // only this thread touches the column node
    A.acc[jb] = make_float2(g.x + (bb.eps + eb), g.y + bb.lk);
  }
}

// The objective's seed, mu^N = dJ/df^N.  Pressure-column threads return at
// once (their neighbours handle them).
__global__ void __launch_bounds__(kAdjBX, 8) adjoint_seed_kernel(const AdjArgs A) {
  const StepArgs &a = A.a;
  const int y = a.y0 + blockIdx.y;
  const int x = blockIdx.x * kAdjBX + threadIdx.x;
  if (x >= a.nx) return;
  if (a.pressure && (x == 0 || x == a.nx - 1)) return;
  const int ex[9] = {0, 1, 0, -1, 0, 1, -1, -1, 1};
  const int ey[9] = {0, 0, 1, 0, -1, 1, 1, -1, -1};
  const long long j = (long long)y * a.pitch + x;
  const float2 g0 = A.acc[j];
  const float2 m = __ldg(A.med + j);
  float mu[9], d[9];
  float rho, mx, my;
  pull_node<StoreF32>(A.fin, a, x, y, d);
  moments(d, a.rho0, rho, mx, my);
  Bar b = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
  if (m.x > 0.0f) {
    const Vel V = vel_forward(rho, mx, my, m.x, m.y, a);
    vel_adjoint<true, false>(V, rho, mx, my, m.x, m.y, A.coef, 0.0f, 0.0f, 0.0f, a, b);
  }
#pragma unroll
  for (int i = 0; i < 9; ++i) mu[i] = 0.0f;
  if (a.pressure && (x == 1 || x == a.nx - 2)) column_seed(A, x, y, rho, mx, my, m, mu, b);
#pragma unroll
  for (int i = 0; i < 9; ++i)
    A.lam_out[i * a.plane + j] = mu[i] + b.rho + ex[i] * b.mx + ey[i] * b.my;
  A.acc[j] = make_float2(g0.x + b.eps, g0.y + b.lk);
}

// What a reverse step reads of one node.
struct RevIn {
  float l[9], r, mx, my;
  float2 med, acc;
};
__device__ __forceinline__ void rev_fields(const AdjArgs &A, long long j, RevIn &n) {
  n.med = __ldg(A.med + j);
  n.acc = A.acc[j];
  n.r = A.mom[j];
  n.mx = A.mom[A.a.plane + j];
  n.my = A.mom[2 * A.a.plane + j];
}
__device__ __forceinline__ void rev_store(const AdjArgs &A, long long j, const float mu[9],
                                          const Bar &b, float2 acc) {
  const int ex[9] = {0, 1, 0, -1, 0, 1, -1, -1, 1};
  const int ey[9] = {0, 0, 1, 0, -1, 1, 1, -1, -1};
#pragma unroll
  for (int i = 0; i < 9; ++i) {
    float s = __fadd_rn(mu[i], b.rho);
    if (ex[i]) s = __fadd_rn(s, ex[i] > 0 ? b.mx : -b.mx);
    if (ey[i]) s = __fadd_rn(s, ey[i] > 0 ? b.my : -b.my);
    A.lam_out[i * A.a.plane + j] = s;
  }
  A.acc[j] = make_float2(acc.x + b.eps, acc.y + b.lk);
}

// The nodes next to the pressure columns and, through them, the columns: four
// lanes a node, one for the node itself and one for each column beside it, so
// that their collision adjoints run at the same time (64 x 64, 400 steps: 4.6 ms
// with one lane that takes them in turn, 3.6 with one each).  The column's
// adjoint, (1 - 1/tau) lambda*_b + its collision adjoint, then goes to the node's
// lane (E^T).  A lane's loads are a row apart: few nodes a warp spread them.
__device__ __forceinline__ void edge_nodes(const AdjArgs &A, int t, int rows) {
  const StepArgs &a = A.a;
  const int role = t & 3, node = t >> 2, side = node >= rows;
  const int xn = side ? a.nx - 2 : 1;
  const int x = role == 0 ? xn : role == 1 ? 0 : a.nx - 1;
  const bool live = node < (a.nx == 3 ? rows : 2 * rows) &&
                    (role == 0 || (role == 1 && xn == 1) || (role == 2 && xn == a.nx - 2));
  const int y = a.y0 + (live ? node - side * rows : 0);
  const long long j = (long long)y * a.pitch + x;
  RevIn n = {};
  Bar b = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
  float v[9] = {};
  float rho = 1.0f;
  if (live) {
    rev_fields(A, j, n);
    reverse_pull(A, x, y, n.l);
    rho = a.rho0 + n.r;
    collide_adjoint(n.l, role != 0, rho, n.mx, n.my, n.med.x, n.med.y, a, b);
    if (role == 0) {
#pragma unroll
      for (int i = 0; i < 9; ++i) v[i] = mul(a.one_m_omega, n.l[i]);
    } else {
      const int ex[9] = {0, 1, 0, -1, 0, 1, -1, -1, 1};
      const int ey[9] = {0, 0, 1, 0, -1, 1, 1, -1, -1};
#pragma unroll
      for (int i = 0; i < 9; ++i)
        v[i] = fmaf(a.one_m_omega, n.l[i], b.rho + ex[i] * b.mx + ey[i] * b.my);
    }
  }
#pragma unroll 1
  for (int k = 1; k <= 2; ++k) {
    float lb[9], eb = 0.0f;
#pragma unroll
    for (int i = 0; i < 9; ++i) lb[i] = __shfl_sync(0xffffffffu, v[i], k, 4);
    const float eps_b = __shfl_sync(0xffffffffu, n.med.x, k, 4);
    if (live && role == 0 && xn == (k == 1 ? 1 : a.nx - 2)) {
      const float rho_b = a.rho0 + (k == 1 ? a.drho_in : a.drho_out);
      neep_adjoint<false>(lb, rho, n.mx, n.my, n.med.x, n.med.y, eps_b, rho_b, a, b, eb);
#pragma unroll
      for (int i = 0; i < 9; ++i) v[i] += lb[i];
    }
    eb = __shfl_sync(0xffffffffu, eb, 0, 4);
    if (role == k) b.eps += eb;
  }
  if (!live) return;
  if (role == 0)
    rev_store(A, j, v, b, n.acc);
  else
    A.acc[j] = make_float2(n.acc.x + b.eps, n.acc.y + b.lk);
}

// One reverse step over the fluid rows: mu^t from mu^{t+1} and f^t.  The first
// `edges` blocks take the nodes next to pressure columns (and through them the
// columns); each further warp takes 32 columns of `seg` rows, upwards in y.
//
// 108 B a node (mu in and out, moments, medium, accumulators) against some 400
// instructions.  With a thread per node it waited for its loads at 54 % of the issue
// slots, and the warps at a pressure column computed three nodes in turn: 26 us
// at 1024^2.  Walking the rows with the next row's 16 values in flight while
// one is computed: 18 us, 6.3 TB/s.  Five blocks of 85 registers an SM (four: +1.9 us,
// six: the same).
__global__ void __launch_bounds__(kAdjBX, kAdjBlocks)
    adjoint_step_kernel(const AdjArgs A, int rows, int edges, int strips, int seg) {
  chain_wait();
  const StepArgs &a = A.a;
  if ((int)blockIdx.x < edges) {
    edge_nodes(A, blockIdx.x * kAdjBX + threadIdx.x, rows);
    return;
  }
  const int task = (blockIdx.x - edges) * (kAdjBX / 32) + threadIdx.x / 32;
  const int part = task / strips;
  const int x = (task - part * strips) * 32 + (threadIdx.x & 31);
  int y = a.y0 + part * seg;
  const int end = min(y + seg, a.y0 + rows);
  if (y >= end || x >= a.nx) return;
  if (a.pressure && (x < 2 || x > a.nx - 3)) return;
  const int west = x > 0 ? -1 : a.nx - 1, east = x < a.nx - 1 ? 1 : 1 - a.nx;
  auto load = [&](int y, RevIn &n) {
    const long long j = (long long)y * a.pitch + x;
    rev_fields(A, j, n);
    if (a.walls && (y == 1 || y == a.ny - 2)) {
      reverse_pull(A, x, y, n.l);
      return;
    }
    const int up = (y < a.ny - 1 ? 1 : 1 - a.ny) * a.pitch, down = (y > 0 ? -1 : a.ny - 1) * a.pitch;
    const float *l = A.lam_in + j;
    const long long P = a.plane;
    n.l[0] = l[0];
    n.l[1] = l[P + east];
    n.l[2] = l[2 * P + up];
    n.l[3] = l[3 * P + west];
    n.l[4] = l[4 * P + down];
    n.l[5] = l[5 * P + up + east];
    n.l[6] = l[6 * P + up + west];
    n.l[7] = l[7 * P + down + west];
    n.l[8] = l[8 * P + down + east];
  };
  RevIn n;
  load(y, n);
  for (; y < end; ++y) {
    RevIn next = n;
    if (y + 1 < end) load(y + 1, next);
    const float rho = a.rho0 + n.r;
    Bar b = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
    collide_adjoint(n.l, false, rho, n.mx, n.my, n.med.x, n.med.y, a, b);
    float mu[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) mu[i] = mul(a.one_m_omega, n.l[i]);
    rev_store(A, (long long)y * a.pitch + x, mu, b, n.acc);
    n = next;
  }
}

// Rows a warp: what fills the chip once beside the edge blocks, at most 16 (8: +1.6 us
// a step at 1024^2, 32: the same).
static cudaError_t launch_adjoint_step(const AdjArgs &A, int rows, int nsm, cudaStream_t s) {
  constexpr int kWarps = kAdjBX / 32;
  const int edges = A.a.pressure ? (8 * rows + kAdjBX - 1) / kAdjBX : 0;  // edge_nodes()
  const int strips = (A.a.nx + 31) / 32;
  const int slots = std::max(nsm * kAdjBlocks - edges, nsm) * kWarps;
  const int parts = std::max(1, slots / strips);
  const int seg = std::min((rows + parts - 1) / parts, kAdjRows);
  const int tasks = strips * ((rows + seg - 1) / seg);
  return launch_chained(adjoint_step_kernel, dim3(edges + (tasks + kWarps - 1) / kWarps),
                        dim3(kAdjBX), 0, s, A, rows, edges, strips, seg);
}

// Folds the FP32 accumulators of the fluid rows into the FP64 gradients
// and clears them.
__global__ void __launch_bounds__(kAdjBX) adjoint_fold_kernel(const AdjArgs A) {
  const StepArgs &a = A.a;
  const int y = a.y0 + blockIdx.y;
  const int x = blockIdx.x * kAdjBX + threadIdx.x;
  chain_wait();
  if (x >= a.nx) return;
  const long long j = (long long)y * a.pitch + x;
  const float2 g = A.acc[j];
  A.g_eps[j] += (double)g.x;
  A.g_lk[j] += (double)g.y;
  A.acc[j] = make_float2(0.0f, 0.0f);
}

// dJ/d ln k_a and dJ/d eps (+ the mean-porosity term of the pressure drop)
// into [ny][nx] float64; plate rows read 0.
__global__ void adjoint_assemble_kernel(const AdjArgs A, double eps_term, double *out_logk,
                                        double *out_eps) {
  const StepArgs &a = A.a;
  const int y = blockIdx.y;
  const int x = blockIdx.x * kAdjBX + threadIdx.x;
  if (x >= a.nx) return;
  const long long o = (long long)y * a.nx + x;
  if (a.walls && (y == 0 || y == a.ny - 1)) {
    out_logk[o] = 0.0;
    out_eps[o] = 0.0;
    return;
  }
  const long long j = (long long)y * a.pitch + x;
  out_logk[o] = A.g_lk[j];
  out_eps[o] = A.g_eps[j] + eps_term;
}

}  // namespace lbmp

// ------------------------------------------------------------------ driver
namespace {

lbmp_status afail(lbmp_status st, const char *fmt, ...) {
  char buf[512];
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(buf, sizeof(buf), fmt, ap);
  va_end(ap);
  lbmp::set_last_error(buf);  // read back with lbmp_last_error()
  return st;
}

struct DevBuf {
  void *p = nullptr;
  ~DevBuf() {
    if (p) cudaFree(p);
  }
};

#define ACK(call)                                                                        \
  do {                                                                                   \
    cudaError_t e_ = (call);                                                             \
    if (e_ != cudaSuccess) {                                                             \
      cudaGetLastError();                                                                \
      return afail(e_ == cudaErrorMemoryAllocation ? LBMP_ENOMEM : LBMP_ECUDA, "%s: %s", \
                   #call, cudaGetErrorString(e_));                                       \
    }                                                                                    \
  } while (0)

// The launches of one backward segment: n recompute steps from checkpoint ck
// (the first step reads it in place, the two state buffers at segp then
// alternate; level t's moments go to mom + t * mom_level; two steps per launch
// by the plan `pairs` unless that is null), then the n reverse steps from
// the last level down, with an FP64 fold after every kFold-th reverse step of the
// whole sweep (`reversed` of them done before this segment).  lam[0] holds
// Lambda^{t+1} of the segment's last level on entry.  Adds its launches to
// *launches.
cudaError_t enqueue_segment(const lbmp::AdjArgs &A0, int rows, const float2 *med, const char *ck,
                            char *segp, size_t state, char *momp, size_t mom_level, int64_t n,
                            float *const lam[2], int64_t reversed, const lbmp::FusedPlan *pairs,
                            int nsm, int64_t *launches, cudaStream_t s) {
  lbmp::AdjArgs A = A0;
  const lbmp::StepArgs &a = A.a;
  cudaError_t e = cudaSuccess;
  const float *in = (const float *)ck;
  int to = 0;
  for (int64_t t = 0; t < n && e == cudaSuccess;) {
    float *out = (float *)(segp + state * to);
    float *m0 = (float *)(momp + mom_level * t), *m1 = (float *)(momp + mom_level * (t + 1));
    if (pairs && t + 1 < n) {
      e = lbmp::launch_fused_moments(a, rows, in, out, med, m0, m1, *pairs, s);
      t += 2;
    } else {
      e = lbmp::launch_step_moments(a, rows, in, out, med, m0, s);
      t += 1;
    }
    ++*launches;
    in = out;
    to ^= 1;
  }
  const dim3 blk(lbmp::kAdjBX), grd((a.nx + lbmp::kAdjBX - 1) / lbmp::kAdjBX, rows);
  int next = 0;
  for (int64_t t = n - 1; t >= 0 && e == cudaSuccess; --t) {
    A.lam_in = lam[next];
    A.lam_out = lam[next ^ 1];
    A.fin = nullptr;
    A.mom = (const float *)(momp + mom_level * t);
    e = lbmp::launch_adjoint_step(A, rows, nsm, s);
    ++*launches;
    next ^= 1;
    if (e == cudaSuccess && ++reversed % lbmp::kFold == 0) {
      e = lbmp::launch_chained(lbmp::adjoint_fold_kernel, grd, blk, 0, s, A);
      ++*launches;
    }
  }
  return e;
}

}  // namespace

extern "C" lbmp_status lbmp_permeability_gradient(lbmp_ctx *c, int64_t nsteps, int64_t every,
                                                  double *k_g, double *d_logk, double *d_eps,
                                                  int32_t where) {
  using lbmp::AdjArgs;
  using lbmp::StepArgs;
  try {
    if (!c || !d_logk || !d_eps)
      return afail(LBMP_EINVAL, "lbmp_permeability_gradient: NULL argument");
    if (where != LBMP_HOST && where != LBMP_DEVICE)
      return afail(LBMP_EINVAL, "where must be LBMP_HOST or LBMP_DEVICE");
    if (nsteps < 1) return afail(LBMP_EINVAL, "nsteps must be >= 1 (got %lld)", (long long)nsteps);
    if (every < 0) return afail(LBMP_EINVAL, "every must be >= 0 (0: sqrt(nsteps))");
    if (!c->fields_set) return afail(LBMP_ESTATE, "lbmp_permeability_gradient: no fields set");
    if (c->p.storage != LBMP_STORE_FP32)
      return afail(LBMP_EINVAL, "lbmp_permeability_gradient needs FP32 storage");
    if (c->p.kn_beta != 0.0)
      return afail(LBMP_EINVAL, "lbmp_permeability_gradient: a dynamic Kn is not available");
    const DeviceScope device_scope(c->device);
    ACK(device_scope.err);
    if (every == 0) every = (int64_t)std::ceil(std::sqrt((double)nsteps));
    every = std::min(every, nsteps);
    const int64_t nseg = (nsteps + every - 1) / every;
    const StepArgs a = c->args();
    const int rows = c->rows();
    const size_t state = c->buf_bytes();
    const size_t field = (size_t)c->plane * sizeof(double);
    cudaStream_t s = c->stream;
    // one allocation (one of each: 0.6 ms more at 1024^2 and 400 steps) for
    // the checkpoints (one per segment), two states for the recompute, the
    // moments of the levels of one segment, the two adjoint levels, the FP64
    // gradient fields with the accumulators
    const size_t mom_level = (size_t)c->plane * 3 * sizeof(float);
    const size_t grad_bytes = 2 * field + (size_t)c->plane * sizeof(float2);
    const size_t sizes[5] = {state * (size_t)nseg, state * 2, mom_level * (size_t)every, state * 2,
                             grad_bytes};
    size_t at[6] = {0};
    for (int k = 0; k < 5; ++k) at[k + 1] = at[k] + (sizes[k] + 511) / 512 * 512;
    DevBuf work, outs;
    ACK(cudaMalloc(&work.p, at[5]));
    char *base = (char *)work.p;
    char *ckp = base, *segp = base + at[1], *momp = base + at[2];
    ACK(cudaMemsetAsync(base + at[3], 0, at[5] - at[3], s));
    float *lam0 = (float *)(base + at[3]), *lam1 = (float *)(base + at[3] + state);
    double *g_eps = (double *)(base + at[4]), *g_lk = (double *)(base + at[4] + field);
    float2 *acc = (float2 *)(base + at[4] + 2 * field);

    // forward pass from rest in the context's own buffers (the step graphs
    // of lbmp_step), checkpointing the first level of every segment
    ACK(cudaMemsetAsync(c->buf[0], 0, state, s));
    ACK(cudaMemsetAsync(c->buf[1], 0, state, s));
    ACK(cudaMemsetAsync(c->d_err, 0, sizeof(unsigned), s));
    c->cur = 0;
    c->steps = 0;
    for (int64_t sg = 0; sg < nseg; ++sg) {
      ACK(cudaMemcpyAsync(ckp + state * sg, c->buf[c->cur], state, cudaMemcpyDeviceToDevice, s));
      lbmp_status fst = lbmp_step(c, std::min(every, nsteps - sg * every));
      if (fst) return fst;
    }
    const int cur = c->cur;
    // J = k_g of level N, exactly as lbmp_permeability reports it
    double J = 0.0;
    lbmp_status st = lbmp_permeability(c, &J, nullptr);
    if (st) return st;
    const lbmp_params &p = c->p;
    const double nu = (p.tau - 0.5) / 3.0 / p.J;
    double geff = p.Gx, kp = 0.0;
    if (p.bc_x == LBMP_BCX_PRESSURE) {
      kp = (p.rho_in - p.rho_out) / 3.0 / c->eps_mean / (p.rho0 * (double)(p.nx - 1));
      geff += kp;
    }
    const double nf = (double)c->fluid_nodes;
    AdjArgs A;
    A.a = a;
    A.med = c->med;
    A.g_eps = g_eps;
    A.g_lk = g_lk;
    A.acc = acc;
    A.coef = (float)(nu / (geff * nf));
    // seed: Lambda^N = dJ/df^N
    const dim3 blk(lbmp::kAdjBX), grd((a.nx + lbmp::kAdjBX - 1) / lbmp::kAdjBX, rows);
    A.fin = (const float *)c->buf[cur];
    A.mom = nullptr;
    A.lam_in = lam1;
    A.lam_out = lam0;
    lbmp::adjoint_seed_kernel<<<grd, blk, 0, s>>>(A);
    ACK(cudaGetLastError());
    // backward, one segment at a time: recompute its levels from the
    // checkpoint (keeping only their moments), then run the reverse steps
    // over them.  The launches go straight into the stream: a graph of a segment
    // (one per fold phase) was captured and instantiated to be replayed a few
    // times (64 x 64, 400 steps: 4.46 ms against 3.73).
    float *lams[2] = {lam0, lam1};  // lams[0]: Lambda^{t+1} of the next reverse step
    const bool pairs = lbmp::fused_covers(LBMP_STORE_FP32, false, a.nx, a.ny);
    lbmp::FusedPlan plan{};
    if (pairs) plan = lbmp::fused_plan(LBMP_STORE_FP32, false, a.nx, rows, c->nsm);
    int64_t reversed = 0;          // the FP32 accumulators fold every kFold reverse steps
    for (int64_t sg = nseg - 1; sg >= 0; --sg) {
      const int64_t t0 = sg * every, n = std::min(every, nsteps - t0);
      ACK(enqueue_segment(A, rows, c->med, ckp + state * sg, segp, state, momp, mom_level, n, lams,
                          reversed, pairs ? &plan : nullptr, c->nsm, &c->launches, s));
      reversed += n;
      if (n & 1) std::swap(lams[0], lams[1]);
    }
    lbmp::adjoint_fold_kernel<<<grd, blk, 0, s>>>(A);
    ACK(cudaGetLastError());
    // d/d eps_z of G_eff through the mean porosity (pressure drive only)
    const double eps_term = (kp != 0.0) ? J * kp / (geff * c->eps_mean * nf) : 0.0;
    const size_t nn = (size_t)a.nx * a.ny;
    double *ol = d_logk, *oe = d_eps;
    if (where == LBMP_HOST) {
      ACK(cudaMalloc(&outs.p, 2 * nn * sizeof(double)));
      ol = (double *)outs.p;
      oe = ol + nn;
    }
    const dim3 g2((a.nx + lbmp::kAdjBX - 1) / lbmp::kAdjBX, a.ny);
    lbmp::adjoint_assemble_kernel<<<g2, blk, 0, s>>>(A, eps_term, ol, oe);
    ACK(cudaGetLastError());
    c->launches += 4;
    if (where == LBMP_HOST) {
      ACK(cudaMemcpyAsync(d_logk, ol, nn * sizeof(double), cudaMemcpyDeviceToHost, s));
      ACK(cudaMemcpyAsync(d_eps, oe, nn * sizeof(double), cudaMemcpyDeviceToHost, s));
    }
    ACK(cudaStreamSynchronize(s));
    unsigned err = 0;
    ACK(cudaMemcpy(&err, c->d_err, sizeof(err), cudaMemcpyDeviceToHost));
    if (err) return afail(LBMP_ETIMEOUT, "a bounded wait of the staged step kernel gave up");
    if (k_g) *k_g = J;
    return LBMP_OK;
  } catch (...) {
    return afail(LBMP_ECUDA, "lbmp_permeability_gradient: unexpected exception");
  }
}
