// Single-phase device helpers shared by the step kernels (step_sp.cu) and the
// adjoint kernels (adjoint.cu): pull-streaming with the link-wise boundary rules,
// moments and the BGK / MRT collisions, all in deviation form.
#pragma once
#include <cuda_runtime.h>

#include "lattice.cuh"
#include "lbm_internal.cuh"
#include "reciprocal.cuh"

namespace lbmk {

enum { BC_PERIODIC = 0, BC_WALL = 1, BC_VELOCITY = 2, BC_PRESSURE = 3, BC_SYMMETRY = 4 };
enum { TBC_NONE = 0, TBC_FLUX = 1, TBC_TEMP = 2, TBC_OUTFLOW = 3, TBC_SYMMETRY = 4, TBC_WETNODE = 5 };

__device__ __forceinline__ int wrap(int a, int n) { return a < 0 ? a + n : (a >= n ? a - n : a); }

// Position of node (i, j) along a side, and the side's length.
__device__ __forceinline__ int along(int side, int i, int j) { return side < 2 ? j : i; }
__device__ __forceinline__ int side_len(const SpParams &P, int side) { return side < 2 ? P.ny : P.nx; }

// Which side the link arriving at (i, j) along c = (cx, cy) comes through (source
// node (i - cx, j - cy) outside the domain), or -1.  A link through a corner takes
// the y-side, unless that y-side is a symmetry side (ysym: bit 0 for y = 0, bit 1
// for y = ny - 1): the mirror image of the link also comes through the x-side, whose
// rule then applies.
__device__ __forceinline__ int entry_side(int i, int j, int cx, int cy, int nx, int ny, int xper, int yper,
                                          int ysym = 0) {
  const int si = i - cx, sj = j - cy;
  const int xs = xper ? -1 : (si < 0 ? 0 : (si >= nx ? 1 : -1));
  if (!yper) {
    if (sj < 0) return (ysym & 1) && xs >= 0 ? xs : 2;
    if (sj >= ny) return (ysym & 2) && xs >= 0 ? xs : 3;
  }
  return xs;
}

// Source of a link entering node (i, j) through symmetry side `side` (Eq. simetria):
// population mirror(q) of the tangential neighbour (i, j) - c_{q,tan} dt, wrapped
// where the tangential axis is periodic, else the node itself where the neighbour
// falls outside.  Returns the element offset of that value.
template <int Q>
__device__ __forceinline__ long long symmetry_source(const SpParams &P, int side, int q, int i, int j, int tper) {
  const int cx = Q == 9 ? cx9(q) : cx5(q), cy = Q == 9 ? cy9(q) : cy5(q);
  int si = i, sj = j, qm;
  if (side >= 2) {
    qm = Q == 9 ? my9(q) : my5(q);
    si = i - cx;
    if (si < 0 || si >= P.nx) si = tper ? wrap(si, P.nx) : i;
  } else {
    qm = Q == 9 ? mx9(q) : mx5(q);
    sj = j - cy;
    if (sj < 0 || sj >= P.ny) sj = tper ? wrap(sj, P.ny) : j;
  }
  return qm * P.plane + (long long)sj * P.pitch + si;
}

// Pre-collision velocity of time t at node n rebuilt from its post-collision
// populations: rho = sum f*, rho u = sum c f* - dt F / 2 (the collision adds dt F
// to the momentum, Eqs. first_moment_f and forcing_term).
template <typename S, typename R>
__device__ __forceinline__ void post_velocity(const SpParams &P, const S *src, int i, int j, R &ux, R &uy, R &rho) {
  long long n = (long long)j * P.pitch + i;
  R f[9];
#pragma unroll
  for (int q = 0; q < 9; q++) f[q] = (R)src[q * P.plane + n];
  R drho = f[0] + f[1] + f[2] + f[3] + f[4] + f[5] + f[6] + f[7] + f[8];
  rho = K<R>(P).rho0 + drho;
  R c = K<R>(P).c;
  R jx = c * ((f[1] - f[3]) + (f[5] - f[6]) + (f[8] - f[7]));
  R jy = c * ((f[2] - f[4]) + (f[5] - f[8]) + (f[6] - f[7]));
  R Fx = K<R>(P).Fx, Fy = K<R>(P).Fy;
  if (P.force) {
    const S *fo = (const S *)P.force;
    Fx += (R)fo[n];
    Fy += (R)fo[P.plane + n];
  }
  if (P.buoy) {
    // buoyancy of T(t) = T0 + sum g* - dt qdot / 2 at this node
    const S *gs = src + (long long)P.gbase * P.plane;
    R sg = (R)0;
#pragma unroll
    for (int q = 0; q < 9; q++)
      if (q < P.qg) sg += (R)gs[q * P.plane + n];
    const R qd = P.qdot ? (R)((const S *)P.qdot)[n] : (R)0;
    const R dT = (K<R>(P).T0 - K<R>(P).T_ref) + sg - (R)0.5 * K<R>(P).dt * qd;
    Fx += K<R>(P).bgx * dT;
    Fy += K<R>(P).bgy * dT;
  }
  const R inv = (R)1 / rho;  // one division for both components
  ux = (jx - (R)0.5 * K<R>(P).dt * Fx) * inv;
  uy = (jy - (R)0.5 * K<R>(P).dt * Fy) * inv;
}

// ---- boundary links ---------------------------------------------------------
// A link along (cx, cy) enters through the x-side cx > 0 ? 0 : 1 or the y-side cy > 0 ?
// 2 : 3, known at compile time; in[s] says whether this node's links enter through side
// s.  Every rule of Sec. 2.1 / 2.2 but the wet node is affine in one stored value:
// f_q = +- raw + w_q (base + cu (lin + quad cu)), cu = c_q . u of the side.  So a node
// gathers one value per link, then goes through the sides it lies on: forms a side's
// coefficients and finishes that side's links.
// The boundary frame is the critical path of a step on small and middle grids: its warps
// run gather, coefficients and links one after the other with few warps beside them.
// Selecting among four sides per link and per attribute took about 4000 instructions a
// warp, whose fetch alone bounded the step (10 of 16 cycles per instruction waiting for
// code).  Measured with the two forms, FP32, back-to-back steps: 2000 x 50 half channel,
// D2Q9 + D2Q9, 13.6 -> 6.8 us; 2048 x 256 channel, D2Q9 + D2Q5, 12.9 -> 10.1 us (64 x 4
// blocks); 128 x 32 channel 7.0 -> 3.7 us.
struct NodeSides {
  bool in[4];
  int xm, xp;             // columns i - 1, i + 1 (wrapped)
  long long r0, rm, rp;   // row offsets of j, j - 1, j + 1 (wrapped)
};

__device__ __forceinline__ NodeSides node_sides(const SpParams &P, int i, int j, int xper, int yper) {
  NodeSides b;
  b.in[0] = !xper && i == 0;
  b.in[1] = !xper && i == P.nx - 1;
  b.in[2] = !yper && j == 0;
  b.in[3] = !yper && j == P.ny - 1;
  b.xm = i == 0 ? P.nx - 1 : i - 1;
  b.xp = i == P.nx - 1 ? 0 : i + 1;
  b.r0 = (long long)j * P.pitch;
  b.rm = (long long)(j == 0 ? P.ny - 1 : j - 1) * P.pitch;
  b.rp = (long long)(j == P.ny - 1 ? 0 : j + 1) * P.pitch;
  return b;
}

// Streaming source of a link along (cx, cy) within its plane.
__device__ __forceinline__ long long stream_at(const NodeSides &b, int i, int cx, int cy) {
  return (cy > 0 ? b.rm : cy < 0 ? b.rp : b.r0) + (cx > 0 ? b.xm : cx < 0 ? b.xp : i);
}

// Whether the link along (cx, cy) enters through side s: a corner link takes the y-side
// unless that one is a symmetry plane (ysym bits) and the x-side stands.
__host__ __device__ constexpr int side_x(int cx) { return cx > 0 ? 0 : 1; }
__host__ __device__ constexpr int side_y(int cy) { return cy > 0 ? 2 : 3; }
__host__ __device__ constexpr bool may_enter(int s, int cx, int cy) {
  return s < 2 ? cx != 0 && side_x(cx) == s : cy != 0 && side_y(cy) == s;
}
template <bool SYM>
__device__ __forceinline__ bool enters(const NodeSides &b, int s, int cx, int cy, int ysym) {
  if (!may_enter(s, cx, cy) || !b.in[s]) return false;
  if (s < 2) return cy == 0 || !b.in[side_y(cy)] || (SYM && ((ysym >> (side_y(cy) - 2)) & 1));
  return !SYM || cx == 0 || !b.in[side_x(cx)] || !((ysym >> (s - 2)) & 1);
}

// Pull of all momentum populations at node (i, j), with boundary links.  SYM: the
// solve has symmetry sides (compiled separately, so that solves without them run the
// shorter boundary code).
template <typename S, typename R, bool SYM = false>
__device__ __forceinline__ void pull_f(const SpParams &P, const S *src, int i, int j, bool interior, R f[9]) {
  const long long n = (long long)j * P.pitch + i;
  if (interior) {
#pragma unroll
    for (int q = 0; q < 9; q++) f[q] = (R)src[q * P.plane + n - (long long)cy9(q) * P.pitch - cx9(q)];
    return;
  }
  if (P.local) {  // src holds f(t) itself (first step after initialisation)
#pragma unroll
    for (int q = 0; q < 9; q++) f[q] = (R)src[q * P.plane + n];
    return;
  }
  // 1. gather, branch-free so that all nine loads are in flight together: the
  //    streaming source (periodic wrap included), or for a link entering through a
  //    side the outgoing population of this node
  //    (a symmetry side gives the mirrored population of the tangential neighbour)
  const NodeSides b = node_sides(P, i, j, P.xper, P.yper);
#pragma unroll
  for (int q = 0; q < 9; q++) {
    const int cx = cx9(q), cy = cy9(q);
    const bool by_x = enters<SYM>(b, side_x(cx), cx, cy, P.fysym), by_y = enters<SYM>(b, side_y(cy), cx, cy, P.fysym);
    long long at = by_x || by_y ? opp9(q) * P.plane + n : q * P.plane + stream_at(b, i, cx, cy);
    if (SYM) {
      if (by_x && P.side[side_x(cx)].kind == BC_SYMMETRY) at = symmetry_source<9>(P, side_x(cx), q, i, j, P.yper);
      if (by_y && P.side[side_y(cy)].kind == BC_SYMMETRY) at = symmetry_source<9>(P, side_y(cy), q, i, j, P.xper);
    }
    f[q] = (R)src[at];
  }
  // 2. the sides this node lies on: walls and velocity inlets (Eq. BB_vel, f_q = f_o* +
  //    2 w rho_w c_q.u_w / c_s^2) and the outlet (Eq. anti_BB_vel in deviation form, f_q =
  //    -f_o* + 2 w [rho_w (1 + (c.u)^2 / 2 c_s^4 - u^2 / 2 c_s^2) - rho0], whose u_w
  //    extrapolates the pre-collision velocities of time t at the boundary node and its
  //    inner neighbour)
  const R ics2 = K<R>(P).inv_cs2;
#pragma unroll
  for (int s = 0; s < 4; s++) {
    if (!b.in[s]) continue;
    const int kind = P.side[s].kind;
    if (SYM && kind == BC_SYMMETRY) continue;
    const R rw = K<R>(P).rho_w[s];
    R ux = 0, uy = 0, base = 0, lin = 0, quad = 0;
    const bool anti = kind == BC_PRESSURE;
    if (anti) {
      R ub, vb, ui, vi, rho;
      post_velocity<S, R>(P, src, i, j, ub, vb, rho);
      post_velocity<S, R>(P, src, i + (s == 0) - (s == 1), j + (s == 2) - (s == 3), ui, vi, rho);
      ux = ub + (R)0.5 * (ub - ui);
      uy = vb + (R)0.5 * (vb - vi);
      base = (R)2 * (rw - K<R>(P).rho0) - rw * (ux * ux + uy * uy) * ics2;
      quad = rw * ics2 * ics2;
    } else {
      const double *uw = P.side[s].uw;
      if (!uw) continue;  // at rest: f_q = f_o*
      const int a = along(s, i, j);
      ux = (R)uw[a];
      uy = (R)uw[side_len(P, s) + a];
      lin = (R)2 * rw * ics2;
    }
#pragma unroll
    for (int q = 1; q < 9; q++) {
      if (!enters<SYM>(b, s, cx9(q), cy9(q), P.fysym)) continue;
      const R cu = K<R>(P).c * ((R)cx9(q) * ux + (R)cy9(q) * uy);
      f[q] = (anti ? -f[q] : f[q]) + w9<R>(q) * (base + cu * (lin + quad * cu));
    }
  }
}

// Pull of the thermal populations (QT = 5: D2Q5, 9: D2Q9) at node (i, j) with
// boundary links.
template <typename S, typename R, int QT = 5, bool SYM = false>
__device__ __forceinline__ void pull_g(const SpParams &P, const S *src, int i, int j, bool interior, R g[QT]) {
  const long long n = (long long)j * P.pitch + i;
  const S *gsrc = src + (long long)P.gbase * P.plane;
  if (interior) {
#pragma unroll
    for (int q = 0; q < QT; q++) g[q] = (R)gsrc[q * P.plane + n - (long long)cyT(QT, q) * P.pitch - cxT(QT, q)];
    return;
  }
  if (P.local) {
#pragma unroll
    for (int q = 0; q < QT; q++) g[q] = (R)gsrc[q * P.plane + n];
    return;
  }
  // 1. gather (branch-free, all loads in flight together)
  const NodeSides b = node_sides(P, i, j, P.txper, P.typer);
#pragma unroll
  for (int q = 0; q < QT; q++) {
    const int cx = cxT(QT, q), cy = cyT(QT, q);
    const bool by_x = enters<SYM>(b, side_x(cx), cx, cy, P.tysym), by_y = enters<SYM>(b, side_y(cy), cx, cy, P.tysym);
    const int tk = by_y ? P.side[side_y(cy)].tkind : P.side[side_x(cx)].tkind;
    long long at = by_x || by_y ? oppT(QT, q) * P.plane + n : q * P.plane + stream_at(b, i, cx, cy);
    if ((by_x || by_y) && tk == TBC_OUTFLOW) {
      // g_q(x_b, t+dt) = g_q(x_b-1, t+dt): the inner node's pull of q (Sec. 2.2, outlet),
      // whose source is in this node's column (row, for a y-side);
      // where that pull itself crosses a symmetry side (the outlet's corner with a
      // symmetry plane) it is that side's mirrored value
      const int si = by_x ? i : min(max(i - cx, 0), P.nx - 1), sj = by_y ? j : min(max(j - cy, 0), P.ny - 1);
      at = q * P.plane + (long long)sj * P.pitch + si;
      if (SYM) {
        const int ii = by_x ? i + cx : i, jj = by_y ? j + cy : j;
        const int cs = entry_side(ii, jj, cx, cy, P.nx, P.ny, P.txper, P.typer, P.tysym);
        bool csym = false;
#pragma unroll
        for (int s = 0; s < 4; s++)
          if (cs == s) csym = P.side[s].tkind == TBC_SYMMETRY;
        if (csym) at = symmetry_source<QT>(P, cs, q, ii, jj, cs >= 2 ? P.txper : P.typer);
      }
    } else if (SYM && (by_x || by_y) && tk == TBC_SYMMETRY) {
      at = symmetry_source<QT>(P, by_y ? side_y(cy) : side_x(cx), q, i, j, by_y ? P.txper : P.typer);
    }
    g[q] = (R)gsrc[at];
  }
  // 2. the sides this node lies on: fixed temperature (Eq. anti_BB_T in deviation form) and
  //    wall flux (Eq. BB_T, lambda_o = 6 w_o on D2Q9, 1 for the single D2Q5 unknown; zero
  //    flux = adiabatic).  D2Q5's one weight is folded into the coefficients
  const R ics2 = K<R>(P).inv_cs2;
  const R wq = QT == 9 ? (R)1 : w5<R>(1);
  R wet[2] = {(R)0, (R)0};
#pragma unroll
  for (int s = 0; s < 4; s++) {
    if (!b.in[s]) continue;
    const int a = along(s, i, j), tk = P.side[s].tkind;
    if (tk == TBC_OUTFLOW || (SYM && tk == TBC_SYMMETRY)) continue;
    const R tw = P.side[s].tw ? (R)P.side[s].tw[a] : (R)0;
    if (SYM && tk == TBC_WETNODE) {
      if (s < 2) wet[s] = tw;
      continue;
    }
    R ux = 0, uy = 0, base, quad = 0;
    const bool anti = tk == TBC_TEMP;
    if (anti) {
      const double *uw = P.side[s].uw;
      if (uw) {
        ux = (R)uw[a];
        uy = (R)uw[side_len(P, s) + a];
      }
      base = wq * ((R)2 * (tw - K<R>(P).T0) - tw * (ux * ux + uy * uy) * ics2);
      quad = wq * (tw * ics2 * ics2);
    } else {
      base = (QT == 9 ? (R)6 : (R)1) * K<R>(P).flux_coef * tw;
    }
#pragma unroll
    for (int q = 1; q < QT; q++) {
      const int cx = cxT(QT, q), cy = cyT(QT, q);
      if (!enters<SYM>(b, s, cx, cy, P.tysym)) continue;
      const R cu = K<R>(P).c * ((R)cx * ux + (R)cy * uy);
      const R v = base + quad * cu * cu;
      g[q] = (anti ? -g[q] : g[q]) + (QT == 9 ? w9<R>(q) * v : v);
    }
  }
  // 3. wet-node x-sides (App. B, Eq. BCs_1D_advection_diffusion): the boundary node lies
  //    on the boundary; its single D2Q5 unknown closes T of Eq. zero_moment_g at T_w,
  //    g_unknown = T_w - dt qdot/2 - (sum of the others), in deviation form
  if (SYM && QT == 5) {
#pragma unroll
    for (int s = 0; s < 2; s++) {
      if (P.side[s].tkind != TBC_WETNODE || i != (s == 0 ? 0 : P.nx - 1)) continue;
      const int qu = s == 0 ? 1 : 3;
      R others = (R)0;
#pragma unroll
      for (int k = 0; k < QT; k++)
        if (k != qu) others += g[k];
      const R qd = P.qdot ? (R)((const S *)P.qdot)[n] : (R)0;
      g[qu] = (wet[s] - K<R>(P).T0) - (R)0.5 * K<R>(P).dt * qd - others;
    }
  }
}

// ----------------------------------------------------------------------------
// Moments and collisions (deviation form)
// ----------------------------------------------------------------------------
// The collisions work on pairs of opposite populations: with a = f_q + f_opp and
// d = f_q - f_opp, a pair changes by (dP + dQ, dP - dQ), dP the change of its even
// moments and dQ of its odd ones.  On the pairs every MRT operator of Sec. 2.1 / 2.2 is a
// handful of products (the same operator as M^-1 Lambda M, with factors folded on the host
// into SpConst).  The changes are formed from the small non-equilibrium parts and added to
// the populations once, so that a population is rounded once per step, and the conserved
// moments are kept by construction.
// Why in this form: on GB300 the FP64 pipe issues one warp instruction every 16 cycles
// per SM and bounds the FP64 step, so the count of FP64 instructions per node is its
// time.  The unfolded form (moments, equilibria and forcing of all nine rates, then
// M^-1) took 198 per node of D2Q9 MRT + D2Q5 MRT, this one 94.  Measured, back-to-back
// steps: FP64 2048 x 256 191.6 -> 102.4 us, FP64 64 x 33 BGK 14.6 -> 8.5 us, FP32 2048 x 256
// 10.1 -> 9.1 us; the error against a 64-bit solution is not larger in either precision.
template <typename R>
struct Macro {
  R drho, rho, ux, uy, Fx, Fy;  // momentum
  R hx, hy, jx, jy;             // lattice-scaled: u / c and rho u / c
  R sumg, qd, dT, T;            // thermal; dT = T - T0
};

template <typename S, typename R>
__device__ __forceinline__ void load_sources(const SpParams &P, long long n, Macro<R> &m) {
  m.Fx = K<R>(P).Fx;
  m.Fy = K<R>(P).Fy;
  if (P.force) {
    const S *fo = (const S *)P.force;
    m.Fx += (R)fo[n];
    m.Fy += (R)fo[P.plane + n];
  }
  m.qd = P.qdot ? (R)((const S *)P.qdot)[n] : (R)0;
}

// Sums over a lattice's populations that moments and collisions share (written once, so
// that both use the same instructions): s14 = f1 + .. + f4, s58 = f5 + .. + f8 and the
// lattice-scaled first moment.
template <typename R>
__device__ __forceinline__ R sum14(const R *f) { return (f[1] + f[3]) + (f[2] + f[4]); }
template <typename R>
__device__ __forceinline__ R sum58(const R *f) { return (f[5] + f[7]) + (f[6] + f[8]); }
template <typename R>
__device__ __forceinline__ R first_x9(const R *f) { return (f[1] - f[3]) + ((f[5] - f[7]) - (f[6] - f[8])); }
template <typename R>
__device__ __forceinline__ R first_y9(const R *f) { return (f[2] - f[4]) + ((f[5] - f[7]) + (f[6] - f[8])); }

template <typename R, int FLOW, int TH>
__device__ __forceinline__ void moments(const SpParams &P, const R f[9], const R *g, Macro<R> &m) {
  if (TH != TH_NONE) {
    // Eq. zero_moment_g
    m.sumg = ThLat<TH>::Q == 9 ? g[0] + (sum14(g) + sum58(g)) : g[0] + sum14(g);
    m.dT = m.sumg;
    if (P.qdot) m.dT += K<R>(P).hdt * m.qd;
    m.T = K<R>(P).T0 + m.dT;
    if (FLOW != FLOW_NONE && P.buoy) {
      // Boussinesq buoyancy with this step's temperature (Eq. buoyancy_force)
      const R dT = (K<R>(P).T0 - K<R>(P).T_ref) + m.dT;
      m.Fx += K<R>(P).bgx * dT;
      m.Fy += K<R>(P).bgy * dT;
    }
  }
  if (FLOW != FLOW_NONE) {
    // Eqs. zero_moment_f and first_moment_f
    m.drho = f[0] + (sum14(f) + sum58(f));
    m.rho = K<R>(P).rho0 + m.drho;
    m.jx = first_x9(f);
    m.jy = first_y9(f);
    if (P.forced) {
      m.jx += K<R>(P).hdt_ic * m.Fx;
      m.jy += K<R>(P).hdt_ic * m.Fy;
    }
    const R inv = recip(m.rho);
    m.hx = m.jx * inv;
    m.hy = m.jy * inv;
    m.ux = K<R>(P).c * m.hx;
    m.uy = K<R>(P).c * m.hy;
  } else {
    m.drho = 0;
    m.rho = K<R>(P).rho0;
    m.ux = K<R>(P).ux_pres;
    m.uy = K<R>(P).uy_pres;
    m.hx = m.ux * K<R>(P).inv_c;
    m.hy = m.uy * K<R>(P).inv_c;
  }
}

// Momentum collision: MRT (Eq. colisao_MRT, [M]_dim of Eq. M_matrix_dim, Guo forcing),
// and BGK as the MRT whose rates all equal dt / tau (set on the host).  With
// h = u / c, j = rho h:
//   even moments   stress: s_nu times the distance of the pair differences from
//                  rho h_x^2 - rho h_y^2 and rho h_x h_y; energy and energy square: at
//                  rate 1 (unit_e) to the equilibrium, else relaxed by the distances of
//                  the two moments (over 1 and 3) from their equilibria;
//   odd moments    axis pairs: (s_q / 6)(t + j - 2 d), t the diagonals' share of the first
//                  moment; diagonal pairs: minus half of that, which keeps the momentum.
template <typename R>
__device__ __forceinline__ void collide_flow(const SpParams &P, const Macro<R> &m, R f[9]) {
  const SpConst<R> &k = K<R>(P);
  const R d13 = f[1] - f[3], d24 = f[2] - f[4], d57 = f[5] - f[7], d68 = f[6] - f[8];
  const R a13 = f[1] + f[3], a24 = f[2] + f[4], a57 = f[5] + f[7], a68 = f[6] + f[8];
  const R s14 = a13 + a24, s58 = a57 + a68;
  const R xx0 = m.jx * m.hx, ru = xx0 + m.jy * m.hy, rxx = xx0 - m.jy * m.hy, rxy = m.jx * m.hy;
  R dX = k.kn * (rxx - (a13 - a24)), dY = k.kn * (rxy - (a57 - a68));
  R ox = k.kq * (((d57 - d68) + m.jx) - (R)2 * d13);
  R oy = k.kq * (((d57 + d68) + m.jy) - (R)2 * d24);
  R d4, d8;  // change of every axis and of every diagonal population's share of the energies
  R f0;
  if (P.unit_e) {
    const R r12 = ru * ((R)1 / (R)12);
    const R e4 = m.drho * ((R)1 / (R)9) + r12, e8 = m.drho * ((R)1 / (R)36) + r12;
    d4 = e4 - (R)0.25 * s14;
    d8 = e8 - (R)0.25 * s58;
    f0 = sizeof(R) == 8 ? m.drho - (R)4 * (e4 + e8) : f[0] - (R)4 * (d4 + d8);  // FP32: see collide_mrt5
  } else {
    const R a1 = k.ke * (((s14 - (R)2 * f[0]) + (R)4 * s58) - (R)3 * ru), a2 = k.kep * ((f[0] - s14) + ru);
    d4 = a1 + (R)2 * a2;
    d8 = -((R)2 * a1 + a2);
    f0 = f[0] + (R)4 * (a1 - a2);
  }
  R w = (R)0.5 * (oy + ox), v = (R)0.5 * (oy - ox);
  if (P.forced) {
    const R px = m.Fx * k.inv_c, py = m.Fy * k.inv_c, uF = m.hx * px + m.hy * py;
    dX += k.gn * (m.hx * px - m.hy * py);
    dY += (R)0.5 * k.gn * (m.hx * py + m.hy * px);
    ox += k.gq * px;
    oy += k.gq * py;
    w -= k.gd * (py + px);
    v -= k.gd * (py - px);
    d4 += k.g4 * uF;
    d8 += k.g8 * uF;
    f0 -= (R)4 * ((k.g4 + k.g8) * uF);
  }
  const R p13 = d4 + dX, p24 = d4 - dX, p57 = d8 + dY, p68 = d8 - dY;
  f[0] = f0;
  f[1] += p13 + ox;
  f[3] += p13 - ox;
  f[2] += p24 + oy;
  f[4] += p24 - oy;
  f[5] += p57 - w;
  f[7] += p57 + w;
  f[6] += p68 - v;
  f[8] += p68 + v;
}

// d - T h without rounding the absolute temperature (T0 and T - T0 apart).
template <typename R>
__device__ __forceinline__ R off_eq(const Macro<R> &m, R T0, R d, R h) { return (d - T0 * h) - m.dT * h; }

// Thermal BGK with source (Eqs. eq_lattice_boltzmann_BGK_T, forcing_term_g, geq_geral)
// on the thermal lattice QT: even pairs by w (omega dT + src) - (omega / 2) a, odd pairs
// by -(omega / 2)(d - d_eq), rest population from the remainder.
template <typename R, int QT>
__device__ __forceinline__ void collide_bgk_T(const SpParams &P, const Macro<R> &m, R *g) {
  const SpConst<R> &k = K<R>(P);
  const R d13 = g[1] - g[3], d24 = g[2] - g[4], a13 = g[1] + g[3], a24 = g[2] + g[4];
  const R om = k.omegaT, ho = k.hsT;
  R b = om * m.dT, dS = (R)0;
  if (P.qdot) {
    const R src = k.tsrc_fac * k.dt * m.qd;
    b += src;
    dS = om * (k.hdt * m.qd) + src;  // sum g changes by the source alone
  }
  if (QT == 5) {
    const R b6 = b * ((R)1 / (R)6);
    const R px = b6 - ho * a13, py = b6 - ho * a24;
    const R ox = ho * off_eq(m, k.T0, d13, m.hx), oy = ho * off_eq(m, k.T0, d24, m.hy);
    g[0] += dS - (R)2 * (px + py);
    g[1] += px - ox;
    g[3] += px + ox;
    g[2] += py - oy;
    g[4] += py + oy;
    return;
  }
  // D2Q9: equilibrium differences (2/3) T h on the axes, T (h_y +- h_x) / 6 on the diagonals
  const R d57 = g[5] - g[7], d68 = g[6] - g[8], a57 = g[5] + g[7], a68 = g[6] + g[8];
  const R b9 = b * ((R)1 / (R)9), b36 = b * ((R)1 / (R)36);
  const R p13 = b9 - ho * a13, p24 = b9 - ho * a24, p57 = b36 - ho * a57, p68 = b36 - ho * a68;
  const R hx = m.hx * ((R)2 / (R)3), hy = m.hy * ((R)2 / (R)3);
  const R ha = (m.hy + m.hx) * ((R)1 / (R)6), hb = (m.hy - m.hx) * ((R)1 / (R)6);
  const R o13 = ho * off_eq(m, k.T0, d13, hx), o24 = ho * off_eq(m, k.T0, d24, hy);
  const R o57 = ho * off_eq(m, k.T0, d57, ha), o68 = ho * off_eq(m, k.T0, d68, hb);
  g[0] += dS - (R)2 * ((p13 + p24) + (p57 + p68));
  g[1] += p13 - o13;
  g[3] += p13 + o13;
  g[2] += p24 - o24;
  g[4] += p24 + o24;
  g[5] += p57 - o57;
  g[7] += p57 + o57;
  g[6] += p68 - o68;
  g[8] += p68 + o68;
}

// Adds x to the rest population; returns what its rounding left of x.
template <typename R>
__device__ __forceinline__ R rest_change(R &g0, R x) {
  const R n = g0 + x, left = x - (n - g0);
  g0 = n;
  return left;
}

// Thermal MRT on D2Q5: moments (1, c_x, c_y, 5|c|^2 - 4c^2, c_x^2 - c_y^2), rates
// (0, 1/tau_T, 1/tau_T, 1/dt, 1/dt), source Delta t (I - dt Lambda/2) M (w qdot).  The two
// even moments at rate 1/dt take every even pair to w S, S = sum g + dt qdot.
// FP64: through S (the rest population is S - 4 p, exact).
// In FP32 a source of one step is about a unit in the last place of sum g, or less: S rounded
// loses or doubles it, the same way step after step at a node, and sum g drifts without a
// source too.  So that form adds changes: of the pairs, w (S - a / 2 w) from a difference that
// is exact, of the rest population, what the source and the pairs leave, and what its own
// rounding leaves of that goes to the axis pairs, whose odd parts keep their rounding from
// repeating.
// T - T_in against the FP64 form, relative L2: 1024 x 128 channel with q = 1e6 W/m^3, 2000 steps
// 1.8e-5 through S, 1.4e-6 with changes, 9.6e-7 with the remainder (1e5 W/m^3, 50000 steps: 1.0e-5
// with changes, 1.3e-6); 700 x 96 without a source, 10000 steps 5.7e-6 through S, 1.3e-6.
// Cost: 0.4 % of the step on 8192 x 4096, 0.6 % on 2048 x 256.
template <typename R>
__device__ __forceinline__ void collide_mrt5(const SpParams &P, const Macro<R> &m, R g[5]) {
  const SpConst<R> &k = K<R>(P);
  const R d13 = g[1] - g[3], d24 = g[2] - g[4], a13 = g[1] + g[3], a24 = g[2] + g[4];
  const R w = (R)1 / (R)6;
  R px, py;
  if (sizeof(R) == 8) {
    const R S = P.qdot ? m.sumg + k.dt * m.qd : m.sumg, p = S * w;
    px = p - (R)0.5 * a13;
    py = p - (R)0.5 * a24;
    g[0] = S - (R)4 * p;
  } else {
    const R dS = P.qdot ? k.dt * m.qd : (R)0;
    px = w * (fma((R)-3, a13, m.sumg) + dS);
    py = w * (fma((R)-3, a24, m.sumg) + dS);
    const R left = rest_change(g[0], dS - (R)2 * (px + py));
    px += (R)0.25 * left;
    py += (R)0.25 * left;
  }
  const R ex = off_eq(m, k.T0, d13, m.hx), ey = off_eq(m, k.T0, d24, m.hy);
  g[1] += px - k.hsT * ex;
  g[3] += px + k.hsT * ex;
  g[2] += py - k.hsT * ey;
  g[4] += py + k.hsT * ey;
}

// Thermal MRT on D2Q9 (Sec. 2.2): the momentum transformation matrices and
// [Lambda_T] = diag(0, 1, 1, omega_T, 1, omega_T, 1, 1, 1), the unit rates read as
// 1/dt; source Delta t (I - dt Lambda/2) M (w qdot).  Every even pair goes to w S,
// S = sum g + dt qdot (in the two forms of D2Q5); of the odd moments the first loses s_T of
// its distance e = j - T h from equilibrium, the third-order ones go to -T h.
template <typename R>
__device__ __forceinline__ void collide_mrt9T(const SpParams &P, const Macro<R> &m, R g[9]) {
  const SpConst<R> &k = K<R>(P);
  const R d13 = g[1] - g[3], d24 = g[2] - g[4], d57 = g[5] - g[7], d68 = g[6] - g[8];
  const R a13 = g[1] + g[3], a24 = g[2] + g[4], a57 = g[5] + g[7], a68 = g[6] + g[8];
  const R w4 = (R)1 / (R)9, w8 = (R)1 / (R)36;
  R p13, p24, p57, p68;
  if (sizeof(R) == 8) {
    const R S = P.qdot ? m.sumg + k.dt * m.qd : m.sumg, p9 = S * w4, p36 = S * w8;
    p13 = p9 - (R)0.5 * a13;
    p24 = p9 - (R)0.5 * a24;
    p57 = p36 - (R)0.5 * a57;
    p68 = p36 - (R)0.5 * a68;
    g[0] = S - (R)4 * (p9 + p36);
  } else {
    const R dS = P.qdot ? k.dt * m.qd : (R)0;
    p13 = w4 * (fma((R)-4.5, a13, m.sumg) + dS);
    p24 = w4 * (fma((R)-4.5, a24, m.sumg) + dS);
    p57 = w8 * (fma((R)-18, a57, m.sumg) + dS);
    p68 = w8 * (fma((R)-18, a68, m.sumg) + dS);
    const R left = rest_change(g[0], dS - (R)2 * ((p13 + p24) + (p57 + p68)));
    p13 += (R)0.25 * left;
    p24 += (R)0.25 * left;
  }
  const R tx = d57 - d68, ty = d57 + d68;  // the diagonals' share of the first moment
  const R ex = off_eq(m, k.T0, d13 + tx, m.hx), ey = off_eq(m, k.T0, d24 + ty, m.hy);
  const R ox = ((R)2 * tx - d13) * ((R)1 / (R)6) - k.q1T * ex, oy = ((R)2 * ty - d24) * ((R)1 / (R)6) - k.q1T * ey;
  const R w = (R)0.5 * (ox + oy) + k.q2T * (ex + ey), v = (R)0.5 * (oy - ox) + k.q2T * (ey - ex);
  g[1] += p13 + ox;
  g[3] += p13 - ox;
  g[2] += p24 + oy;
  g[4] += p24 - oy;
  g[5] += p57 - w;
  g[7] += p57 + w;
  g[6] += p68 - v;
  g[8] += p68 + v;
}

template <typename R, int FLOW, int TH>
__device__ __forceinline__ void collide(const SpParams &P, const Macro<R> &m, R f[9], R *g) {
  if (FLOW != FLOW_NONE) collide_flow<R>(P, m, f);
  if (TH == TH_BGK) collide_bgk_T<R, 5>(P, m, g);
  if (TH == TH_MRT) collide_mrt5<R>(P, m, g);
  if (TH == TH_BGK9) collide_bgk_T<R, 9>(P, m, g);
  if (TH == TH_MRT9) collide_mrt9T<R>(P, m, g);
}

}  // namespace lbmk
