// Reverse-time (discrete) adjoint of the single-phase fused step: D2Q9 MRT
// momentum + D2Q5 MRT thermal, FP64 or FP32 (the adjoint of the FP32 deviation
// form: states stored as FP32 deviations, adjoint variables and arithmetic in FP32,
// parameter gradients accumulated to FP64 precision: FP64 sums, or in the FP32 form
// compensated FP32 pairs), with the channel boundary rules
// (BB-velocity inlet and walls, anti-BB pressure outlet with extrapolated
// velocity, anti-BB temperature inlet, heat-flux walls, thermal outflow).
//
// Forward (step_sp.cu): X_t = C(P(X_{t-1})), where P is the pull with boundary
// links and C the local collision; X_{-1} is the pre-collision initial state.
// Loss: L = (1/ny) sum_j (T(nx-1, j; N) - T_target(j))^2 with T of P(X_{N-1}).
// Reverse step t (N-1 >= t >= 0), one launch per node grid:
//   Lam_X(t)   = P^T Lam_pre(t+1)       gather from the consumers of X_t: the
//                                        streaming neighbour, the node's own
//                                        reflected links, the thermal outflow,
//                                        and the outlet velocity extrapolation;
//   Lam_pre(t) = C'(pre(t))^T Lam_X(t)   local transposed Jacobian of the MRT
//                                        collisions (moments, equilibria,
//                                        forcing, u = j/rho, T = sum g + dt qdot/2),
// with pre(t) recomputed by pulling X_{t-1}.  Parameter gradients accumulate per
// node (qdot, wall flux) or per block (the two nu-dependent MRT rates), so the
// result does not depend on scheduling.
#include <cuda_runtime.h>

#include "lattice.cuh"
#include "lbm_internal.cuh"
#include "sp_device.cuh"
#include "compensated.cuh"

namespace lbmk {

namespace {

__device__ __forceinline__ long long nidx(const SpParams &P, int i, int j) { return (long long)j * P.pitch + i; }

// The outlet's velocity extrapolation u_w = 1.5 u(x_b) - 0.5 u(x_b-1) seen from the node
// (i, j) itself (`on`, the boundary node of side s) or from its inner neighbour: the
// adjoint of u_w, G = sum over the side's unknown populations p of Lam_pre_p
// d(pre_p)/d(u_w), times d(u_w)/d(u at this node) / rho; and this node's velocity.
template <typename S, typename R>
__device__ __forceinline__ void outlet_adjoint(const SpParams &P, const S *Xt, const R *LPn, int s, bool on, int i, int j,
                                               R &Gx, R &Gy, R &ux, R &uy) {
  const int di = (s == 0) - (s == 1), dj = (s == 2) - (s == 3);  // inward
  const int bi = on ? i : i - di, bj = on ? j : j - dj;
  R ub, vb, ui, vi, rb, ri;
  post_velocity<S, R>(P, Xt, bi, bj, ub, vb, rb);
  post_velocity<S, R>(P, Xt, bi + di, bj + dj, ui, vi, ri);
  const R wx = ub + (R)0.5 * (ub - ui), wy = vb + (R)0.5 * (vb - vi);
  const R c = K<R>(P).c, ics2 = K<R>(P).inv_cs2, rw = K<R>(P).rho_w[s];
  const long long nb = nidx(P, bi, bj);
  Gx = 0;
  Gy = 0;
#pragma unroll
  for (int p = 1; p < 9; p++) {
    if (entry_side(bi, bj, cx9(p), cy9(p), P.nx, P.ny, P.xper, P.yper) != s) continue;
    // d/d u_w of the anti-BB rule 2 w rho_w ((c.u)^2 / 2 c_s^4 - u^2 / 2 c_s^2)
    const R cx = c * (R)cx9(p), cy = c * (R)cy9(p);
    const R k = (R)2 * w9<R>(p) * rw * ics2 * LPn[p * P.plane + nb], cu = (cx * wx + cy * wy) * ics2;
    Gx += k * (cu * cx - wx);
    Gy += k * (cu * cy - wy);
  }
  const R coef = (on ? (R)1.5 : (R)-0.5) / (on ? rb : ri);
  Gx *= coef;
  Gy *= coef;
  ux = on ? ub : ui;
  uy = on ? vb : vi;
}

// Lam_X(t) = P^T Lam_pre(t+1) at a node within two cells of a side.  Population q of this
// node is consumed by the streaming neighbour along c_q, or where that link leaves the
// domain by the node's own reflected link opp(q) of that side; the outlet and the thermal
// outflow add theirs.
template <typename S, typename R>
__device__ __forceinline__ void gather_frame(const SpParams &P, const S *Xt, const R *LPn, int i, int j, R lx[9], R lg[5],
                                             double *grad_flux2, double *grad_flux3) {
  const long long n = nidx(P, i, j);
  const NodeSides b = node_sides(P, i, j, P.xper, P.yper);
#pragma unroll
  for (int q = 0; q < 9; q++) {
    const int p = opp9(q), cx = cx9(p), cy = cy9(p);
    const bool by_x = enters<false>(b, side_x(cx), cx, cy, 0), by_y = enters<false>(b, side_y(cy), cx, cy, 0);
    const int kind = by_y ? P.side[side_y(cy)].kind : P.side[side_x(cx)].kind;
    // (the streaming source of opp(q) is the consumer of q)
    const R v = LPn[by_x || by_y ? p * P.plane + n : q * P.plane + stream_at(b, i, cx, cy)];
    lx[q] = (by_x || by_y) && kind == BC_PRESSURE ? -v : v;
  }
#pragma unroll 1
  for (int s = 0; s < 4; s++) {
    if (P.side[s].kind != BC_PRESSURE) continue;
    const int d = s == 0 ? i : s == 1 ? P.nx - 1 - i : s == 2 ? j : P.ny - 1 - j;  // distance from the side
    if (d > 1) continue;
    R Gx, Gy, ux, uy;
    outlet_adjoint<S, R>(P, Xt, LPn, s, d == 0, i, j, Gx, Gy, ux, uy);
    const R c = K<R>(P).c;
#pragma unroll
    for (int q = 0; q < 9; q++) lx[q] += Gx * (c * (R)cx9(q) - ux) + Gy * (c * (R)cy9(q) - uy);
  }
  const R *LPng = LPn + (long long)P.gbase * P.plane;
  const NodeSides t = node_sides(P, i, j, P.txper, P.typer);
#pragma unroll
  for (int q = 0; q < 5; q++) {
    const int p = opp5(q), cx = cx5(p), cy = cy5(p);
    const int s = cx != 0 ? side_x(cx) : side_y(cy);  // an axis link has one side
    const bool out = enters<false>(t, s, cx, cy, 0);
    const int tk = P.side[s].tkind;
    R v = LPng[out ? p * P.plane + n : q * P.plane + stream_at(t, i, cx, cy)];
    if (out) v = tk == TBC_FLUX ? v : tk == TBC_TEMP ? -v : (R)0;
    // wall heat flux gradient: pre_p = X_q + flux_coef q''(a) on flux sides
    if (out && s >= 2 && tk == TBC_FLUX) (s == 2 ? grad_flux2 : grad_flux3)[i] += P.flux_coef * (double)v;
    // outflow consumer: the unknown q of an outflow side reads X_q of this node
    const int sq = cx != 0 ? side_x(-cx) : side_y(-cy);
    if (enters<false>(t, sq, -cx, -cy, 0) && P.side[sq].tkind == TBC_OUTFLOW) v += LPng[q * P.plane + n];
    lg[q] = v;
  }
}

}  // namespace

// Per-node parameter-gradient accumulators (8 bytes per node): an FP64 sum, or in the
// FP32 form a compensated FP32 pair (hi, lo) in the same 8 bytes, so that the reverse
// step runs no FP64 instruction per node.  grad_value() gives the FP64 value.
__device__ __forceinline__ void grad_add(double *g, long long n, double v) { g[n] += v; }
__device__ __forceinline__ void grad_add(double *g, long long n, float v) {
  float2 *g2 = reinterpret_cast<float2 *>(g);
  float2 a = g2[n];
  float e;
  two_sum(a.x, v, a.x, e);
  a.y += e;
  g2[n] = a;
}
// An FP64 value into the accumulator of a form with working precision R.
template <typename R> __device__ __forceinline__ void grad_add_fp64(double *g, long long n, double v);
template <> __device__ __forceinline__ void grad_add_fp64<double>(double *g, long long n, double v) { g[n] += v; }
template <> __device__ __forceinline__ void grad_add_fp64<float>(double *g, long long n, double v) {
  const float hi = (float)v, lo = (float)(v - (double)hi);  // v = hi + lo to ~2^-48
  float2 *g2 = reinterpret_cast<float2 *>(g);
  float2 a = g2[n];
  float e;
  two_sum(a.x, hi, a.x, e);
  a.y += e + lo;
  g2[n] = a;
}

// Loss at the outlet column and the seed Lam_pre(N).  One thread per row j.  T - T_target
// is formed in FP64 in both forms (FP32 would resolve T ~ 300 K only to ~3e-5 K).
template <typename S, typename R>
__global__ void k_adj_loss(const SpParams P, const double *Ttarget, R *LP, double *grad_qdot, double *loss_rows) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= P.ny) return;
  const int i = P.nx - 1;
  const S *src = (const S *)P.src;
  const bool interior = false;
  R g[5];
  pull_g<S, R>(P, src, i, j, interior, g);
  const long long n = nidx(P, i, j);
  const double qd = P.qdot ? (double)((const S *)P.qdot)[n] : 0.0;
  const double T = P.T0 + (double)((g[0] + g[1]) + (g[2] + g[3]) + g[4]) + 0.5 * P.dt * qd;
  const double e = T - Ttarget[j];
  loss_rows[j] = e * e / P.ny;
  const double dLdT = 2.0 * e / P.ny;
  R *LPg = LP + (long long)P.gbase * P.plane;
#pragma unroll
  for (int q = 0; q < 5; q++) LPg[q * P.plane + n] = (R)dLdT;
  grad_add_fp64<R>(grad_qdot, n, 0.5 * P.dt * dLdT);
}

// The node's share of a reverse step after Lam_X(t) is known: pre(t) from X_{t-1}, the
// transposed collisions (the pair forms of sp_device.cuh, reversed line by line), the
// parameter gradients and Lam_pre(t).  dn, dq: this node's share of 4 dL/ds_nu and 6 dL/ds_q.
template <typename S, typename R, bool INNER>
__device__ __forceinline__ void reverse_node(const SpParams &P, int i, int j, R lx[9], R lg[5], R *LP, double *grad_qdot,
                                             R &dn, R &dq) {
  const long long n = nidx(P, i, j);
  const SpConst<R> &k = K<R>(P);
  const S *src = (const S *)P.src;
  R f[9], g[5];
  if (INNER) {  // P.local (t = 0): the node's own values are the pre-collision state
    const S *gs = src + (long long)P.gbase * P.plane;
    const long long row = P.local ? 0 : P.pitch;
    const int col = P.local ? 0 : 1;
#pragma unroll
    for (int q = 0; q < 9; q++) f[q] = (R)src[q * P.plane + n - cy9(q) * row - cx9(q) * col];
#pragma unroll
    for (int q = 0; q < 5; q++) g[q] = (R)gs[q * P.plane + n - cy5(q) * row - cx5(q) * col];
  } else {
    const bool interior = !P.local && (i > 0) && (i < P.nx - 1) && (j > 0) && (j < P.ny - 1);
    pull_f<S, R>(P, src, i, j, interior, f);
    pull_g<S, R>(P, src, i, j, interior, g);
  }
  Macro<R> m;
  load_sources<S, R>(P, n, m);
  moments<R, FLOW_MRT, TH_MRT>(P, f, g, m);
  const R inv = recip(m.rho), hx = m.hx, hy = m.hy;
  const R half = (R)0.5, two = (R)2;

  // thermal D2Q5 MRT: S = sum g + dt qdot to the weights, e = d - T h at rate s_T
  const R m13 = lg[1] - lg[3], m24 = lg[2] - lg[4];
  const R X = -k.hsT * m13, Y = -k.hsT * m24;
  // (2 l0 + l1 + .. + l4) / 6 from the differences, so that equal ones stay exactly equal
  const R lS = lg[0] + (((lg[1] + lg[3]) + (lg[2] + lg[4])) - (R)4 * lg[0]) * ((R)1 / (R)6);
  const R lT = -(hx * X + hy * Y);
  grad_add(grad_qdot, n, (R)(k.dt * lS + k.hdt * lT));
  R Hx = -m.T * X, Hy = -m.T * Y;  // adjoint of h through the advected heat
  const R lsum = lS + lT;
  R *LPg = LP + (long long)P.gbase * P.plane;
  const R kT = half - k.hsT;
  LPg[n] = lsum;
  LPg[1 * P.plane + n] = lsum + kT * m13;
  LPg[3 * P.plane + n] = lsum - kT * m13;
  LPg[2 * P.plane + n] = lsum + kT * m24;
  LPg[4 * P.plane + n] = lsum - kT * m24;

  // momentum D2Q9 MRT: adjoints of the pair changes ...
  const R p13 = lx[1] + lx[3], o13 = lx[1] - lx[3], p24 = lx[2] + lx[4], o24 = lx[2] - lx[4];
  const R p57 = lx[5] + lx[7], o57 = lx[5] - lx[7], p68 = lx[6] + lx[8], o68 = lx[6] - lx[8];
  const R A4 = p13 + p24, AX = p13 - p24, A8 = p57 + p68, AY = p57 - p68;
  const R Ox = o13 - half * (o57 - o68), Oy = o24 - half * (o57 + o68);
  const R kx = k.kq * Ox, ky = k.kq * Oy, bX = k.kn * AX, bY = k.kn * AY;
  // ... of the energies (s4, s8: what is left of half the pair sums; l0: of f_0) ...
  R s4 = 0, s8 = 0, l0 = 0, lr, lru;
  if (P.unit_e) {
    const R E4 = A4 - (R)4 * lx[0], E8 = A8 - (R)4 * lx[0];
    lr = lx[0] + (E4 * ((R)1 / (R)9) + E8 * ((R)1 / (R)36));
    lru = (E4 + E8) * ((R)1 / (R)12);
  } else {
    const R c1 = k.ke * ((A4 - two * A8) + (R)4 * lx[0]), c2 = k.kep * ((two * A4 - A8) - (R)4 * lx[0]);
    lr = 0;
    lru = c2 - (R)3 * c1;
    l0 = lx[0] + (c2 - two * c1);
    s4 = (R)0.25 * A4 + (c1 - c2);
    s8 = (R)0.25 * A8 + (R)4 * c1;
  }
  // ... of the stress: rho u^2 terms through j and rho ...
  const R u2 = two * (lru + bX), v2 = two * (lru - bX);
  R Jx = u2 * hx + bY * hy, Jy = v2 * hy + bY * hx;
  lr -= half * (hx * Jx + hy * Jy);
  // 4 d L / d s_nu and 6 d L / d s_q
  const R xx = (f[1] + f[3]) - (f[2] + f[4]), xy = (f[5] + f[7]) - (f[6] + f[8]);
  const R tx = (f[5] - f[7]) - (f[6] - f[8]), ty = (f[5] - f[7]) + (f[6] - f[8]);
  const R xx0 = m.jx * hx;
  dn = AX * ((xx0 - m.jy * hy) - xx) + AY * (m.jx * hy - xy);
  dq = Ox * ((tx + m.jx) - two * (f[1] - f[3])) + Oy * ((ty + m.jy) - two * (f[2] - f[4]));
  if (P.forced) {
    const R px = m.Fx * k.inv_c, py = m.Fy * k.inv_c;
    const R gX = k.gn * AX, gY = half * k.gn * AY;
    R lF = k.g4 * A4 + k.g8 * A8 - (R)4 * (k.g4 + k.g8) * lx[0];
    Hx += (lF + gX) * px + gY * py;
    Hy += (lF - gX) * py + gY * px;
    dn -= k.dt * (AX * (hx * px - hy * py) + half * AY * (hx * py + hy * px));
    dq -= half * k.dt * (Ox * px + Oy * py);
  }
  // ... and of h = j / rho
  Hx *= inv;
  Hy *= inv;
  lr -= hx * Hx + hy * Hy;
  Jx += kx + Hx;
  Jy += ky + Hy;
  const R qx = Jx + kx, qy = Jy + ky;  // of the diagonals' share of the first moment
  const R d13 = half * o13 + (Jx - two * kx), d24 = half * o24 + (Jy - two * ky);
  const R d57 = half * o57 + (qy + qx), d68 = half * o68 + (qy - qx);
  const R kr = (R)0.25 - k.kn;
  const R e4 = lr + s4, e8 = lr + s8, a13 = e4 + kr * AX, a24 = e4 - kr * AX, a57 = e8 + kr * AY, a68 = e8 - kr * AY;
  LP[n] = lr + l0;
  LP[1 * P.plane + n] = a13 + d13;
  LP[3 * P.plane + n] = a13 - d13;
  LP[2 * P.plane + n] = a24 + d24;
  LP[4 * P.plane + n] = a24 - d24;
  LP[5 * P.plane + n] = a57 + d57;
  LP[7 * P.plane + n] = a57 - d57;
  LP[6 * P.plane + n] = a68 + d68;
  LP[8 * P.plane + n] = a68 - d68;
}

// Nodes within two cells of a side, each once: the rows j < 2 and j >= ny - 2, then the
// columns i < 2 and i >= nx - 2 between them.
__host__ __device__ inline int adj_frame_nodes(int nx, int ny) {
  const int rows = ny < 4 ? ny : 4, cols = nx < 4 ? nx : 4;
  return rows * nx + cols * (ny - rows);
}
__device__ __forceinline__ bool adj_frame_node(int nx, int ny, int f, int &i, int &j) {
  const int rows = ny < 4 ? ny : 4, cols = nx < 4 ? nx : 4, inner = ny - rows;
  if (f < rows * nx) {
    const int r = f / nx;
    i = f - r * nx;
    j = ny < 4 || r < 2 ? r : ny - 4 + r;
    return true;
  }
  f -= rows * nx;
  if (inner <= 0 || f >= cols * inner) return false;
  const int c = f / inner;
  i = nx < 4 || c < 2 ? c : nx - 4 + c;
  j = 2 + f - c * inner;
  return true;
}

// One reverse step.  P.src = X_{t-1} (P.local = 1 when t = 0), Xt = X_t,
// LPn = Lam_pre(t+1), LP = Lam_pre(t) (output).
// The first nfb blocks take the nodes within two cells of a side (the long path; they
// start first and share no warp with others), the others 64 nodes of a row each, whose
// consumers are all ordinary streaming links, with the boundary code compiled out: in one
// mixed launch the step waited for the warps that ran both paths one after the other and
// for their code.
// cn, cq: (1/4) d s_nu / d nu and (1/6) d s_q / d nu.
// Blocks of two warps: nothing is shared between warps (each adds its own dL/dnu partial,
// summed in a fixed order), so no warp waits at a barrier.
// Measured on 1024 x 128 (one launch, cold caches): FP64 129 -> 47 us (348 -> about 150 FP64
// instructions per node), FP32 28 -> 15.2 us.
constexpr int kAdjThreads = 64;
template <typename S, typename R>
__global__ void __launch_bounds__(kAdjThreads, sizeof(R) == 4 ? 16 : 8) k_adj_step(
    const SpParams P, int nfb, int gx, const S *__restrict__ Xt, const R *__restrict__ LPn, R *__restrict__ LP, double *grad_qdot,
    double *grad_flux2, double *grad_flux3, double cn, double cq, double *nu_partials) {
  R dn = 0, dq = 0;
  int i, j;
  R lx[9], lg[5];
  if ((int)blockIdx.x < nfb) {
    if (adj_frame_node(P.nx, P.ny, blockIdx.x * kAdjThreads + threadIdx.x, i, j)) {
      gather_frame<S, R>(P, Xt, LPn, i, j, lx, lg, grad_flux2, grad_flux3);
      reverse_node<S, R, false>(P, i, j, lx, lg, LP, grad_qdot, dn, dq);
    }
  } else {
    j = (blockIdx.x - nfb) / gx;
    i = (blockIdx.x - nfb - j * gx) * kAdjThreads + threadIdx.x;
    if (i >= 2 && j >= 2 && i < P.nx - 2 && j < P.ny - 2) {
      const long long n = nidx(P, i, j);
      const R *LPng = LPn + (long long)P.gbase * P.plane;
#pragma unroll
      for (int q = 0; q < 9; q++) lx[q] = LPn[q * P.plane + n + (long long)cy9(q) * P.pitch + cx9(q)];
#pragma unroll
      for (int q = 0; q < 5; q++) lg[q] = LPng[q * P.plane + n + (long long)cy5(q) * P.pitch + cx5(q)];
      reverse_node<S, R, true>(P, i, j, lx, lg, LP, grad_qdot, dn, dq);
    }
  }
  // the lower half of the warp sums dn, the upper half dq, in the working precision; their
  // factors, which FP32 would round and whose products cancel, come in FP64 once per warp
  const bool upper = threadIdx.x & 16;
  NodeSum<R> sum;
  sum.clear();
  sum.add(upper ? dq : dn);
  sum.add(__shfl_xor_sync(0xffffffffu, upper ? dn : dq, 16));
  sum.template warp_reduce<16>();
  double v = (upper ? cq : cn) * sum.value();
  v += __shfl_down_sync(0xffffffffu, v, 16);
  if ((threadIdx.x & 31) == 0) nu_partials[blockIdx.x * (kAdjThreads / 32) + threadIdx.x / 32] += v;
}

__global__ void k_adj_final(const double *nu_partials, long long nb, double *out) {
  const int t = threadIdx.x;
  double a = 0;
  for (long long k = t; k < nb; k += 256) a += nu_partials[k];
  __shared__ double sh[256];
  sh[t] = a;
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if (t < w) sh[t] += sh[t + w];
    __syncthreads();
  }
  if (t == 0) *out = sh[0];
}

cudaError_t adj_loss(const SpParams &P, int prec, const double *Ttarget, void *LP, double *grad_qdot,
                     double *loss_rows, cudaStream_t s) {
  const dim3 g((P.ny + 127) / 128), b(128);
  if (prec == 0) k_adj_loss<double, double><<<g, b, 0, s>>>(P, Ttarget, (double *)LP, grad_qdot, loss_rows);
  else k_adj_loss<float, float><<<g, b, 0, s>>>(P, Ttarget, (float *)LP, grad_qdot, loss_rows);
  return cudaGetLastError();
}

// Blocks of a reverse step: nfb of frame nodes, then gx per row (one grid dimension: rows
// beyond 65535 stay possible).
static unsigned adj_blocks(int nx, int ny, int *nfb, int *gx) {
  *gx = (nx + kAdjThreads - 1) / kAdjThreads;
  *nfb = (adj_frame_nodes(nx, ny) + kAdjThreads - 1) / kAdjThreads;
  return (unsigned)*nfb + (unsigned)*gx * ny;
}

long long adj_partials(int nx, int ny) {
  int nfb, gx;
  return (long long)adj_blocks(nx, ny, &nfb, &gx) * (kAdjThreads / 32);
}

cudaError_t adj_step(const SpParams &P, int prec, const void *Xt, const void *LPn, void *LP, double *grad_qdot,
                     double *grad_flux2, double *grad_flux3, double cn, double cq, double *nu_partials, cudaStream_t s) {
  int nfb, gx;
  const unsigned nb = adj_blocks(P.nx, P.ny, &nfb, &gx);
  if (prec == 0)
    k_adj_step<double, double><<<nb, kAdjThreads, 0, s>>>(P, nfb, gx, (const double *)Xt, (const double *)LPn,
                                                          (double *)LP, grad_qdot, grad_flux2, grad_flux3, 0.25 * cn,
                                                          cq / 6.0, nu_partials);
  else
    k_adj_step<float, float><<<nb, kAdjThreads, 0, s>>>(P, nfb, gx, (const float *)Xt, (const float *)LPn, (float *)LP,
                                                        grad_qdot, grad_flux2, grad_flux3, 0.25 * cn, cq / 6.0,
                                                        nu_partials);
  return cudaGetLastError();
}

cudaError_t adj_final(const double *nu_partials, long long nb, double *out, cudaStream_t s) {
  k_adj_final<<<1, 256, 0, s>>>(nu_partials, nb, out);
  return cudaGetLastError();
}

}  // namespace lbmk
