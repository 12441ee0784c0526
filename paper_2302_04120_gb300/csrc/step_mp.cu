// Two-phase kernels: conservative Allen-Cahn h_i (D2Q5, BGK) coupled to the
// pressure-evolution z_i (D2Q9, MRT or BGK) of the model described in Sec. 2.3
// of Martins, Alvarino & Cabezas-Gomez (arXiv:2302.04120), all in SI units.
//
// A step is ONE launch (k_mp_collide) over 32 x 8 tiles:
//   * pull h_i for the tile and for a one-node halo ring (periodic, or beyond a
//     resting wall the mirror image of the boundary node) and stage
//     phi = sum h_i (Eq. zero_moment_h) in shared memory (the node's own h stay
//     in registers; halo h re-reads hit L2, so DRAM sees each h once);
//   * isotropic gradient and Laplacian (Eqs. gradient, laplacian, D2Q9 weights),
//     chemical potential (Eq. chemical_potential), guarded normal, F_s = mu grad
//     phi, grad rho; pull z_i; recover u (Eq. u_Liang) and p (Eq. p_Liang);
//   * collide h (Eqs. eq_lattice_boltzmann_interface, heq_liang,
//     source_term_interface) and z (Eq. colisao_MRT with the multiphase
//     [Lambda]_dim of Sec. 3, Eqs. zeq_liang, s_i_Liang,
//     forcing_term_pressure_evolution); store h*, z* and phi u for the next
//     explicit d_t(phi u).
// The collisions work on pairs of opposite populations (as in sp_device.cuh): the FP64
// form is bound by GB300's FP64 pipe, so its time is the number of FP64 instructions per
// node; lengths, dt and c are folded into host-filled constants.
// In the FP32 form the populations and (phi u) are stored in FP32 and the
// collision runs in FP32, while rho(phi), u and p are recovered in pairs of floats
// (hi + lo, about 48 bits) across the interface and in the gas (phi < 0.999): at the
// ~43000 density ratio of saturated water u = j / rho divides by rho_g = 0.023.  In the
// liquid bulk FP32 resolves them.  The pairs run on the FP32 pipe; the same recovery in
// FP64 (about 60 instructions of 16 cycles a warp) held whole tiles of the gas on the
// FP64 pipe.  Results are rounded to FP32 either way.
// Measured before and after pairs of populations, float pairs and the narrow blocks: FP32
// 512^2 bubble 12.9 -> 10.7 us per step, 4096^2 435 -> 390 us, error against a 64-bit
// solution after 100 steps 6.6e-6 -> 3.5e-6; FP64 10 x 400 layered flow 15.9 -> 9.5 us.
#include <cuda_runtime.h>

#include "compensated.cuh"
#include "lattice.cuh"
#include "lbm_mp.cuh"
#include "reciprocal.cuh"

namespace lbmk {

namespace {

// Tiles are 32 nodes wide and BY = 8 rows high, or 2 rows on grids too small to give
// every SM several 32 x 8 tiles (the FP64 collision is then spread over more SMs).
// Grids of at most kNarrow columns (layered flow between plates, uniform along x) take
// one-warp blocks of whole rows (BY = 0): a warp holds 32 / nx rows instead of 32 / nx
// warps each nx lanes, and the halo is the two rows beside the block.
constexpr int BX = 32;
constexpr int kSmallGridBlocks = 608;  // 4 x 152 SMs: fewer 32 x 8 tiles take BY = 2
constexpr int kNarrow = 16;
constexpr int kNarrowTile = 104;       // (rows + 2) (nx + 2), rows = 32 / nx, nx = 1..kNarrow

__device__ __forceinline__ int wrapi(int a, int n) { return a < 0 ? a + n : (a >= n ? a - n : a); }
__device__ __forceinline__ int modi(int a, int n) { int r = a % n; return r < 0 ? r + n : r; }

// Source of the pull of population q (velocity (cx, cy), opposite o) at node (i, j):
// the upstream node, wrapped on a periodic axis; on a walled axis a link whose
// upstream node lies beyond the wall is the node's own opposite population
// (half-way bounce-back at a resting wall).  Returns the element offset.
__device__ __forceinline__ long long pull_src(const MpParams &P, int q, int o, int cx, int cy, int i, int j) {
  if (P.local) return q * P.plane + (long long)j * P.pitch + i;
  const int si = i - cx, sj = j - cy;
  const bool out = (P.xwall && (si < 0 || si >= P.nx)) || (P.ywall && (sj < 0 || sj >= P.ny));
  if (out) return o * P.plane + (long long)j * P.pitch + i;
  return q * P.plane + (long long)wrapi(sj, P.ny) * P.pitch + wrapi(si, P.nx);
}

// Node whose phi stands at stencil position a along an axis of n nodes: wrapped on a
// periodic axis; on a walled axis the mirror image of the boundary node for the one
// layer beyond the wall (further positions are never read by a live node).
__device__ __forceinline__ int stencil_node(int a, int n, int wall) {
  if (wall) return a < 0 ? 0 : (a >= n ? n - 1 : a);
  return a < 0 || a >= n ? modi(a, n) : a;
}

template <typename S, typename R>
__device__ __forceinline__ void pull_h(const MpParams &P, const S *src, int i, int j, R h[5]) {
  const S *hs = src + 9ll * P.plane;
#pragma unroll
  for (int q = 0; q < 5; q++) h[q] = (R)hs[pull_src(P, q, opp5(q), cx5(q), cy5(q), i, j)];
}

// The same pulls for a node whose sources cannot wrap (blocks away from the grid's
// periodic seams): sn points at the node in plane 0; every plane offset is uniform.
template <typename S, typename R>
__device__ __forceinline__ void pull_h_at(const MpParams &P, const S *sn, R h[5]) {
  const S *hs = sn + 9ll * P.plane;
#pragma unroll
  for (int q = 0; q < 5; q++) h[q] = (R)hs[q * P.plane - (long long)cy5(q) * P.pitch - cx5(q)];
}

template <typename S, typename R>
__device__ __forceinline__ void pull_z_at(const MpParams &P, const S *sn, R z[9]) {
#pragma unroll
  for (int q = 0; q < 9; q++) z[q] = (R)sn[q * P.plane - (long long)cy9(q) * P.pitch - cx9(q)];
}

template <typename S, typename R>
__device__ __forceinline__ void pull_z(const MpParams &P, const S *src, int i, int j, R z[9]) {
#pragma unroll
  for (int q = 0; q < 9; q++) z[q] = (R)src[pull_src(P, q, opp9(q), cx9(q), cy9(q), i, j)];
}

// Macroscopic state of a node in the working precision.  h = u / c; j = rho h; rx, ry are
// 36 / (3 / dx) grad phi; the half force H = dt F / (2 c) and U = (dt / 2) u . grad rho are
// what the collision needs of F and grad rho; Pp = p / c_s^2.
template <typename R>
struct MpMacro {
  R phi, rx, ry, rn, Hx, Hy, snu;  // snu = dt / tau
  R rho, hx, hy, jx, jy, ru, U, Pp;
};

// Liquid nodes with phi above this use the working-precision recovery of rho, u, p;
// all others (the interface, its tanh tails and the gas) recover in float pairs.
constexpr float kPhiFineBelow = 0.999f;

// Sums of floats with the rounding errors carried along, s + e.
struct Pair {
  float s, e;
  __device__ __forceinline__ void add(float x) {
    float r;
    two_sum(s, x, s, r);
    e += r;
  }
  // exact product added
  __device__ __forceinline__ void add_product(float a, float b) {
    const float p = __fmul_rn(a, b);  // (not contracted into the sum)
    e += fmaf(a, b, -p);
    add(p);
  }
  __device__ __forceinline__ void renorm() {
    float r;
    two_sum(s, e, s, r);
    e = r;
  }
};

// rho, u and p of Eqs. u_Liang and p_Liang (u first).  jz and znz: lattice-scaled first
// moment and sum of z_1..8.
__device__ __forceinline__ void recover(const MpParams &P, const double z[9], MpMacro<double> &m, double Gx, double Gy) {
  const MpConst<double> &K = P.kd;
  const double tx = (z[5] - z[7]) - (z[6] - z[8]), ty = (z[5] - z[7]) + (z[6] - z[8]);
  m.rho = K.rho_g + m.phi * K.drl;
  const double inv = rcp(m.rho);
  m.jx = ((z[1] - z[3]) + tx) + m.Hx;
  m.jy = ((z[2] - z[4]) + ty) + m.Hy;
  m.hx = m.jx * inv;
  m.hy = m.jy * inv;
  m.ru = m.jx * m.hx + m.jy * m.hy;
  m.U = m.hx * Gx + m.hy * Gy;
  const double znz = ((z[1] + z[3]) + (z[2] + z[4])) + ((z[5] + z[7]) + (z[6] + z[8]));
  m.Pp = 1.8 * ((znz + m.U) - (2.0 / 3.0) * m.ru);
}

__device__ __forceinline__ void recover(const MpParams &P, const float z[9], MpMacro<float> &m, float Gx, float Gy) {
  const MpConst<float> &K = P.kf;
  if (m.phi < kPhiFineBelow) {
    Pair jx = {z[1], 0.0f}, jy = {z[2], 0.0f}, n = {z[1], 0.0f}, rho = {K.rho_g, K.rho_g_lo};
    jx.add(-z[3]); jx.add(z[5]); jx.add(-z[7]); jx.add(-z[6]); jx.add(z[8]); jx.add(m.Hx);
    jy.add(-z[4]); jy.add(z[5]); jy.add(-z[7]); jy.add(z[6]); jy.add(-z[8]); jy.add(m.Hy);
    n.add(z[3]); n.add(z[2]); n.add(z[4]); n.add(z[5]); n.add(z[7]); n.add(z[6]); n.add(z[8]);
    rho.add_product(m.phi, K.drl);
    rho.e = fmaf(m.phi, K.drl_lo, rho.e);
    jx.renorm();
    jy.renorm();
    rho.renorm();
    float inv = rcp(rho.s);
    inv = fmaf(inv, fmaf(-rho.s, inv, 1.0f), inv);
    // h = j / rho: quotient of the leading parts and its remainder
    Pair hx = {__fmul_rn(jx.s, inv), 0.0f}, hy = {__fmul_rn(jy.s, inv), 0.0f};
    hx.e = inv * (fmaf(-hx.s, rho.s, jx.s) + fmaf(-hx.s, rho.e, jx.e));
    hy.e = inv * (fmaf(-hy.s, rho.s, jy.s) + fmaf(-hy.s, rho.e, jy.e));
    hx.renorm();
    hy.renorm();
    Pair ru = {0.0f, 0.0f}, U = {0.0f, 0.0f};
    ru.add_product(jx.s, hx.s);
    ru.add_product(jy.s, hy.s);
    ru.e += jx.s * hx.e + jx.e * hx.s + jy.s * hy.e + jy.e * hy.s;
    U.add_product(hx.s, Gx);
    U.add_product(hy.s, Gy);
    U.e += hx.e * Gx + hy.e * Gy;
    ru.renorm();
    U.renorm();
    // znz + U - (2/3) ru, then 1.8 times that, the constants as hi + lo
    constexpr float k23 = (float)(2.0 / 3.0), k23l = (float)(2.0 / 3.0 - (double)k23);
    constexpr float k18 = 1.8f, k18l = (float)(1.8 - (double)k18);
    n.add(U.s);
    n.add_product(ru.s, -k23);
    n.e += U.e - (ru.e * k23 + ru.s * k23l);
    n.renorm();
    m.rho = rho.s;
    m.jx = jx.s;
    m.jy = jy.s;
    m.hx = hx.s;
    m.hy = hy.s;
    m.ru = ru.s;
    m.U = U.s;
    m.Pp = fmaf(k18, n.s, fmaf(k18, n.e, k18l * n.s));
    return;
  }
  // liquid (rho within 0.1 % of rho_l): the working precision resolves u and p
  const float tx = (z[5] - z[7]) - (z[6] - z[8]), ty = (z[5] - z[7]) + (z[6] - z[8]);
  m.rho = K.rho_g + m.phi * K.drl;
  const float inv = rcp(m.rho);
  m.jx = ((z[1] - z[3]) + tx) + m.Hx;
  m.jy = ((z[2] - z[4]) + ty) + m.Hy;
  m.hx = m.jx * inv;
  m.hy = m.jy * inv;
  m.ru = m.jx * m.hx + m.jy * m.hy;
  m.U = m.hx * Gx + m.hy * Gy;
  const float znz = ((z[1] + z[3]) + (z[2] + z[4])) + ((z[5] + z[7]) + (z[6] + z[8]));
  m.Pp = 1.8f * ((znz + m.U) - (float)(2.0 / 3.0) * m.ru);
}

// Gradient and Laplacian of phi from the shared tile (t: the node's entry, ld: row
// stride), then the half force, tau, rho, u and p.
template <typename R>
__device__ __forceinline__ void mp_macro(const MpParams &P, const R *t, int ld, const R z[9], R fext_x, R fext_y,
                                         MpMacro<R> &m) {
  const MpConst<R> &K = KM<R>(P);
  const R pc = t[0];
  const R pE = t[1], pW = t[-1], pN = t[ld], pS = t[-ld];
  const R pNE = t[ld + 1], pNW = t[ld - 1], pSW = t[-ld - 1], pSE = t[-ld + 1];
  m.phi = pc;
  // Eq. gradient: sum_i w_i c_i phi_i / (c_s^2 dt) = (3/dx) sum_i w_i e_i phi_i, here 36 sum
  const R da = pNE - pSW, db = pNW - pSE;
  m.rx = (R)4 * (pE - pW) + (da - db);
  m.ry = (R)4 * (pN - pS) + (da + db);
  // Eq. laplacian: (6/dx^2) sum_i w_i (phi_i - phi), here 36 sum
  const R l36 = (R)4 * ((pE + pW) + (pN + pS) - (R)4 * pc) + ((pNE + pSW) + (pNW + pSE) - (R)4 * pc);
  // dt / (2 c) F of Eq. chemical_potential: F = mu grad phi + F_b
  const R hmu = K.kb * pc * ((pc - (R)1) * (pc - (R)0.5)) - K.kl * l36;
  m.Hx = hmu * m.rx;
  m.Hy = hmu * m.ry;
  if (P.forced) {
    m.Hx += K.hdt_ic * (K.Fx + fext_x);
    m.Hy += K.hdt_ic * (K.Fy + fext_y);
  }
  // 1 / (36 / (3 / dx) |grad phi|), 0 where the gradient vanishes
  m.rn = inv_norm(m.rx * m.rx + m.ry * m.ry);
  recover(P, z, m, K.kg * m.rx, K.kg * m.ry);
  // tau / dt = nu / (c_s^2 dt) + 1/2 (Eq. eq_kinematic_viscosity)
  const R tau = P.nu_rule == 0 ? K.tau0 + pc * K.dtau : (K.zg + pc * K.dzeta) * rcp(m.rho) + (R)0.5;
  m.snu = rcp(tau);
}

template <typename R>
__device__ __forceinline__ void collide_h(const MpParams &P, const MpMacro<R> &m, R dpux, R dpuy, R h[5]) {
  const MpConst<R> &K = KM<R>(P);
  const R d13 = h[1] - h[3], d24 = h[2] - h[4], a13 = h[1] + h[3], a24 = h[2] + h[4];
  // pairs (Eqs. heq_liang, source_term_interface): even ones relax to phi / 6, odd ones to
  // phi h / 2, with the source of d_t(phi u) and of the interface flux
  // (c_s^2 4 phi (1 - phi) / W) n
  const R p6 = m.phi * ((R)1 / (R)6), flux = K.s2 * (m.phi * ((R)1 - m.phi)) * m.rn;
  const R px = K.om_h * (p6 - (R)0.5 * a13), py = K.om_h * (p6 - (R)0.5 * a24);
  const R ox = K.hom_h * (m.phi * m.hx - d13) + K.s1 * dpux + flux * m.rx;
  const R oy = K.hom_h * (m.phi * m.hy - d24) + K.s1 * dpuy + flux * m.ry;
  // the rest population takes the remainder: sum h stays phi in the working precision
  h[0] -= (R)2 * (px + py);
  h[1] += px + ox;
  h[3] += px - ox;
  h[2] += py + oy;
  h[4] += py - oy;
}

template <typename R>
__device__ __forceinline__ void collide_z(const MpParams &P, const MpMacro<R> &m, R z[9]) {
  const MpConst<R> &K = KM<R>(P);
  // u . grad rho terms: rho_grad holds dt c grad rho
  const R gx = (R)2 * K.kg * m.rx, gy = (R)2 * K.kg * m.ry;
  if (!P.z_mrt) {
    // BGK, Eq. eq_lattice_boltzmann_pressure (lattice-scaled)
    const R om = m.snu, sfac = (R)1 - (R)0.5 * m.snu;
    const R hu = (R)1.5 * m.ru;
#pragma unroll
    for (int q = 0; q < 9; q++) {
      const R ch = (R)cx9(q) * m.hx + (R)cy9(q) * m.hy, cj = (R)cx9(q) * m.jx + (R)cy9(q) * m.jy;
      const R si = w9<R>(q) * (cj * ((R)3 + (R)4.5 * ch) - hu);                 // rho s_i(u)
      const R zeq = m.Pp * (w9<R>(q) - (q == 0 ? (R)1 : (R)0)) + si;            // Eq. zeq_liang
      const R Fz = w9<R>(q) * ((R)6 * ((R)cx9(q) * m.Hx + (R)cy9(q) * m.Hy) +
                               (R)3 * ch * ((R)cx9(q) * gx + (R)cy9(q) * gy));  // dt F^z_i
      z[q] = z[q] - om * (z[q] - zeq) + sfac * Fz;
    }
    return;
  }
  // MRT, multiphase [Lambda]_dim (Sec. 3): rate 1/dt everywhere except omega_q2 (q_x, and
  // q_y by the isotropic reading) and 1/tau for the stress moments; omega_q2 dt = 3 (2 -
  // omega_nu dt) / (3 - omega_nu dt).  At rate 1 a moment goes to its equilibrium plus half
  // its forcing: sum z' = U, e' = 3 ru + 2 Pp, eps' = -3 ru - 3 Pp - U, j' = j + H.  So the
  // even pairs keep only the stress of z and the odd ones only q.
  const R d13 = z[1] - z[3], d24 = z[2] - z[4], d57 = z[5] - z[7], d68 = z[6] - z[8];
  const R xx = (z[1] + z[3]) - (z[2] + z[4]), xy = (z[5] + z[7]) - (z[6] + z[8]);
  const R snu = m.snu, sq = ((R)6 - (R)3 * snu) * rcp((R)3 - snu);
  const R sqy = P.qy_literal ? (R)1 : sq;
  const R r3 = m.ru * ((R)1 / (R)12), p36 = m.Pp * ((R)1 / (R)36), u12 = m.U * ((R)1 / (R)12);
  const R e4 = (R)2 * u12 + (r3 + (R)4 * p36), e8 = u12 + (r3 + p36);
  const R xx0 = m.jx * m.hx, rxx = xx0 - m.jy * m.hy, rxy = m.jx * m.hy;
  const R f3 = ((R)1 - (R)0.5 * snu) * ((R)1 / (R)3);
  const R gxx = m.hx * gx, Fxx = (R)2 * (gxx - m.hy * gy), Fxy = m.hx * gy + m.hy * gx;
  const R X = (R)0.25 * (xx + snu * (rxx - xx) + f3 * Fxx), Y = (R)0.25 * (xy + snu * (rxy - xy) + f3 * Fxy);
  const R qx = ((d57 - d68) - (R)2 * d13), qy = ((d57 + d68) - (R)2 * d24);
  const R jx = m.jx + m.Hx, jy = m.jy + m.Hy;
  const R qxn = qx - (sq * (qx + m.jx) + ((R)2 - sq) * m.Hx), qyn = qy - (sqy * (qy + m.jy) + ((R)2 - sqy) * m.Hy);
  const R Qx = (jx - qxn) * ((R)1 / (R)6), Qy = (jy - qyn) * ((R)1 / (R)6);
  const R bx = (R)0.5 * jx - Qx, by = (R)0.5 * jy - Qy;
  const R w = (R)0.5 * (bx + by), v = (R)0.5 * (by - bx);
  const R P13 = e4 + X, P24 = e4 - X, P57 = e8 + Y, P68 = e8 - Y;
  z[0] = m.U - (R)4 * (e4 + e8);
  z[1] = P13 + Qx;
  z[3] = P13 - Qx;
  z[2] = P24 + Qy;
  z[4] = P24 - Qy;
  z[5] = P57 + w;
  z[7] = P57 - w;
  z[6] = P68 + v;
  z[8] = P68 - v;
}

enum { MODE_STEP = 0, MODE_MOMENTS = 2, MODE_INTEGRALS = 3 };

__device__ __forceinline__ void reduce4_block(double v[4], double *out) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    v[0] += __shfl_down_sync(0xffffffffu, v[0], o);
    v[1] += __shfl_down_sync(0xffffffffu, v[1], o);
    v[2] = fmax(v[2], __shfl_down_sync(0xffffffffu, v[2], o));
    v[3] += __shfl_down_sync(0xffffffffu, v[3], o);
  }
  __shared__ double sh[8][4];
  const int tid = threadIdx.y * blockDim.x + threadIdx.x, nw = (blockDim.x * blockDim.y) / 32;
  if ((tid & 31) == 0) { sh[tid >> 5][0] = v[0]; sh[tid >> 5][1] = v[1]; sh[tid >> 5][2] = v[2]; sh[tid >> 5][3] = v[3]; }
  __syncthreads();
  if (tid == 0) {
    double a = 0, b = 0, mx = 0, cnt = 0;
    for (int w = 0; w < nw; w++) { a += sh[w][0]; b += sh[w][1]; mx = fmax(mx, sh[w][2]); cnt += sh[w][3]; }
    out[0] = a; out[1] = b; out[2] = mx; out[3] = cnt;
  }
}

// Resident 32 x 8 blocks per SM asked of the compiler for the FP32 form: 5 caps it
// at 48 registers (the unbounded build takes 56, i.e. 4 blocks), more warps to cover
// the HBM latency of the pulls.
#ifndef LBM_MP_FP32_BLOCKS_PER_SM
#define LBM_MP_FP32_BLOCKS_PER_SM 5
#endif

template <int BY> constexpr int mp_threads() { return BY ? BX * BY : 32; }

// One step (and its moments / integrals variants).  BY = 0: one-warp blocks of whole rows
// (narrow grids).
template <int PREC, int MODE, int BY>
__global__ void __launch_bounds__(mp_threads<BY>(), (PREC == 1 && BY == 8) ? LBM_MP_FP32_BLOCKS_PER_SM : 0)
k_mp_collide(const MpParams P, unsigned mask, double *out) {
  typedef typename Prec<PREC>::S S;
  typedef typename Prec<PREC>::R R;
  __shared__ R tile[BY ? (BY + 2) * (BX + 2) : kNarrowTile];
  const S *src = (const S *)P.src;
  int i, j, ld, at;  // node, row stride of the tile, the node's entry in it
  bool live, inner = false;
  // phi = sum_i h_i (Eq. zero_moment_h) of the tile and of a one-node halo, from pulled h:
  // this node's h stays in registers for its collision.  The node's z, (phi u)_prev and
  // force do not depend on the tile: their loads are issued before the barrier
  R h[5], z[9];
  R prevx = 0, prevy = 0, fex = 0, fey = 0;
  auto load_node = [&](long long n) {
    if (P.force) {
      fex = (R)((const S *)P.force)[n];
      fey = (R)((const S *)P.force)[P.plane + n];
    }
    if (inner) pull_z_at<S, R>(P, src + n, z);
    else pull_z<S, R>(P, src, i, j, z);
    if (MODE == MODE_STEP) {
      prevx = (R)src[14ll * P.plane + n];
      prevy = (R)src[15ll * P.plane + n];
    }
  };
  auto sum5 = [](const R *a) { return (a[0] + a[1]) + (a[2] + a[3]) + a[4]; };
  if (BY == 0) {
    const int nx = P.nx, rows = 32 / nx, j0 = blockIdx.x * rows, r = min(rows, P.ny - j0);
    const int ty = threadIdx.x / nx;
    ld = nx + 2;
    i = threadIdx.x - ty * nx;
    j = j0 + ty;
    at = (ty + 1) * ld + i + 1;
    live = ty < r;
    // an entry and, for the first and last column, its image beside the row
    auto put = [&](int row, int col, R phi) {
      tile[row * ld + col + 1] = phi;
      if (col == 0) tile[row * ld + (P.xwall ? 0 : nx + 1)] = phi;
      if (col == nx - 1) tile[row * ld + (P.xwall ? nx + 1 : 0)] = phi;
    };
    if (live) {
      pull_h<S, R>(P, src, i, j, h);
      load_node((long long)j * P.pitch + i);
      put(ty + 1, i, sum5(h));
    }
    for (int t = threadIdx.x; t < 2 * nx; t += 32) {  // the rows below and above the block
      const int up = t >= nx, col = up ? t - nx : t;
      R hh[5];
      pull_h<S, R>(P, src, col, stencil_node(up ? j0 + r : j0 - 1, P.ny, P.ywall), hh);
      put(up ? r + 1 : 0, col, sum5(hh));
    }
  } else {
    const int i0 = blockIdx.x * BX, j0 = blockIdx.y * BY;
    const int tid = threadIdx.y * BX + threadIdx.x;
    i = i0 + threadIdx.x;
    j = j0 + threadIdx.y;
    ld = BX + 2;
    at = (threadIdx.y + 1) * (BX + 2) + threadIdx.x + 1;
    live = (i < P.nx) && (j < P.ny);
    // a block whose tile, halo and their pull sources stay off the periodic seams
    // (the bulk of the grid) pulls with plain offsets: no wrap, no modulo
    inner = !P.local && i0 >= 2 && j0 >= 2 && i0 + BX + 2 <= P.nx && j0 + BY + 2 <= P.ny;
    if (inner) pull_h_at<S, R>(P, src + ((long long)j * P.pitch + i), h);
    else pull_h<S, R>(P, src, stencil_node(i, P.nx, P.xwall), stencil_node(j, P.ny, P.ywall), h);
    if (live) load_node((long long)j * P.pitch + i);
    tile[at] = sum5(h);
    constexpr int kHalo = 2 * (BX + 2) + 2 * BY;
    for (int t = tid; t < kHalo; t += BX * BY) {
      int tx, ty;
      if (t < BX + 2) { tx = t; ty = 0; }                            // row below the tile
      else if (t < 2 * (BX + 2)) { tx = t - (BX + 2); ty = BY + 1; }  // row above
      else if (t < 2 * (BX + 2) + BY) { tx = 0; ty = t - 2 * (BX + 2) + 1; }  // left column
      else { tx = BX + 1; ty = t - 2 * (BX + 2) - BY + 1; }           // right column
      R hh[5];
      if (inner) {
        pull_h_at<S, R>(P, src + ((long long)(j0 + ty - 1) * P.pitch + (i0 + tx - 1)), hh);
      } else {
        pull_h<S, R>(P, src, stencil_node(i0 + tx - 1, P.nx, P.xwall), stencil_node(j0 + ty - 1, P.ny, P.ywall), hh);
      }
      tile[ty * (BX + 2) + tx] = sum5(hh);
    }
  }
  __syncthreads();
  double red[4] = {0.0, 0.0, 0.0, 0.0};
  if (live) {
    const long long n = (long long)j * P.pitch + i;
    MpMacro<R> m;
    mp_macro<R>(P, tile + at, BY ? BX + 2 : ld, z, fex, fey, m);
    if (MODE == MODE_STEP) {
      const R pux = m.phi * (KM<R>(P).c * m.hx), puy = m.phi * (KM<R>(P).c * m.hy);
      collide_h<R>(P, m, pux - prevx, puy - prevy, h);  // explicit Euler d_t(phi u)
      collide_z<R>(P, m, z);
      S *dst = (S *)P.dst;
#pragma unroll
      for (int q = 0; q < 9; q++) dst[q * P.plane + n] = (S)z[q];
#pragma unroll
      for (int q = 0; q < 5; q++) dst[(9 + q) * P.plane + n] = (S)h[q];
      dst[14ll * P.plane + n] = (S)pux;
      dst[15ll * P.plane + n] = (S)puy;
    } else if (MODE == MODE_MOMENTS) {
      const long long N = (long long)P.nx * P.ny, k = (long long)j * P.nx + i;
      int slot = 0;
      if (mask & 1u) out[(slot++) * N + k] = (double)m.rho;
      if (mask & 2u) out[(slot++) * N + k] = P.c * (double)m.hx;
      if (mask & 4u) out[(slot++) * N + k] = P.c * (double)m.hy;
      if (mask & 8u) out[(slot++) * N + k] = 0.0;
      if (mask & 16u) out[(slot++) * N + k] = P.cs2 * (double)m.Pp;
      if (mask & 32u) out[(slot++) * N + k] = (double)m.phi;
    } else {
      const double ux = P.c * (double)m.hx, uy = P.c * (double)m.hy, rho = (double)m.rho, pr = (double)m.Pp;
      const double umag = sqrt(ux * ux + uy * uy);
      const bool bad = !isfinite(rho) || !isfinite(umag) || !isfinite(pr) || umag >= P.c;
      // a bad node (non-finite, or |u| >= c) is counted and adds nothing else
      red[0] = bad ? 0.0 : rho * P.dx * P.dx;
      red[1] = bad ? 0.0 : (double)m.phi;
      red[2] = bad ? 0.0 : umag;
      red[3] = bad ? 1.0 : 0.0;
    }
  }
  if (MODE == MODE_INTEGRALS) reduce4_block(red, out + 4ll * (blockIdx.y * gridDim.x + blockIdx.x));
}

__global__ void k_mp_final(const double *partials, int nb, double *out5, const double *flag) {
  const int lane = threadIdx.x;
  double v[4] = {0.0, 0.0, 0.0, 0.0};
  for (int b = lane; b < nb; b += 32) {
    v[0] += partials[4 * b + 0];
    v[1] += partials[4 * b + 1];
    v[2] = fmax(v[2], partials[4 * b + 2]);
    v[3] += partials[4 * b + 3];
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    v[0] += __shfl_down_sync(0xffffffffu, v[0], o);
    v[1] += __shfl_down_sync(0xffffffffu, v[1], o);
    v[2] = fmax(v[2], __shfl_down_sync(0xffffffffu, v[2], o));
    v[3] += __shfl_down_sync(0xffffffffu, v[3], o);
  }
  if (lane == 0) { out5[0] = v[0]; out5[1] = v[1]; out5[2] = v[2]; out5[3] = v[3]; out5[4] = *flag; }
}

// Equilibria of the given fields (Eqs. heq_liang, zeq_liang, s_i_Liang) as the
// pre-collision state of time 0; (phi u)_prev = phi0 u0.  Defaults: phi 1, u 0, p 0.
template <typename S>
__global__ void k_mp_init(const MpParams P, const double *A, const double *UX, const double *UY, const double *B) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int j = blockIdx.y * blockDim.y + threadIdx.y;
  if (i >= P.nx || j >= P.ny) return;
  const long long n = (long long)j * P.pitch + i;
  const int k = j * P.nx + i;
  S *dst = (S *)P.dst;
  // FP64 in both forms, on pairs of opposite populations (no division per node: with one
  // per population and term, initialising a 4096 x 4096 grid took as long as 23 steps)
  const double ph = A ? A[k] : 1.0, u0 = UX ? UX[k] : 0.0, v0 = UY ? UY[k] : 0.0;
  const double hx = u0 * P.inv_c, hy = v0 * P.inv_c;
  const double rho = P.rho_g + ph * (P.rho_l - P.rho_g), Pp = B ? B[k] * (3.0 * P.inv_c * P.inv_c) : 0.0;
  const double jx = rho * hx, jy = rho * hy, xx0 = jx * hx, ru = xx0 + jy * hy;
  const double X = 0.25 * (xx0 - jy * hy), Y = 0.25 * (jx * hy), r12 = ru * (1.0 / 12.0);
  const double e4 = Pp * (1.0 / 9.0) + r12, e8 = Pp * (1.0 / 36.0) + r12;
  const double qx = jx * (1.0 / 3.0), qy = jy * (1.0 / 3.0), w = 0.25 * (qx + qy), v = 0.25 * (qy - qx);
  const double p6 = ph * (1.0 / 6.0), ox = 0.5 * (ph * hx), oy = 0.5 * (ph * hy);
  auto put = [&](int q, double a) { dst[q * P.plane + n] = (S)a; };
  put(0, -4.0 * (e4 + e8));
  put(1, (e4 + X) + qx);
  put(3, (e4 + X) - qx);
  put(2, (e4 - X) + qy);
  put(4, (e4 - X) - qy);
  put(5, (e8 + Y) + w);
  put(7, (e8 + Y) - w);
  put(6, (e8 - Y) + v);
  put(8, (e8 - Y) - v);
  put(9, ph - 4.0 * p6);
  put(10, p6 + ox);
  put(12, p6 - ox);
  put(11, p6 + oy);
  put(13, p6 - oy);
  put(14, ph * u0);
  put(15, ph * v0);
}

// Blocks of a launch: rows BY of a tile by size, 0 (whole rows) on narrow grids.
dim3 mp_grid(int nx, int ny, int by) {
  if (by == 0) return dim3((ny + 32 / nx - 1) / (32 / nx));
  return dim3((nx + BX - 1) / BX, (ny + by - 1) / by);
}
int mp_rows(int nx, int ny) {
  if (nx <= kNarrow) return 0;
  return (int)(mp_grid(nx, ny, 8).x * mp_grid(nx, ny, 8).y) >= kSmallGridBlocks ? 8 : 2;
}

template <int PREC, int MODE>
void launch_collide(const MpParams &P, unsigned mask, double *out, cudaStream_t s) {
  const int by = mp_rows(P.nx, P.ny);
  const dim3 g = mp_grid(P.nx, P.ny, by);
  if (by == 8) k_mp_collide<PREC, MODE, 8><<<g, dim3(BX, 8), 0, s>>>(P, mask, out);
  else if (by == 2) k_mp_collide<PREC, MODE, 2><<<g, dim3(BX, 2), 0, s>>>(P, mask, out);
  else k_mp_collide<PREC, MODE, 0><<<g, 32, 0, s>>>(P, mask, out);
}

}  // namespace

int mp_integral_blocks(int nx, int ny) {
  dim3 g = mp_grid(nx, ny, mp_rows(nx, ny));
  return (int)(g.x * g.y);
}

cudaError_t mp_step(const MpParams &P, int prec, cudaStream_t s) {
  if (prec == 0) launch_collide<0, MODE_STEP>(P, 0u, nullptr, s);
  else launch_collide<1, MODE_STEP>(P, 0u, nullptr, s);
  return cudaGetLastError();
}

cudaError_t mp_init(const MpParams &P, int prec, const double *phi0, const double *ux0, const double *uy0,
                    const double *p0, cudaStream_t s) {
  dim3 b(BX, 8), g = mp_grid(P.nx, P.ny, 8);
  if (prec == 0) k_mp_init<double><<<g, b, 0, s>>>(P, phi0, ux0, uy0, p0);
  else k_mp_init<float><<<g, b, 0, s>>>(P, phi0, ux0, uy0, p0);
  return cudaGetLastError();
}

cudaError_t mp_moments(const MpParams &P, int prec, unsigned mask, double *out, cudaStream_t s) {
  if (prec == 0) launch_collide<0, MODE_MOMENTS>(P, mask, out, s);
  else launch_collide<1, MODE_MOMENTS>(P, mask, out, s);
  return cudaGetLastError();
}

cudaError_t mp_integrals(const MpParams &P, int prec, double *partials, int max_blocks, double *out5, const double *flag,
                         cudaStream_t s) {
  const int nb = mp_integral_blocks(P.nx, P.ny);
  if (nb > max_blocks) return cudaErrorInvalidValue;
  if (prec == 0) launch_collide<0, MODE_INTEGRALS>(P, 0u, partials, s);
  else launch_collide<1, MODE_INTEGRALS>(P, 0u, partials, s);
  k_mp_final<<<1, 32, 0, s>>>(partials, nb, out5, flag);
  return cudaGetLastError();
}

}  // namespace lbmk
