// Discrete adjoint of the FP32 rollout: gradients of a loss on the recorded trajectory with
// respect to each env's hydrodynamic coefficients (added mass, linear and quadratic damping
// diagonals of Eq. 1) and to the buffered throttle actions (Eq. 3).
//
// The forward pass (k_rollout_fwd) writes the state after every sub-step and the full state every
// C sub-steps.  The backward kernels, one env per lane: for each checkpoint segment, last first,
// the segment's sub-steps are re-run from the checkpoint, then walked in reverse, applying the
// transpose Jacobian of one sub-step
//     s+ = N(s + h/6 (k1 + 2 k2 + 2 k3 + k4)),  N = quaternion renormalisation,
// through N, the RK4 combination and the four right-hand-side evaluations (reverse mode of
// rhs(), written out below).  It is the adjoint of the discrete map the forward computes, so it
// matches finite differences of the rollout itself, not of the continuous equations.
//
// The throttle lag is linear with the command held (LagEnv): with d = n - c the step gives n+ = n +
// g d, and the later stages' throttles are n+ + h_i d.  So with e_i the adjoint of stage i's
// throttle through the thrust, n+ has mu = lambda_n + e_2 + e_3 + e_4, d has delta = g mu + sum h_i
// e_i, the throttle's own adjoint goes lambda_n <- mu + delta + e_1 and the command's gains -delta;
// the throttles stay out of the stage combinations.
//
// Parameter paths, as the forward has:
//   - diagonal mass (r_g = 0, no off-diagonal extension): rhs_vjp_diag, the transpose of the step's
//     own coefficient form (StepDiag, or StepMirrored with its thrust sums);
//   - general (GEN): rhs_vjp_gen, off-centre gravity (the m r_g coupling of M_RB and C_RB,
//     off-diagonal I_o) and the off-diagonal added mass and linear damping of the extension record
//     (zeros when the fleet has none), with the full M^-1.
// A diagonal coefficient theta = M_A,jj enters M = M_RB + M_A, so nu' = M^-1 f gets d nu'/d theta =
// -M^-1 e_j nu'_j, whose contribution to the gradient is -(M^-1 g)_j nu'_j for the loss adjoint g
// of nu' (M^-1 is symmetric).  nu' itself comes recorded with the stage states.
#include <type_traits>

#include "mg_advance.cuh"

namespace mg {

namespace {

constexpr int kAdjThreads = 128;

// Which transpose a kernel is compiled for.
enum AdjPath {
  ADJ_GEN = 0, ADJ_GEN_MIRRORED = 1, ADJ_DENSE = 2, ADJ_MIRRORED = 3, ADJ_MIRRORED_G = 4
};
__host__ __device__ constexpr bool adj_general(int path) { return path <= ADJ_GEN_MIRRORED; }

// The thruster allocation of the re-run: the forward's (the vectored one only skips exact zeros of
// the dense one), so the states are the forward's bit for bit.
__host__ __device__ constexpr int adj_layout(int path) {
  return path == ADJ_MIRRORED || path == ADJ_GEN_MIRRORED ? MG_LAYOUT_MIRRORED
         : path == ADJ_MIRRORED_G                         ? MG_LAYOUT_MIRRORED_G
                                                          : MG_LAYOUT_DENSE;
}

// Sums over stages and sub-steps that the coefficient gradients are formed from at the end.
// General path: the gradients themselves (mv: M_A,jj through M^-1).
struct GradGen {
  float ma[3], J[3], mv[6], dl[6], dq[6];
};
// Diagonal mass, with g the loss adjoint of nu' (trans/rotational rows i, i1 = i+1, i2 = i+2 mod
// 3):
//   dl, dq   sum g_j x_j, sum g_j |x_j| x_j         (x = r, w)
//   own      sum g_i (w_i2 c_i1 - w_i1 c_i2), c = v - r the current seen from the body
//   up, dn   sum g_i w_i2 r_i1, sum g_i w_i1 r_i2
//   munk     sum g_3+i r_i1 r_i2;  gyro  sum g_3+i w_i1 w_i2;  mv  sum g_j nu'_j
struct GradDiag {
  float dl[6], dq[6], own[3], up[3], dn[3], munk[3], gyro[3], mv[6];
};
template <int PATH>
using Grad = typename std::conditional<adj_general(PATH), GradGen, GradDiag>::type;

template <typename G>
__device__ __forceinline__ void zero_grad(G &g) {
  float *f = reinterpret_cast<float *>(&g);
#pragma unroll
  for (int i = 0; i < (int)(sizeof(G) / sizeof(float)); ++i) f[i] = 0.f;
}

// What the adjoint reads for one env: the coefficients the forward step used and, on the general
// path, the env's off-diagonal hydrodynamic coefficients (a row of MG_NXPARAM floats in shared
// memory).
template <int PATH>
struct AdjEnv {
  Coef<!adj_general(PATH), adj_layout(PATH)> F;
  LagEnv L;
  const float *xh;
};

// Off-diagonal entries of the extension record (layout of mg.h): M_A above its diagonal
// (01 02 03 04 05 12 13 14 15 23 24 25 34 35 45, mirrored below), then D_l's off-diagonal
// entries row by row (5 per row).
__device__ __forceinline__ float xa(const float *xh, int i, int j) {
  const int a = i < j ? i : j, b = i < j ? j : i;
  return xh[5 * a - a * (a - 1) / 2 + (b - a - 1)];
}
__device__ __forceinline__ float xd(const float *xh, int i, int j) {
  return xh[15 + 5 * i + (j < i ? j : j - 1)];
}

// Every multiply-add of the adjoint code below, and of the right-hand side it re-runs, is written
// as an explicit fmaf, and a product that only a plain addition follows as __fmul_rn, so the
// compiler forms no fused operation of its own: the results do not depend on the surrounding code
// the functions are inlined into (the one-warp and two-warp backward kernels agree bit for bit; so
// does this file compiled without contraction).

__device__ __forceinline__ void cross_vjp(const float a[3], const float b[3], const float gc[3],
                                          float ga[3], float gb[3]) {
  // c = a x b:  ga += b x gc,  gb += gc x a.
  ga[0] = fmaf(b[1], gc[2], fmaf(-b[2], gc[1], ga[0]));
  ga[1] = fmaf(b[2], gc[0], fmaf(-b[0], gc[2], ga[1]));
  ga[2] = fmaf(b[0], gc[1], fmaf(-b[1], gc[0], ga[2]));
  gb[0] = fmaf(gc[1], a[2], fmaf(-gc[2], a[1], gb[0]));
  gb[1] = fmaf(gc[2], a[0], fmaf(-gc[0], a[2], gb[1]));
  gb[2] = fmaf(gc[0], a[1], fmaf(-gc[1], a[0], gb[2]));
}

// Packed symmetric M^-1 (general path) times x.
__device__ __forceinline__ void minv_apply(const ParGen &P, const float x[6], float y[6]) {
  const float *o = P.mo;  // 01 02 03 04 05 12 13 14 15 23 24 25 34 35 45
  y[0] = fmaf(P.mi[0], x[0], fmaf(o[0], x[1], fmaf(o[1], x[2], fmaf(o[2], x[3],
         fmaf(o[3], x[4], o[4] * x[5])))));
  y[1] = fmaf(o[0], x[0], fmaf(P.mi[1], x[1], fmaf(o[5], x[2], fmaf(o[6], x[3],
         fmaf(o[7], x[4], o[8] * x[5])))));
  y[2] = fmaf(o[1], x[0], fmaf(o[5], x[1], fmaf(P.mi[2], x[2], fmaf(o[9], x[3],
         fmaf(o[10], x[4], o[11] * x[5])))));
  y[3] = fmaf(o[2], x[0], fmaf(o[6], x[1], fmaf(o[9], x[2], fmaf(P.mi[3], x[3],
         fmaf(o[12], x[4], o[13] * x[5])))));
  y[4] = fmaf(o[3], x[0], fmaf(o[7], x[1], fmaf(o[10], x[2], fmaf(o[12], x[3],
         fmaf(P.mi[4], x[4], o[14] * x[5])))));
  y[5] = fmaf(o[4], x[0], fmaf(o[8], x[1], fmaf(o[11], x[2], fmaf(o[13], x[3],
         fmaf(o[14], x[4], P.mi[5] * x[5])))));
}

// A rigid-body quantity of the transposes: the pose's and velocity's parts of a state adjoint.
struct Body {
  float p[3], q[4], v[3], w[3];
};

// gs = (d rhs / d s)^T gd for the pose and velocity of stage state s, with en[i] the adjoint of the
// stage throttle n_i through the thrust and the coefficient sums accumulated into G; nud is the
// stage's recorded nu'.  The forward quantities are recomputed from Eq. 1 in the general path's
// Kirchhoff form; gd.q is the adjoint of d.q = q (x) (0, w) (the doubled quaternion rate rhs()
// stores).
template <int MT, int PATH>
__device__ void rhs_vjp_gen(const St<MT> &s, const float (&nud)[6], const AdjEnv<PATH> &A,
                            const float4 *gdir, const float4 *garm, int nt, bool current_accel,
                            const Body &gd, Body &gs, GradGen &G, float (&en)[MT]) {
  const auto &P = A.F;
  const float *xh = A.xh;
  // ---------------- forward recomputation
  const float qw = s.q[0], qx = s.q[1], qy = s.q[2], qz = s.q[3];
  float R[3][3];
  R[0][0] = fmaf(-2.f, fmaf(qy, qy, qz * qz), 1.f);
  R[0][1] = 2.f * fmaf(qx, qy, -qw * qz);
  R[0][2] = 2.f * fmaf(qx, qz, qw * qy);
  R[1][0] = 2.f * fmaf(qx, qy, qw * qz);
  R[1][1] = fmaf(-2.f, fmaf(qx, qx, qz * qz), 1.f);
  R[1][2] = 2.f * fmaf(qy, qz, -qw * qx);
  R[2][0] = 2.f * fmaf(qx, qz, -qw * qy);
  R[2][1] = 2.f * fmaf(qy, qz, qw * qx);
  R[2][2] = fmaf(-2.f, fmaf(qx, qx, qy * qy), 1.f);
  const float v[3] = {s.v[0], s.v[1], s.v[2]}, w[3] = {s.w[0], s.w[1], s.w[2]};
  const float vc[3] = {P.vc0, P.vc1, P.vc2}, ma[3] = {P.ma0, P.ma1, P.ma2};
  const float J[3] = {P.J0, P.J1, P.J2}, G3[3] = {P.G0, P.G1, P.G2};
  float cb[3], r[3], qm[3], h[3], k[3], c[3] = {0.f, 0.f, 0.f}, am[3] = {0.f, 0.f, 0.f};
  const float mrg[3] = {P.mrg0, P.mrg1, P.mrg2};
  for (int i = 0; i < 3; ++i)
    cb[i] = fmaf(R[2][i], vc[2], fmaf(R[1][i], vc[1], R[0][i] * vc[0]));
  for (int i = 0; i < 3; ++i) {
    r[i] = v[i] - cb[i];
    qm[i] = ma[i] * r[i];
    k[i] = J[i] * w[i];
  }
  const float nur[6] = {r[0], r[1], r[2], w[0], w[1], w[2]};
  // off-diagonal added mass in the momenta; w x m r_g; off-diagonal I_o w + m r_g x v
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 6; ++j) {
      if (j != i) qm[i] = fmaf(xa(xh, i, j), nur[j], qm[i]);
      if (j != 3 + i) k[i] = fmaf(xa(xh, 3 + i, j), nur[j], k[i]);
    }
  am[0] = fmaf(w[1], mrg[2], -w[2] * mrg[1]);
  am[1] = fmaf(w[2], mrg[0], -w[0] * mrg[2]);
  am[2] = fmaf(w[0], mrg[1], -w[1] * mrg[0]);
  k[0] = fmaf(P.Ixy, w[1], fmaf(P.Ixz, w[2], fmaf(mrg[1], v[2], fmaf(-mrg[2], v[1], k[0]))));
  k[1] = fmaf(P.Ixy, w[0], fmaf(P.Iyz, w[2], fmaf(mrg[2], v[0], fmaf(-mrg[0], v[2], k[1]))));
  k[2] = fmaf(P.Ixz, w[0], fmaf(P.Iyz, w[1], fmaf(mrg[0], v[1], fmaf(-mrg[1], v[0], k[2]))));
  for (int i = 0; i < 3; ++i) h[i] = fmaf(P.m, v[i], qm[i]) + am[i];
  if (current_accel) {
    c[0] = fmaf(w[1], cb[2], -w[2] * cb[1]);
    c[1] = fmaf(w[2], cb[0], -w[0] * cb[2]);
    c[2] = fmaf(w[0], cb[1], -w[1] * cb[0]);
  }
  const float e[3] = {R[2][0], R[2][1], R[2][2]};

  // ---------------- reverse
  // nu' = M^-1 f: gf = M^-1 g (symmetric), and M_jj's share -gf_j nu'_j
  const float gnu[6] = {gd.v[0], gd.v[1], gd.v[2], gd.w[0], gd.w[1], gd.w[2]};
  float gf[6], gt[6];
  minv_apply(P, gnu, gf);
  for (int j = 0; j < 6; ++j) {
    G.mv[j] = fmaf(-gf[j], nud[j], G.mv[j]);
    gt[j] = P.kT * gf[j];
  }
  float gw[3] = {0.f, 0.f, 0.f}, gv[3] = {0.f, 0.f, 0.f}, gr[3] = {0.f, 0.f, 0.f};
  float gh[3] = {0.f, 0.f, 0.f}, gk[3] = {0.f, 0.f, 0.f}, gqm[3] = {0.f, 0.f, 0.f};
  float gcb[3] = {0.f, 0.f, 0.f}, ge[3] = {0.f, 0.f, 0.f}, gc[3] = {0.f, 0.f, 0.f};
  float gam[3] = {0.f, 0.f, 0.f}, gnur[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  // off-diagonal current term and linear damping
#pragma unroll
  for (int i = 0; i < 6; ++i)
#pragma unroll
    for (int j = 0; j < 6; ++j) {
      if (j < 3 && j != i) gc[j] = fmaf(-xa(xh, i, j), gf[i], gc[j]);
      if (j != i) gnur[j] = fmaf(-xd(xh, i, j), gf[i], gnur[j]);
    }
  // rotational force
  const float gfr[3] = {gf[3], gf[4], gf[5]};
  const float ngfr[3] = {-gf[3], -gf[4], -gf[5]};
  cross_vjp(r, qm, ngfr, gr, gqm);   // - r x Q1
  cross_vjp(w, k, ngfr, gw, gk);     // - w x k
  cross_vjp(v, am, ngfr, gv, gam);  // - v x (w x m r_g)
  for (int j = 0; j < 3; ++j) {
    const float aw = fabsf(w[j]);
    gw[j] = fmaf(-fmaf(2.f * P.dq[3 + j], aw, P.dl[3 + j]), gfr[j], gw[j]);
    G.dl[3 + j] = fmaf(-w[j], gfr[j], G.dl[3 + j]);
    G.dq[3 + j] = fmaf(-aw * w[j], gfr[j], G.dq[3 + j]);
  }
  {
    float gG[3] = {0.f, 0.f, 0.f};
    cross_vjp(G3, e, gfr, gG, ge);   // + G x e
  }
  // translational force
  const float gfl[3] = {gf[0], gf[1], gf[2]};
  const float ngfl[3] = {-gf[0], -gf[1], -gf[2]};
  for (int j = 0; j < 3; ++j) ge[j] = fmaf(P.wb, gfl[j], ge[j]);
  cross_vjp(w, h, ngfl, gw, gh);     // - w x h
  for (int j = 0; j < 3; ++j) {
    const float ar = fabsf(r[j]);
    gr[j] = fmaf(-fmaf(2.f * P.dq[j], ar, P.dl[j]), gfl[j], gr[j]);
    G.dl[j] = fmaf(-r[j], gfl[j], G.dl[j]);
    G.dq[j] = fmaf(-ar * r[j], gfl[j], G.dq[j]);
  }
  if (current_accel) {
    for (int j = 0; j < 3; ++j) {
      G.ma[j] = fmaf(-c[j], gfl[j], G.ma[j]);
      gc[j] = fmaf(-ma[j], gfl[j], gc[j]);
    }
    cross_vjp(w, cb, gc, gw, gcb);   // c = w x v_c^b
  }
  // k += off-diagonal I_o w + m r_g x v;  h += w x m r_g
  gw[0] = fmaf(P.Ixy, gk[1], fmaf(P.Ixz, gk[2], gw[0]));
  gw[1] = fmaf(P.Ixy, gk[0], fmaf(P.Iyz, gk[2], gw[1]));
  gw[2] = fmaf(P.Ixz, gk[0], fmaf(P.Iyz, gk[1], gw[2]));
  gv[0] = fmaf(gk[1], mrg[2], fmaf(-gk[2], mrg[1], gv[0]));
  gv[1] = fmaf(gk[2], mrg[0], fmaf(-gk[0], mrg[2], gv[1]));
  gv[2] = fmaf(gk[0], mrg[1], fmaf(-gk[1], mrg[0], gv[2]));
  for (int j = 0; j < 3; ++j) gam[j] += gh[j];
  float gmrg[3] = {0.f, 0.f, 0.f};
  cross_vjp(w, mrg, gam, gw, gmrg);
  // off-diagonal added mass in the momenta (Q1 enters through h and through r x Q1)
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 6; ++j) {
      if (j != i) gnur[j] = fmaf(xa(xh, i, j), gqm[i] + gh[i], gnur[j]);
      if (j != 3 + i) gnur[j] = fmaf(xa(xh, 3 + i, j), gk[i], gnur[j]);
    }
  // k = J w, h = m v + Q1, Q1 = M_A r, r = v - v_c^b
  for (int j = 0; j < 3; ++j) {
    gw[j] = fmaf(J[j], gk[j], gw[j]);
    G.J[j] = fmaf(w[j], gk[j], G.J[j]);
    gv[j] = fmaf(P.m, gh[j], gv[j]);
    gqm[j] += gh[j];
    gr[j] = fmaf(ma[j], gqm[j], gr[j]);
    G.ma[j] = fmaf(r[j], gqm[j], G.ma[j]);
    gr[j] += gnur[j];
    gw[j] += gnur[3 + j];
    gv[j] += gr[j];
    gcb[j] -= gr[j];
  }
  // R entries: v_c^b = R^T v_c, e = third row of R, p' = R v
  float gR[3][3];
  for (int i = 0; i < 3; ++i)
    for (int j = 0; j < 3; ++j) gR[i][j] = fmaf(vc[i], gcb[j], gd.p[i] * v[j]);
  for (int j = 0; j < 3; ++j) {
    gR[2][j] += ge[j];
    gv[j] = fmaf(R[0][j], gd.p[0], fmaf(R[1][j], gd.p[1], fmaf(R[2][j], gd.p[2], gv[j])));
  }
  // d.q = q (x) (0, w)
  const float g0 = gd.q[0], g1 = gd.q[1], g2 = gd.q[2], g3 = gd.q[3];
  gw[0] = fmaf(-qx, g0, fmaf(qw, g1, fmaf(qz, g2, fmaf(-qy, g3, gw[0]))));
  gw[1] = fmaf(-qy, g0, fmaf(-qz, g1, fmaf(qw, g2, fmaf(qx, g3, gw[1]))));
  gw[2] = fmaf(-qz, g0, fmaf(qy, g1, fmaf(-qx, g2, fmaf(qw, g3, gw[2]))));
  float gq[4];
  gq[0] = fmaf(w[0], g1, fmaf(w[1], g2, w[2] * g3));
  gq[1] = fmaf(-w[0], g0, fmaf(-w[2], g2, w[1] * g3));
  gq[2] = fmaf(-w[1], g0, fmaf(w[2], g1, -w[0] * g3));
  gq[3] = fmaf(-w[2], g0, fmaf(-w[1], g1, w[0] * g2));
  // R(q) -> q
  {
    const float s0 = fmaf(-qz, gR[0][1], fmaf(qz, gR[1][0], fmaf(qy, gR[0][2],
                     fmaf(-qy, gR[2][0], fmaf(-qx, gR[1][2], qx * gR[2][1])))));
    const float s1 = fmaf(qy, gR[0][1], fmaf(qy, gR[1][0], fmaf(qz, gR[0][2],
                     fmaf(qz, gR[2][0], fmaf(-qw, gR[1][2], qw * gR[2][1])))));
    const float s2 = fmaf(qx, gR[0][1], fmaf(qx, gR[1][0], fmaf(qw, gR[0][2],
                     fmaf(-qw, gR[2][0], fmaf(qz, gR[1][2], qz * gR[2][1])))));
    const float s3 = fmaf(-qw, gR[0][1], fmaf(qw, gR[1][0], fmaf(qx, gR[0][2],
                     fmaf(qx, gR[2][0], fmaf(qy, gR[1][2], qy * gR[2][1])))));
    gq[0] = fmaf(2.f, s0, gq[0]);
    gq[1] = fmaf(2.f, s1, fmaf(-4.f * qx, gR[1][1] + gR[2][2], gq[1]));
    gq[2] = fmaf(2.f, s2, fmaf(-4.f * qy, gR[0][0] + gR[2][2], gq[2]));
    gq[3] = fmaf(2.f, s3, fmaf(-4.f * qz, gR[0][0] + gR[1][1], gq[3]));
  }
  // thrust: t = sum_i n_i|n_i| b_i
#pragma unroll
  for (int i = 0; i < MT; ++i) {
    en[i] = 0.f;
    if (i >= nt) continue;
    const float4 dd = gdir[i], aa = garm[i];
    const float gfi = fmaf(dd.x, gt[0], fmaf(dd.y, gt[1], fmaf(dd.z, gt[2],
                      fmaf(aa.x, gt[3], fmaf(aa.y, gt[4], aa.z * gt[5])))));
    en[i] = __fmul_rn(2.f * fabsf(s.n[i]), gfi);
  }
  for (int i = 0; i < 4; ++i) gs.q[i] = gq[i];
  for (int i = 0; i < 3; ++i) {
    gs.v[i] = gv[i];
    gs.w[i] = gw[i];
  }
}

// The transpose of the diagonal-mass right-hand side (rhs with StepDiag or StepMirrored): gs = (d
// rhs / d s)^T gd for the pose and velocity, en[i] the adjoint of the stage throttle n_i through
// the thrust, the sums of GradDiag accumulated.  With u_i = v_i1 + bp_i r_i1, x_i = v_i2 + bm_i
// r_i2 the rows are v'_i = ... + w_i2 u_i - w_i1 x_i - (dlt_i + dqt_i |r_i|) r_i and w'_i = ... +
// B_i r_i1 r_i2 + C_i w_i1 w_i2 - (dlr_i + dqr_i |w_i|) w_i.  About 290 operations a stage where
// the general path's form of the same transpose (which this path used before) takes some 700: the
// consumer warp of the two-warp kernel, a chain of these, is what bounds a small fleet's backward
// pass: 4,096 envs x 200 sub-steps 918 -> 330 us together with the re-run's single evaluation of
// each sub-step and the 16-byte records (ncu: 2,390 instead of 4,580 instructions a sub-step in the
// two warps).
template <int MT, int PATH>
__device__ __forceinline__ void rhs_vjp_diag(const St<MT> &s, const float (&nud)[6],
                                             const AdjEnv<PATH> &A, const float4 *gdir,
                                             const float4 *garm, int nt, const Body &gd, Body &gs,
                                             GradDiag &G, float (&en)[MT]) {
  const auto &P = A.F;
  const float qw = s.q[0], qx = s.q[1], qy = s.q[2], qz = s.q[3];
  float R[3][3];
  {
    const float tx = qx + qx, ty = qy + qy, tz = qz + qz;
    const float zd = fmaf(-qz, tz, 1.f), xy = qx * ty, xz = qx * tz, yz = qy * tz;
    R[0][0] = fmaf(-qy, ty, zd);
    R[1][1] = fmaf(-qx, tx, zd);
    R[2][2] = fmaf(-qx, tx, fmaf(-qy, ty, 1.f));
    R[0][1] = fmaf(-qw, tz, xy);
    R[1][0] = fmaf(qw, tz, xy);
    R[0][2] = fmaf(qw, ty, xz);
    R[2][0] = fmaf(-qw, ty, xz);
    R[1][2] = fmaf(-qw, tx, yz);
    R[2][1] = fmaf(qw, tx, yz);
  }
  const float v[3] = {s.v[0], s.v[1], s.v[2]}, w[3] = {s.w[0], s.w[1], s.w[2]};
  const float vc[3] = {P.vc0, P.vc1, P.vc2};
  const float gv[3] = {gd.v[0], gd.v[1], gd.v[2]}, gw[3] = {gd.w[0], gd.w[1], gd.w[2]};
  float cb[3], r[3], gr[3], ov[3], ow[3] = {0.f, 0.f, 0.f};  // ov, ow: adjoints of v, w
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    cb[j] = fmaf(R[2][j], vc[2], fmaf(R[1][j], vc[1], R[0][j] * vc[0]));
    r[j] = v[j] - cb[j];
  }
  // damping
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    const float ar = fabsf(r[j]), aw = fabsf(w[j]);
    const float hr = gv[j] * r[j], hw = gw[j] * w[j];
    G.dl[j] = fmaf(gv[j], r[j], G.dl[j]);
    G.dl[3 + j] = fmaf(gw[j], w[j], G.dl[3 + j]);
    G.dq[j] = fmaf(ar, hr, G.dq[j]);
    G.dq[3 + j] = fmaf(aw, hw, G.dq[3 + j]);
    gr[j] = -fmaf(P.dqt[j], ar + ar, P.dlt[j]) * gv[j];
    ow[j] = -fmaf(P.dqr[j], aw + aw, P.dlr[j]) * gw[j];
    G.mv[j] = fmaf(gv[j], nud[j], G.mv[j]);
    G.mv[3 + j] = fmaf(gw[j], nud[3 + j], G.mv[3 + j]);
    ov[j] = 0.f;
  }
  // translational Coriolis terms, Munk and gyroscopic products
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const int i1 = (i + 1) % 3, i2 = (i + 2) % 3;
    const float u = fmaf(P.bp[i], r[i1], v[i1]), x = fmaf(P.bm[i], r[i2], v[i2]);
    const float gu = gv[i] * w[i2], gx = gv[i] * w[i1];  // adjoints of u_i and -x_i
    ow[i2] = fmaf(gv[i], u, ow[i2]);
    ow[i1] = fmaf(-gv[i], x, ow[i1]);
    ov[i1] = fmaf(gv[i], w[i2], ov[i1]);
    ov[i2] = fmaf(-gv[i], w[i1], ov[i2]);
    gr[i1] = fmaf(P.bp[i], gu, gr[i1]);
    gr[i2] = fmaf(-P.bm[i], gx, gr[i2]);
    G.up[i] = fmaf(gu, r[i1], G.up[i]);
    G.dn[i] = fmaf(gx, r[i2], G.dn[i]);
    G.own[i] = fmaf(gu, cb[i1], fmaf(-gx, cb[i2], G.own[i]));
    const float gm = gw[i] * r[i1], gg = gw[i] * w[i1];
    G.munk[i] = fmaf(gm, r[i2], G.munk[i]);
    G.gyro[i] = fmaf(gg, w[i2], G.gyro[i]);
    gr[i2] = fmaf(P.B[i], gm, gr[i2]);
    gr[i1] = fmaf(P.B[i] * gw[i], r[i2], gr[i1]);
    ow[i2] = fmaf(P.C[i], gg, ow[i2]);
    ow[i1] = fmaf(P.C[i] * gw[i], w[i2], ow[i1]);
  }
  // R: p' = R v, r = v - R^T v_c, (W - B) k_e and G x k_e with k_e the third row
  float gR[3][3];
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) gR[i][j] = fmaf(-vc[i], gr[j], gd.p[i] * v[j]);
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    gR[2][j] = fmaf(P.Wt[j], gv[j], gR[2][j]);
    ov[j] += gr[j];
    gs.v[j] = fmaf(R[0][j], gd.p[0], fmaf(R[1][j], gd.p[1], fmaf(R[2][j], gd.p[2], ov[j])));
  }
  if constexpr (mirrored_sums(adj_layout(PATH))) {
    gR[2][1] = fmaf(-P.Gr, gw[0], gR[2][1]);
    gR[2][0] = fmaf(P.Gp, gw[1], gR[2][0]);
    if constexpr (PATH == ADJ_MIRRORED_G) {
      gR[2][0] = fmaf(-P.Gyy, gw[2], gR[2][0]);
      gR[2][1] = fmaf(P.Gyx, gw[2], gR[2][1]);
      gR[2][2] = fmaf(P.Gry, gw[0], fmaf(-P.Gpx, gw[1], gR[2][2]));
    }
  } else {
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const int i1 = (i + 1) % 3, i2 = (i + 2) % 3;
      gR[2][i2] = fmaf(P.Gp[i], gw[i], gR[2][i2]);
      gR[2][i1] = fmaf(-P.Gm[i], gw[i], gR[2][i1]);
    }
  }
  // d.q = q (x) (0, w)
  const float g0 = gd.q[0], g1 = gd.q[1], g2 = gd.q[2], g3 = gd.q[3];
  gs.w[0] = fmaf(-qx, g0, fmaf(qw, g1, fmaf(qz, g2, fmaf(-qy, g3, ow[0]))));
  gs.w[1] = fmaf(-qy, g0, fmaf(-qz, g1, fmaf(qw, g2, fmaf(qx, g3, ow[1]))));
  gs.w[2] = fmaf(-qz, g0, fmaf(qy, g1, fmaf(-qx, g2, fmaf(qw, g3, ow[2]))));
  // R(q) -> q: the antisymmetric and symmetric parts of gR
  {
    const float a0 = gR[2][1] - gR[1][2], a1 = gR[0][2] - gR[2][0], a2 = gR[1][0] - gR[0][1];
    const float b0 = gR[2][1] + gR[1][2], b1 = gR[0][2] + gR[2][0], b2 = gR[1][0] + gR[0][1];
    const float d0 = gR[1][1] + gR[2][2], d1 = gR[0][0] + gR[2][2], d2 = gR[0][0] + gR[1][1];
    const float m0 = -2.f * d0, m1 = -2.f * d1, m2 = -2.f * d2;
    const float s0 = fmaf(qx, a0, fmaf(qy, a1, qz * a2));
    const float s1 = fmaf(qw, a0, fmaf(qy, b2, fmaf(qz, b1, qx * m0)));
    const float s2 = fmaf(qw, a1, fmaf(qx, b2, fmaf(qz, b0, qy * m1)));
    const float s3 = fmaf(qw, a2, fmaf(qx, b1, fmaf(qy, b0, qz * m2)));
    gs.q[0] = fmaf(2.f, s0, fmaf(w[0], g1, fmaf(w[1], g2, w[2] * g3)));
    gs.q[1] = fmaf(2.f, s1, fmaf(-w[0], g0, fmaf(-w[2], g2, w[1] * g3)));
    gs.q[2] = fmaf(2.f, s2, fmaf(-w[1], g0, fmaf(w[2], g1, -w[0] * g3)));
    gs.q[3] = fmaf(2.f, s3, fmaf(-w[2], g0, fmaf(-w[1], g1, w[0] * g2)));
  }
  // thrust: n|n| of each thruster into the rows
  float gf[MT];
  if constexpr (mirrored_sums(adj_layout(PATH))) {
    const float gX = fmaf(P.At[0], gv[0], P.Mh * gw[1]), gY = fmaf(P.At[1], gv[1], P.Kh * gw[0]);
    const float gZ = P.At[2] * gv[2];
    const float sm = gX + gY, df = gX - gY;
    gf[0] = fmaf(P.Nh, gw[2], sm);
    gf[1] = fmaf(-P.Nh, gw[2], df);
    gf[2] = fmaf(-P.Nh, gw[2], -df);
    gf[3] = fmaf(P.Nh, gw[2], -sm);
    gf[4] = fmaf(-P.Kv, gw[0], gZ);
    gf[5] = fmaf(P.Kv, gw[0], gZ);
    if constexpr (MT > 6) {
      gf[6] = fmaf(P.Mv, gw[1], gf[4]);
      gf[7] = fmaf(P.Mv, gw[1], gf[5]);
      gf[4] = fmaf(-P.Mv, gw[1], gf[4]);
      gf[5] = fmaf(-P.Mv, gw[1], gf[5]);
    }
  } else {
    float gt[6];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      gt[i] = P.At[i] * gv[i];
      gt[3 + i] = P.Ar[i] * gw[i];
    }
#pragma unroll
    for (int i = 0; i < MT; ++i) {
      const float4 dd = gdir[i], aa = garm[i];
      gf[i] = fmaf(dd.x, gt[0], fmaf(dd.y, gt[1], fmaf(dd.z, gt[2],
              fmaf(aa.x, gt[3], fmaf(aa.y, gt[4], aa.z * gt[5])))));
    }
  }
  (void)nt;
#pragma unroll
  for (int i = 0; i < MT; ++i) en[i] = __fmul_rn(2.f * fabsf(s.n[i]), gf[i]);
}

// The stage states of one sub-step and the step itself: stage(i, y, nu') is called with stage i's
// state (the same four states rk4_step evaluates, the throttles in closed form) and its nu'; zq
// receives the quaternion before renormalisation and S the next start state.  The operations are
// rk4_step's.
template <int MT, int PATH, typename Stage>
__device__ __forceinline__ void stage_step(St<MT> &S, const float (&c)[MT], const AdjEnv<PATH> &A,
                                           const float4 *gdir, const float4 *garm, int nt, bool ca,
                                           const RkStep &rk, float (&zq)[4], Stage stage) {
  constexpr bool DIAG = !adj_general(PATH);
  constexpr int NH = adj_layout(PATH);
  St<MT> k, y = S, acc;
  float d[MT];
#pragma unroll
  for (int g = 0; g < 4; ++g) {
    rhs<MT, DIAG, true, NH, !DIAG>(y, A.F, gdir, garm, nt, ca, k, A.xh);
    const float nud[6] = {k.v[0], k.v[1], k.v[2], k.w[0], k.w[1], k.w[2]};
    stage(g, y, nud);
    if (g == 0) axpy<MT>(acc, S, rk.h6, rk.q12, k);
    else if (g < 3) axpy<MT>(acc, acc, rk.h3, rk.h6, k);
    else axpy<MT>(S, acc, rk.h6, rk.q12, k);
    if (g < 2) axpy<MT>(y, S, rk.hh, rk.qh, k);
    else if (g == 2) axpy<MT>(y, S, rk.h, rk.hh, k);
    const float hi = g == 0 ? A.L.h2 : g == 1 ? A.L.h3 : A.L.h4;
#pragma unroll
    for (int i = 0; i < MT; ++i) {
      if (g == 0) {
        d[i] = S.n[i] - c[i];
        S.n[i] = fmaf(A.L.g, d[i], S.n[i]);
      }
      if (g < 3) y.n[i] = fmaf(hi, d[i], S.n[i]);
    }
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) zq[i] = S.q[i];
  const float inv = rsqrtf(fmaf(zq[0], zq[0], fmaf(zq[1], zq[1],
                                fmaf(zq[2], zq[2], zq[3] * zq[3]))));
#pragma unroll
  for (int i = 0; i < 4; ++i) S.q[i] *= inv;
}

// lam (pose, velocity) and lamn (throttles): in, the adjoint of the sub-step's output s+; out, the
// adjoint of its input s; gc receives the command's.  stage(i, y, nu') gives stage i's record.
//   s+ = N(z)
// reverse:  lk4 = h/6 W lz,            ly4 = J(y4)^T lk4
//           lk3 = h/3 W lz + h W ly4,   ly3 = J(y3)^T lk3
//           lk2 = h/3 W lz + h/2 W ly3, ly2 = J(y2)^T lk2
//           lk1 = h/6 W lz + h/2 W ly2, ly1 = J(s)^T lk1
//           ls  = lz + ly4 + ly3 + ly2 + ly1
// (W: the quaternion takes half of each weight, because rhs() stores its rate doubled; p does not
// enter the right-hand side, so its adjoint passes through).  The general path's four stages share
// one rolled loop body, a quarter of the code, which the instruction cache holds (unrolled, 4,096
// envs x 200 sub-steps: 707 -> 1,054 us); the diagonal path's smaller transposes are unrolled (one
// warp per 32 envs 476 -> 451 us, two 307 -> 309; 16,384 envs 629 -> 594, 530 -> 506).
template <int MT, int PATH, typename Stage>
__device__ __forceinline__ void step_vjp(Stage stage, const float (&zq)[4], const AdjEnv<PATH> &A,
                                         const float4 *gdir, const float4 *garm, int nt, bool ca,
                                         const RkStep &rk, Body &lam, float (&lamn)[MT],
                                         Grad<PATH> &G, float (&gc)[MT]) {
  // renormalisation q+ = z_q / |z_q|:  lz_q = (lam_q - q+ (q+ . lam_q)) / |z_q|
  const float inv = rsqrtf(fmaf(zq[0], zq[0], fmaf(zq[1], zq[1],
                                fmaf(zq[2], zq[2], zq[3] * zq[3]))));
  float qn[4], dot = 0.f;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    qn[i] = zq[i] * inv;
    dot = fmaf(qn[i], lam.q[i], dot);
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) lam.q[i] = fmaf(-qn[i], dot, lam.q[i]) * inv;
  const Body lz = lam;
  Body ly{};
#pragma unroll
  for (int i = 0; i < MT; ++i) gc[i] = 0.f;  // sum h_i e_i, until the first stage
  auto transpose = [&](int i) {
    const bool outer = i == 3 || i == 0;
    const float a = outer ? rk.h6 : rk.h3, aq = outer ? rk.q12 : rk.h6;
    const float b = i == 3 ? 0.f : i == 2 ? rk.h : rk.hh, bq = 0.5f * b;
    const float hi = i == 3 ? A.L.h4 : i == 2 ? A.L.h3 : A.L.h2;
    Body lk;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      lk.p[j] = a * lz.p[j];
      lk.v[j] = fmaf(b, ly.v[j], a * lz.v[j]);
      lk.w[j] = fmaf(b, ly.w[j], a * lz.w[j]);
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) lk.q[j] = fmaf(bq, ly.q[j], aq * lz.q[j]);
    St<MT> y;
    float nud[6], en[MT];
    stage(i, y, nud);
    if constexpr (adj_general(PATH))
      rhs_vjp_gen<MT, PATH>(y, nud, A, gdir, garm, nt, ca, lk, ly, G, en);
    else
      rhs_vjp_diag<MT, PATH>(y, nud, A, gdir, garm, nt, lk, ly, G, en);
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      lam.v[j] += ly.v[j];
      lam.w[j] += ly.w[j];
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) lam.q[j] += ly.q[j];
#pragma unroll
    for (int j = 0; j < MT; ++j) {
      if (i > 0) {
        lamn[j] += en[j];
        gc[j] = fmaf(hi, en[j], gc[j]);
      } else {
        const float delta = fmaf(A.L.g, lamn[j], gc[j]);
        lamn[j] = (lamn[j] + delta) + en[j];
        gc[j] = -delta;
      }
    }
  };
  if constexpr (adj_general(PATH)) {
#pragma unroll 1
    for (int i = 3; i >= 0; --i) transpose(i);
  } else {
#pragma unroll
    for (int i = 3; i >= 0; --i) transpose(i);
  }
}

constexpr int kMaxSeg = 32;  // largest checkpoint interval

// The held command along a forward walk over sub-steps (the forward's own schedule).
template <int MT>
struct CommandWalk {
  int64_t seg;
  int32_t left;
  float c[MT];

  __device__ __forceinline__ CommandWalk(const FleetView &fv, int64_t e, int nt, int64_t step0) {
    scheduled_start<MT>(fv, e, nt, step0, c, seg, left);
    prefetch_commands(fv, e, seg);
  }
  __device__ __forceinline__ void next(const FleetView &fv, int64_t e, int nt) {
    if (--left == 0) {
      ++seg;
      left = fv.hold;
      load_commands<MT>(fv, e, seg, nt, c);
      prefetch_commands(fv, e, seg);
    }
  }
};

template <int MT, int PATH>
__device__ __forceinline__ void load_checkpoint(const float *__restrict__ ckpt, int32_t sg,
                                                int64_t n, int64_t e, int nt, St<MT> &S) {
  const float *ck = ckpt + (int64_t)sg * MG_NSTATE * n + e;
  for (int i = 0; i < 3; ++i) S.p[i] = ck[(int64_t)(i)*n];
  for (int i = 0; i < 4; ++i) S.q[i] = ck[(int64_t)(3 + i) * n];
  for (int i = 0; i < 3; ++i) S.v[i] = ck[(int64_t)(7 + i) * n];
  for (int i = 0; i < 3; ++i) S.w[i] = ck[(int64_t)(10 + i) * n];
  for (int i = 0; i < MT; ++i) S.n[i] = ck[(int64_t)(13 + i) * n];
  drop_unused_lag<MT, true, adj_layout(PATH)>(S, nt);
}

// lam += the loss adjoint of the state after sub-step t.
__device__ __forceinline__ void add_traj_adjoint(const float *__restrict__ g, int64_t stride,
                                                 Body &lam) {
  for (int i = 0; i < 3; ++i) lam.p[i] += g[i * stride];
  for (int i = 0; i < 4; ++i) lam.q[i] += g[(3 + i) * stride];
  for (int i = 0; i < 3; ++i) lam.v[i] += g[(7 + i) * stride];
  for (int i = 0; i < 3; ++i) lam.w[i] += g[(10 + i) * stride];
}

// Command adjoints of the sub-steps that share an action segment, summed in registers and added
// to the caller's buffer when the backward walk leaves the segment.
template <int MT>
struct ActionAdjoint {
  int64_t seg;   // the segment being summed
  int64_t left;  // its sub-steps still ahead of the walk
  float g[MT];

  // The walk starts at cursor position t.
  __device__ __forceinline__ ActionAdjoint(const FleetView &fv, int64_t t) {
    seg = t / fv.hold;
    if (seg > fv.n_seg - 1) seg = fv.n_seg - 1;  // the last segment holds for good
    left = t - seg * fv.hold + 1;
#pragma unroll
    for (int i = 0; i < MT; ++i) g[i] = 0.f;
  }
  __device__ __forceinline__ void flush(const FleetView &fv, int64_t e, int nt, float *dact) {
    if (!dact || seg < 0) return;
    float *da = dact + (seg * fv.n + e) * fv.act_w;
#pragma unroll
    for (int i = 0; i < MT; ++i) {
      if (i < nt) da[i] += g[i];
      g[i] = 0.f;
    }
  }
  // One sub-step's command adjoint.
  __device__ __forceinline__ void add(const FleetView &fv, int64_t e, int nt,
                                      const float (&gc)[MT], float *dact) {
#pragma unroll
    for (int i = 0; i < MT; ++i) g[i] += gc[i];
    if (--left == 0) {
      flush(fv, e, nt, dact);
      --seg;
      left = fv.hold;
    }
  }
};

// Coefficient gradients from their sums, in the order M_A, D_l, D_q.  M_A,jj enters the momenta (Q1
// for j < 3, J = diag(I_o) + M_A,rot for j >= 3), the current term and M (mv); D_l and D_q their
// damping terms.
__device__ __forceinline__ void coefficient_gradients(const GradGen &G, const ParamPlanes &,
                                                      int64_t, float *dc) {
  for (int j = 0; j < 3; ++j) {
    dc[j] = G.ma[j] + G.mv[j];
    dc[3 + j] = G.J[j] + G.mv[3 + j];
  }
  for (int j = 0; j < 6; ++j) {
    dc[6 + j] = G.dl[j];
    dc[12 + j] = G.dq[j];
  }
}
// Row k's terms in M_A,i are mi_k times: own_i (k = i), up_k - dn_k' (the neighbours' Coriolis
// terms), the Munk products and, rotational, the gyroscopic products; M's share is -mi sum g nu'.
__device__ __forceinline__ void coefficient_gradients(const GradDiag &G, const ParamPlanes &pa,
                                                      int64_t e, float *dc) {
  const float4 m = ldg4(pa.d7, e);
  const float2 n = __ldg(pa.d8 + e);
  const float mi[6] = {m.x, m.y, m.z, m.w, n.x, n.y};
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const int b = (i + 2) % 3, f = (i + 1) % 3;  // rows in which i is i1, and i2
    float a = mi[i] * (G.own[i] - G.mv[i]);
    a = fmaf(mi[b], G.up[b], a);
    a = fmaf(-mi[f], G.dn[f], a);
    a = fmaf(mi[3 + b], G.munk[b], fmaf(-mi[3 + f], G.munk[f], a));
    dc[i] = a;
    dc[3 + i] = fmaf(mi[3 + b], G.gyro[b], fmaf(-mi[3 + f], G.gyro[f], -mi[3 + i] * G.mv[3 + i]));
  }
#pragma unroll
  for (int j = 0; j < 6; ++j) {
    dc[6 + j] = -mi[j] * G.dl[j];
    dc[12 + j] = -mi[j] * G.dq[j];
  }
}

template <int MT, typename G>
__device__ __forceinline__ void write_gradients(const G &grad, const ParamPlanes &pa,
                                                const Body &lam, const float (&lamn)[MT],
                                                int64_t e, float *__restrict__ dcoef,
                                                float *__restrict__ dstate0) {
  coefficient_gradients(grad, pa, e, dcoef + e * 18);
  if (dstate0) {
    float *o = dstate0 + e * MG_NSTATE;
    for (int i = 0; i < 3; ++i) o[i] = lam.p[i];
    for (int i = 0; i < 4; ++i) o[3 + i] = lam.q[i];
    for (int i = 0; i < 3; ++i) o[7 + i] = lam.v[i];
    for (int i = 0; i < 3; ++i) o[10 + i] = lam.w[i];
    for (int i = 0; i < MG_MAX_THR; ++i) o[13 + i] = i < MT ? lamn[i] : 0.f;
  }
}

__device__ __forceinline__ void stage_geometry(const FleetView &fv,
                                               float4 (*sgeo)[2 * MG_MAX_THR]) {
  for (int i = threadIdx.x; i < fv.n_types * 2 * MG_MAX_THR; i += blockDim.x) {
    const int t = i / (2 * MG_MAX_THR), j = i % (2 * MG_MAX_THR);
    sgeo[t][j] = j < MG_MAX_THR ? fv.geo[t].dir[j] : fv.geo[t].arm[j - MG_MAX_THR];
  }
}

// General path: rows [0, count) of sx receive the off-diagonal coefficients of envs env0, ...,
// or zeros when the fleet has no extension (off-centre gravity only).
__device__ __forceinline__ void stage_xh_or_zero(const FleetView &fv, int64_t env0, int count,
                                                 float *sx) {
  if (fv.xh) {
    stage_xh(fv.xh, fv.n, env0, count, sx);
  } else {
    for (int i = threadIdx.x; i < count * MG_NXPARAM; i += blockDim.x) sx[i] = 0.f;
  }
}

template <int PATH>
__device__ __forceinline__ void load_env(const FleetView &fv, int64_t e, const float *sxh_row,
                                         const float4 *gdir, const float4 *garm, AdjEnv<PATH> &A) {
  constexpr bool DIAG = !adj_general(PATH);
  Par<DIAG> P;
  load_par<DIAG>(fv.pa, e, P);
  A.F = make_coef<DIAG, adj_layout(PATH)>(P, gdir, garm);
  A.L = lag_env(P.itau, fv.dt);
  A.xh = DIAG ? nullptr : sxh_row;
}

// A stage record: what the transposes read of one stage, in float4 words (q, nu, nu', n), so that a
// lane moves it in 16-byte pieces: word w of an env's record is a plane over the envs.
template <int MT>
__host__ __device__ constexpr int stage_words() { return (16 + MT + 3) / 4; }
// A sub-step's: four stages and the quaternion before renormalisation.
template <int MT>
__host__ __device__ constexpr int rec_words() { return 4 * stage_words<MT>() + 1; }

template <int MT>
__device__ __forceinline__ void put_stage(float4 *__restrict__ r, int64_t stride, const St<MT> &y,
                                          const float (&nud)[6]) {
  r[0] = make_float4(y.q[0], y.q[1], y.q[2], y.q[3]);
  r[stride] = make_float4(y.v[0], y.v[1], y.v[2], y.w[0]);
  r[2 * stride] = make_float4(y.w[1], y.w[2], nud[0], nud[1]);
  r[3 * stride] = make_float4(nud[2], nud[3], nud[4], nud[5]);
  r[4 * stride] = make_float4(y.n[0], y.n[1], y.n[2], y.n[3]);
  if constexpr (MT > 6) r[5 * stride] = make_float4(y.n[4], y.n[5], y.n[6], y.n[7]);
  else r[5 * stride] = make_float4(y.n[4], y.n[5], 0.f, 0.f);
}
template <int MT>
__device__ __forceinline__ void get_stage(const float4 *r, int64_t stride, St<MT> &y,
                                          float (&nud)[6]) {
  const float4 a = r[0], b = r[stride], c = r[2 * stride], d = r[3 * stride], f = r[4 * stride];
  const float4 g = r[5 * stride];
  y.q[0] = a.x; y.q[1] = a.y; y.q[2] = a.z; y.q[3] = a.w;
  y.v[0] = b.x; y.v[1] = b.y; y.v[2] = b.z;
  y.w[0] = b.w; y.w[1] = c.x; y.w[2] = c.y;
  nud[0] = c.z; nud[1] = c.w; nud[2] = d.x; nud[3] = d.y; nud[4] = d.z; nud[5] = d.w;
  y.n[0] = f.x; y.n[1] = f.y; y.n[2] = f.z; y.n[3] = f.w; y.n[4] = g.x; y.n[5] = g.y;
  if constexpr (MT > 6) {
    y.n[6] = g.z;
    y.n[7] = g.w;
  }
}

// One thread per env.  ckpt [n_ck][MG_NSTATE][n] (state at sub-steps 0, C, 2C, ...),
// dtraj [T][MG_NTRAJ][n] (loss adjoint of the state after each sub-step).  Outputs: dcoef
// [n][18] (M_A, Dl, Dq diagonals), dact [n_seg][n][w] accumulated, dstate0 [n][21] or null.
// The segment's step-start states are kept in local memory, each sub-step's stages recomputed.
// General path: dynamic shared memory [blockDim.x][MG_NXPARAM] for the block's off-diagonal
// coefficients.
template <int MT, int PATH>
__global__ void __launch_bounds__(kAdjThreads)
    k_adjoint(const FleetView fv, const int32_t *__restrict__ types, const float *__restrict__ ckpt,
              const float *__restrict__ dtraj, int32_t T, int32_t C, int64_t step0,
              float *__restrict__ dcoef, float *__restrict__ dact, float *__restrict__ dstate0) {
  __shared__ float4 sgeo[MG_MAX_TYPES][2 * MG_MAX_THR];
  extern __shared__ float sxh[];
  stage_geometry(fv, sgeo);
  const int64_t env0 = (int64_t)blockIdx.x * blockDim.x;
  if constexpr (adj_general(PATH))
    stage_xh_or_zero(fv, env0, (int)min((int64_t)blockDim.x, fv.n - env0), sxh);
  __syncthreads();
  const int64_t e = env0 + threadIdx.x;
  if (e >= fv.n) return;
  const int type = types[e];
  const float4 *gdir = sgeo[type], *garm = sgeo[type] + MG_MAX_THR;
  const int nt = fv.geo[type].n_thr;
  const bool ca = !(fv.model_flags & MG_MODEL_NO_CURRENT_ACCEL);
  const int64_t n = fv.n;
  AdjEnv<PATH> A;
  load_env<PATH>(fv, e, sxh + threadIdx.x * MG_NXPARAM, gdir, garm, A);

  Grad<PATH> G;
  zero_grad(G);
  Body lam{};
  float lamn[MT];
#pragma unroll
  for (int i = 0; i < MT; ++i) lamn[i] = 0.f;
  St<MT> S[kMaxSeg];
  float4 rec[4 * stage_words<MT>()];
  float gc[MT], zq[4];
  ActionAdjoint<MT> act(fv, step0 + T - 1);

  const int32_t n_ck = (T + C - 1) / C;
  for (int32_t sg = n_ck - 1; sg >= 0; --sg) {
    const int32_t t0 = sg * C, len = min(C, T - t0);
    // re-run the segment from its checkpoint
    load_checkpoint<MT, PATH>(ckpt, sg, n, e, nt, S[0]);
    {
      CommandWalk<MT> cmd(fv, e, nt, step0 + t0);
      St<MT> x = S[0];
      for (int32_t j = 1; j < len; ++j) {
        rk4_step<MT, !adj_general(PATH), true, adj_layout(PATH), adj_general(PATH)>(
            x, cmd.c, A.L, A.F, gdir, garm, nt, ca, fv.rk, A.xh);
        S[j] = x;
        cmd.next(fv, e, nt);
      }
    }
    // walk it backwards
    for (int32_t j = len - 1; j >= 0; --j) {
      const int64_t t = t0 + j;
      add_traj_adjoint(dtraj + t * MG_NTRAJ * n + e, n, lam);
      int64_t cs;
      int32_t cl;
      float c[MT];
      scheduled_start<MT>(fv, e, nt, step0 + t, c, cs, cl);
      St<MT> x = S[j];
      stage_step<MT, PATH>(x, c, A, gdir, garm, nt, ca, fv.rk, zq,
                           [&](int g, const St<MT> &y, const float (&nud)[6]) {
                             put_stage<MT>(rec + g * stage_words<MT>(), 1, y, nud);
                           });
      auto stage = [&](int i, St<MT> &y, float (&nud)[6]) {
        get_stage<MT>(rec + i * stage_words<MT>(), 1, y, nud);
      };
      step_vjp<MT, PATH>(stage, zq, A, gdir, garm, nt, ca, fv.rk, lam, lamn, G, gc);
      act.add(fv, e, nt, gc, dact);
    }
  }
  act.flush(fv, e, nt, dact);
  write_gradients<MT>(G, fv.pa, lam, lamn, e, dcoef, dstate0);
}

// ---------------------------------------------------------------- two-warp form
// For fleets with fewer 32-env warps than the GPU has schedulers, where the one-warp kernel
// above leaves most of them idle and runs on instruction latency: blocks of two warps over the
// same 32 envs.  Warp 0 re-runs each checkpoint segment, one evaluation of the step per sub-step,
// and writes the stage records the transposes need to a workspace; warp 1 applies step_vjp from
// those records, one segment behind.  The workspace holds two segments, used alternately; a block
// barrier at each segment boundary hands one over.  The per-env arithmetic is k_adjoint's.
constexpr int kWsThreads = 64;

// Warp 0: segment sg re-run from its checkpoint; record j of `rec` gets sub-step t0 + j.
template <int MT, int PATH>
__device__ __forceinline__ void produce_segment(const FleetView &fv, int64_t e,
                                                const AdjEnv<PATH> &A, const float4 *gdir,
                                                const float4 *garm, int nt, bool ca,
                                                const float *__restrict__ ckpt, int32_t sg,
                                                int32_t C, int32_t T, int64_t step0,
                                                float4 *__restrict__ rec) {
  constexpr int W = rec_words<MT>();
  const int64_t n = fv.n;
  const int32_t t0 = sg * C, len = min(C, T - t0);
  St<MT> S;
  load_checkpoint<MT, PATH>(ckpt, sg, n, e, nt, S);
  float zq[4];
  CommandWalk<MT> cmd(fv, e, nt, step0 + t0);
  for (int32_t j = 0; j < len; ++j) {
    float4 *r = rec + (int64_t)j * W * n;
    stage_step<MT, PATH>(S, cmd.c, A, gdir, garm, nt, ca, fv.rk, zq,
                         [&](int g, const St<MT> &y, const float (&nud)[6]) {
                           put_stage<MT>(r + (int64_t)g * stage_words<MT>() * n, n, y, nud);
                         });
    r[(int64_t)(W - 1) * n] = make_float4(zq[0], zq[1], zq[2], zq[3]);
    cmd.next(fv, e, nt);
  }
}

// Per-lane asynchronous copies global -> shared (sm_80+ cp.async), so that the consumer warp's next
// record is in flight while it works on the current one.
__device__ __forceinline__ void cp_async4(float *smem, const float *gmem) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(sa), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async16(float4 *smem, const float4 *gmem) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(sa), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() {
  asm volatile("cp.async.commit_group;\n" ::: "memory");
}
__device__ __forceinline__ void cp_async_wait_all_but_one() {
  asm volatile("cp.async.wait_group 1;\n" ::: "memory");
}

// What the consumer reads per sub-step, double-buffered in shared memory: the stage records [W][32]
// float4 and the loss adjoint of the sub-step's output [MG_NTRAJ][32].
template <int MT>
struct Fetch {
  float4 rec[2][rec_words<MT>()][32];
  float adj[2][MG_NTRAJ][32];
};

// Queue the copies of sub-step t0 + j's inputs into slot j & 1 (this lane's column).
template <int MT>
__device__ __forceinline__ void fetch_substep(const FleetView &fv, int64_t e, int lane,
                                              const float4 *__restrict__ rec,
                                              const float *__restrict__ dtraj, int64_t t0,
                                              int32_t j, Fetch<MT> &buf) {
  constexpr int W = rec_words<MT>();
  const int64_t n = fv.n;
  const float4 *r = rec + (int64_t)j * W * n;
#pragma unroll
  for (int f = 0; f < W; ++f) cp_async16(&buf.rec[j & 1][f][lane], r + (int64_t)f * n);
  const float *g = dtraj + (t0 + j) * MG_NTRAJ * n + e;
#pragma unroll
  for (int f = 0; f < MG_NTRAJ; ++f) cp_async4(&buf.adj[j & 1][f][lane], g + (int64_t)f * n);
  cp_async_commit();
}

// Warp 1: segment sg walked backwards from its records, each sub-step's inputs copied into
// shared memory while the previous one is processed.
template <int MT, int PATH>
__device__ __forceinline__ void consume_segment(const FleetView &fv, int64_t e, int lane,
                                                const AdjEnv<PATH> &A, const float4 *gdir,
                                                const float4 *garm, int nt, bool ca,
                                                const float *__restrict__ dtraj, int32_t sg,
                                                int32_t C, int32_t T,
                                                const float4 *__restrict__ rec, Fetch<MT> &buf,
                                                float *__restrict__ dact, ActionAdjoint<MT> &act,
                                                Body &lam, float (&lamn)[MT], Grad<PATH> &G) {
  constexpr int W = rec_words<MT>();
  const int32_t t0 = sg * C, len = min(C, T - t0);
  float gc[MT];
  fetch_substep<MT>(fv, e, lane, rec, dtraj, t0, len - 1, buf);
  for (int32_t j = len - 1; j >= 0; --j) {
    if (j > 0)
      fetch_substep<MT>(fv, e, lane, rec, dtraj, t0, j - 1, buf);
    else
      cp_async_commit();  // an empty group keeps "all but the newest" meaning sub-step j
    cp_async_wait_all_but_one();
    const float4 *b = &buf.rec[j & 1][0][lane];
    add_traj_adjoint(&buf.adj[j & 1][0][lane], 32, lam);
    const float4 z = b[(W - 1) * 32];
    const float zq[4] = {z.x, z.y, z.z, z.w};
    auto stage = [&](int i, St<MT> &y, float (&nud)[6]) {
      get_stage<MT>(b + i * stage_words<MT>() * 32, 32, y, nud);
    };
    step_vjp<MT, PATH>(stage, zq, A, gdir, garm, nt, ca, fv.rk, lam, lamn, G, gc);
    act.add(fv, e, nt, gc, dact);
  }
}

// ws: [2][C][rec_words<MT>()][n] float4.  Grid: one block per 32 envs.  General path: dynamic
// shared memory [32][MG_NXPARAM] for the block's off-diagonal coefficients (both warps read a
// lane's row).
template <int MT, int PATH>
__global__ void __launch_bounds__(kWsThreads)
    k_adjoint_ws(const FleetView fv, const int32_t *__restrict__ types,
                 const float *__restrict__ ckpt, const float *__restrict__ dtraj, int32_t T,
                 int32_t C, int64_t step0, float *__restrict__ dcoef, float *__restrict__ dact,
                 float *__restrict__ dstate0, float4 *__restrict__ ws) {
  __shared__ float4 sgeo[MG_MAX_TYPES][2 * MG_MAX_THR];
  __shared__ Fetch<MT> sbuf;
  extern __shared__ float sxh[];
  stage_geometry(fv, sgeo);
  const int64_t env0 = (int64_t)blockIdx.x * 32;
  if constexpr (adj_general(PATH))
    stage_xh_or_zero(fv, env0, (int)min((int64_t)32, fv.n - env0), sxh);
  __syncthreads();
  const int warp = (int)(threadIdx.x >> 5), lane = (int)(threadIdx.x & 31);
  const int64_t e = env0 + lane;
  const bool live = e < fv.n;  // lanes past the fleet only take part in the barriers
  const int64_t el = live ? e : 0;
  const int type = types[el];
  const float4 *gdir = sgeo[type], *garm = sgeo[type] + MG_MAX_THR;
  const int nt = fv.geo[type].n_thr;
  const bool ca = !(fv.model_flags & MG_MODEL_NO_CURRENT_ACCEL);
  AdjEnv<PATH> A;
  load_env<PATH>(fv, el, sxh + lane * MG_NXPARAM, gdir, garm, A);
  const int64_t slot = (int64_t)C * rec_words<MT>() * fv.n;

  const int32_t n_ck = (T + C - 1) / C;
  if (warp == 0 && live)
    produce_segment<MT, PATH>(fv, e, A, gdir, garm, nt, ca, ckpt, n_ck - 1, C, T, step0,
                              ws + ((n_ck - 1) & 1) * slot + e);
  __syncthreads();
  Grad<PATH> G;
  zero_grad(G);
  Body lam{};
  float lamn[MT];
#pragma unroll
  for (int i = 0; i < MT; ++i) lamn[i] = 0.f;
  ActionAdjoint<MT> act(fv, step0 + T - 1);
  for (int32_t sg = n_ck - 1; sg >= 0; --sg) {
    if (warp == 0) {
      if (live && sg > 0)
        produce_segment<MT, PATH>(fv, e, A, gdir, garm, nt, ca, ckpt, sg - 1, C, T, step0,
                                  ws + ((sg - 1) & 1) * slot + e);
    } else if (live) {
      consume_segment<MT, PATH>(fv, e, lane, A, gdir, garm, nt, ca, dtraj, sg, C, T,
                                ws + (sg & 1) * slot + e, sbuf, dact, act, lam, lamn, G);
    }
    __syncthreads();
  }
  if (warp == 1 && live) {
    act.flush(fv, e, nt, dact);
    write_gradients<MT>(G, fv.pa, lam, lamn, e, dcoef, dstate0);
  }
}

template <int MT, int PATH>
cudaError_t launch_adjoint_t(const FleetView &fv, const int32_t *types, const float *ckpt,
                             const float *dtraj, int32_t T, int32_t C, int64_t step0,
                             float *dcoef, float *dact, float *dstate0, bool split, void *ws,
                             int n_sm, cudaStream_t stream) {
  if (split) {
    const int grid = (int)((fv.n + 31) / 32);
    const size_t smem = adj_general(PATH) ? sizeof(float) * 32 * MG_NXPARAM : 0;
    k_adjoint_ws<MT, PATH><<<grid, kWsThreads, smem, stream>>>(
        fv, types, ckpt, dtraj, T, C, step0, dcoef, dact, dstate0, static_cast<float4 *>(ws));
    return cudaGetLastError();
  }
  // One warp per block while the fleet has fewer warps than the GPU has SMs x 4 (the backward
  // pass is latency-bound, so its warps should be spread over all SMs, each with its own L1 for
  // the threads' recompute buffers), larger blocks beyond.
  const int64_t warps = (fv.n + 31) / 32;
  const int threads = warps <= 4 * (int64_t)n_sm ? 32 : kAdjThreads;
  const int grid = (int)((fv.n + threads - 1) / threads);
  const size_t smem = adj_general(PATH) ? sizeof(float) * threads * MG_NXPARAM : 0;
  k_adjoint<MT, PATH><<<grid, threads, smem, stream>>>(fv, types, ckpt, dtraj, T, C, step0, dcoef,
                                                       dact, dstate0);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- forward pass
// The forward of the differentiable rollout in one launch: T sub-steps from the sim's state on
// the static grid, the state written to ckpt [n_ck][MG_NSTATE][n] (record order, lag entries
// past the vehicle's thrusters zero) before sub-steps 0, C, 2C, ... and the trajectory recorded
// after every sub-step into traj [T][MG_NTRAJ][n].  Per env the arithmetic is advance_env's
// (the same step code, commands and lag segments), so the result equals a chain of recording
// launches of C sub-steps each, bit for bit, without the launches or the state's round trips.
template <int MT>
__device__ __forceinline__ void write_checkpoint(float *__restrict__ ck, int64_t n, int64_t e,
                                                 const St<MT> &s) {
  float *c = ck + e;
  for (int i = 0; i < 3; ++i) c[(int64_t)i * n] = s.p[i];
  for (int i = 0; i < 4; ++i) c[(int64_t)(3 + i) * n] = s.q[i];
  for (int i = 0; i < 3; ++i) c[(int64_t)(7 + i) * n] = s.v[i];
  for (int i = 0; i < 3; ++i) c[(int64_t)(10 + i) * n] = s.w[i];
#pragma unroll
  for (int i = 0; i < MG_MAX_THR; ++i) c[(int64_t)(13 + i) * n] = i < MT ? s.n[i] : 0.f;
}

template <int NTV, bool DIAG, int NH, bool XH>
__global__ void __maxnreg__(XH ? kRegsXH : DIAG ? kRegsWide : kRegsGeneral)
    k_rollout_fwd(const FleetView fv, const BlockDesc *__restrict__ blocks, const int32_t T,
                  const int32_t C, float *__restrict__ traj, float *__restrict__ ckpt) {
  constexpr int MT = (NTV == NT_6) ? 6 : 8;
  constexpr bool MIXED = (NTV == NT_MIXED);
  __shared__ float4 sdir[MG_MAX_THR], sarm[MG_MAX_THR];
  __shared__ unsigned s_done;
  __shared__ int64_t s_cursor;
  extern __shared__ float sxh[];
  const BlockDesc bd = blocks[blockIdx.x];
  if (threadIdx.x < MG_MAX_THR) {
    sdir[threadIdx.x] = fv.geo[bd.type].dir[threadIdx.x];
    sarm[threadIdx.x] = fv.geo[bd.type].arm[threadIdx.x];
  }
  if (threadIdx.x == 0) {
    s_done = 0u;
    s_cursor = launch_cursor(fv);
  }
  if constexpr (XH) stage_xh(fv.xh, fv.n, bd.env0, bd.count, sxh);
  __syncthreads();
  if ((int)threadIdx.x >= bd.count) return;
  const int64_t e = (int64_t)bd.env0 + threadIdx.x;
  const int64_t n = fv.n;
  const int nt = MIXED ? bd.n_thr : MT;
  const bool current_accel = !(fv.model_flags & MG_MODEL_NO_CURRENT_ACCEL);
  const float *xh = XH ? sxh + threadIdx.x * MG_NXPARAM : nullptr;

  St<MT> s;
  load_state<MT>(fv.st, e, s);
  drop_unused_lag<MT, MIXED, NH>(s, nt);
  Coef<DIAG, NH> P;
  {
    Par<DIAG> raw;
    load_par<DIAG>(fv.pa, e, raw);
    P = make_coef<DIAG, NH>(raw, sdir, sarm);
  }
  const int64_t step0 = s_cursor + fv.cursor_off;
  int64_t seg = step0 / fv.hold;
  int32_t left = fv.hold - (int32_t)(step0 - seg * fv.hold);
  const LagEnv L = lag_env(P.itau, fv.dt);
  float c[MT];
  load_commands<MT>(fv, e, seg, nt, c);
  if (left < T) prefetch_commands(fv, e, seg);
  for (int32_t it = 0; it < T; ++it) {
    if (it % C == 0) write_checkpoint<MT>(ckpt + (int64_t)(it / C) * MG_NSTATE * n, n, e, s);
    if (left == 0) {
      ++seg;
      left = fv.hold;
      load_commands<MT>(fv, e, seg, nt, c);
      if (left < T - it) prefetch_commands(fv, e, seg);
    }
    // packed updates (axpy), packed / not, 200 sub-steps: eight thrusters 179 / 187 us at 30,000
    // envs, 109 / 109 at 4,096 (general path 269 / 277, 158 / 162); six 173 / 175 and 105 / 103
    if constexpr (XH || MT > 6)
      rk4_step<MT, DIAG, MIXED, NH, XH>(s, c, L, P, sdir, sarm, nt, current_accel, fv.rk2, xh);
    else
      rk4_step<MT, DIAG, MIXED, NH, XH>(s, c, L, P, sdir, sarm, nt, current_accel, fv.rk, xh);
    --left;
    record<MT>(traj + (int64_t)it * MG_NTRAJ * n, n, e, s);
  }
  store_and_flag<MT, false>(fv, e, s);
  if (fv.cursor_adv) finish_envs(fv, &s_done, bd.count, fv.cursor_adv);
}

template <int NTV, bool DIAG, int NH, bool XH>
cudaError_t rollout_fwd_t(const FleetView &fv, const BlockDesc *blocks, int n_blocks,
                          int threads, int32_t T, int32_t C, float *traj, float *ckpt,
                          cudaStream_t stream) {
  const size_t smem = XH ? sizeof(float) * threads * MG_NXPARAM : 0;  // <= 46,080 B
  k_rollout_fwd<NTV, DIAG, NH, XH><<<n_blocks, threads, smem, stream>>>(fv, blocks, T, C, traj,
                                                                         ckpt);
  return cudaGetLastError();
}

template <int NTV>
cudaError_t rollout_fwd_d(const FleetView &fv, const BlockDesc *blocks, int n_blocks,
                          int threads, bool diag, int layout, int32_t T, int32_t C,
                          float *traj, float *ckpt, cudaStream_t stream) {
  if (diag)
    return with_layout<true>(layout, [&](auto l) {
      return rollout_fwd_t<NTV, true, decltype(l)::value, false>(fv, blocks, n_blocks, threads, T,
                                                                 C, traj, ckpt, stream);
    });
  return with_layout<false>(layout, [&](auto l) {
    constexpr int L = decltype(l)::value;
    return fv.xh ? rollout_fwd_t<NTV, false, L, true>(fv, blocks, n_blocks, threads, T, C, traj,
                                                      ckpt, stream)
                 : rollout_fwd_t<NTV, false, L, false>(fv, blocks, n_blocks, threads, T, C, traj,
                                                       ckpt, stream);
  });
}

}  // namespace

cudaError_t launch_rollout_forward(const FleetView &fv, const BlockDesc *blocks, int n_blocks,
                                   int threads, NtVariant ntv, bool diag, int layout,
                                   int32_t T, int32_t C, float *traj, float *ckpt,
                                   cudaStream_t stream) {
  if (threads < 32 || threads > 256 || threads % 32 || n_blocks < 1 || T < 1 || C < 1 ||
      (fv.xh && diag))
    return cudaErrorInvalidValue;
  switch (ntv) {
    case NT_6:
      return rollout_fwd_d<NT_6>(fv, blocks, n_blocks, threads, diag, layout, T, C, traj,
                                 ckpt, stream);
    case NT_8:
      return rollout_fwd_d<NT_8>(fv, blocks, n_blocks, threads, diag, layout, T, C, traj,
                                 ckpt, stream);
    default:
      return rollout_fwd_d<NT_MIXED>(fv, blocks, n_blocks, threads, diag, layout, T, C,
                                     traj, ckpt, stream);
  }
}

namespace {

cudaError_t sm_count(int *n_sm) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(n_sm, cudaDevAttrMultiProcessorCount, dev);
  return e;
}

}  // namespace

cudaError_t adjoint_split(int64_t n, int mode, bool *split) {
  if (mode == 1 || mode == 2) {
    *split = mode == 2;
    return cudaSuccess;
  }
  // By fleet size: the two-warp form while all its blocks are resident at once (four per SM, 19,456
  // envs).  200 sub-steps, checkpoints every 20, one-warp / two-warp, us: diagonal mass 4,096 envs
  // 453 / 303, 18,000 568 / 516, 20,480 787 / 935, 32,768 837 / 987; general 4,096 1,148 / 695,
  // 18,000 1,349 / 1,005, 20,480 1,794 / 1,935, 32,768 1,968 / 1,973.
  int n_sm = 0;
  cudaError_t e = sm_count(&n_sm);
  if (e != cudaSuccess) return e;
  *split = (n + 31) / 32 <= 4 * (int64_t)n_sm;
  return cudaSuccess;
}

size_t adjoint_workspace_bytes(bool eight, int64_t n, int32_t C) {
  return 2 * (size_t)C * (size_t)(eight ? rec_words<8>() : rec_words<6>()) * (size_t)n *
         sizeof(float4);
}

cudaError_t launch_adjoint(const FleetView &fv, const int32_t *types, bool eight, bool general,
                           int layout, const float *ckpt, const float *dtraj, int32_t T, int32_t C,
                           int64_t step0, float *dcoef, float *dact, float *dstate0, bool split,
                           void *ws, cudaStream_t stream) {
  if (C < 1 || C > kMaxSeg || T < 1 || (split && !ws)) return cudaErrorInvalidValue;
  int n_sm = 0;
  cudaError_t e = sm_count(&n_sm);
  if (e != cudaSuccess) return e;
  auto run = [&](auto launch) {
    return launch(fv, types, ckpt, dtraj, T, C, step0, dcoef, dact, dstate0, split, ws, n_sm,
                  stream);
  };
  auto on_path = [&](auto p) {
    return eight ? run(launch_adjoint_t<8, decltype(p)::value>)
                 : run(launch_adjoint_t<6, decltype(p)::value>);
  };
  if (general)
    return layout == MG_LAYOUT_MIRRORED
               ? on_path(std::integral_constant<int, ADJ_GEN_MIRRORED>())
               : on_path(std::integral_constant<int, ADJ_GEN>());
  if (layout == MG_LAYOUT_MIRRORED) return on_path(std::integral_constant<int, ADJ_MIRRORED>());
  if (layout == MG_LAYOUT_MIRRORED_G) return on_path(std::integral_constant<int, ADJ_MIRRORED_G>());
  return on_path(std::integral_constant<int, ADJ_DENSE>());
}

int adjoint_max_interval() { return kMaxSeg; }

}  // namespace mg
