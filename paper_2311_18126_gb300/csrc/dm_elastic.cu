// Elastic forces and Hessians of the implicit DER step, FP64, sm_103a.
//
//  k_edge     -- one thread per edge: tangent, time-parallel reference frame
//                (Sec. III), material frame, stretching force and Hessian
//                (Sec. III-A, Eq. 2-3).
//  k_stencil  -- one thread per bend-twist stencil: material curvatures
//                (Eq. 4, 5), reference twist and twist (Eq. 7), and the
//                gradient and Hessian of 1/2 EI/V |kappa - kappabar|^2 +
//                1/2 GJ/V (tau - taubar)^2 (Eq. 6, 8) in closed form.
//
// With C the 3 x 3 rotation from one edge's material frame to the other's and
// chi = 1 + C33, the strains are kappa1 = (C13 - C31)/chi, kappa2 = (C23 -
// C32)/chi, and twist = the angle of (C11 + C22, C21 - C12); a rotation of a
// frame maps entries of C to entries of C, so gradient and Hessian over the six
// variables (two tangent-plane directions and the angle, per edge) are short
// polynomials in C's nine entries.  They are formed in these variables (21
// entries instead of 36 in space), the holonomy of the time-parallel transport
// shifts the angles there too, and only the result goes to space.
//
// What bounds these kernels is the FP64 pipe: it charges a full warp slot (64
// cycles of an SM partition) for every FP64 instruction whatever its active
// mask, so each thread owns one whole edge or stencil and all 32 lanes do
// useful work; reciprocals run on the integer pipe.  FP64 instructions per
// stencil, from the kernels' times: gradient 295 -> 195, Hessian 1060 -> 570,
// both in one pass 1000 -> 525.  4096 rods (450046 stencils): fused pass 846 ->
// 444 us, a step's Hessians 1.24 -> 0.67 ms and gradients 0.60 -> 0.39 ms.
#include <cooperative_groups.h>

#include "dm_internal.h"
#include "dm_kernels.cuh"
#include "dm_terms.cuh"

namespace dm {

// One edge (the work of one thread); returns early when inactive.
__device__ __forceinline__ void k_edge_one(EdgeArgs a, const int e) {
  const bool act = e < a.ne && a.sys_active[a.edge_sys[e]];
  count_units(a.units, act);
  if (!act) return;
  const int s = a.edge_sys[e];
  const int ia = a.edge_a[e], ib = a.edge_b[e];
  const double ex = a.q[ib] - a.q[ia];
  const double ey = a.q[ib + 1] - a.q[ia + 1];
  const double ez = a.q[ib + 2] - a.q[ia + 2];
  const double l2 = ex * ex + ey * ey + ez * ez;
  if (!(l2 > 0.0)) {
    atomicMax(&a.sys_status[s], (int)DM_ERR_DEGENERATE);
    return;
  }
  const double il = rsqrt(l2);
  const double l = l2 * il;
  const double tx = ex * il, ty = ey * il, tz = ez * il;
  const int NE = a.ne;
  const double nx = a.tn[e], ny = a.tn[NE + e], nz = a.tn[2 * NE + e];
  const double c = 1.0 + nx * tx + ny * ty + nz * tz;
  if (!(c > 1e-12)) {  // edge reversed within one step: transport undefined
    atomicMax(&a.sys_status[s], (int)DM_ERR_DEGENERATE);
    return;
  }
  // time-parallel transport of d1 from t_n to t (d1 normal to t_n)
  const double px = a.d1n[e], py = a.d1n[NE + e], pz = a.d1n[2 * NE + e];
  const double k = (px * tx + py * ty + pz * tz) * rcp64(c);  // c in (1e-12, 2]
  const double d1x = px - k * (nx + tx), d1y = py - k * (ny + ty), d1z = pz - k * (nz + tz);
  const double d2x = ty * d1z - tz * d1y, d2y = tz * d1x - tx * d1z, d2z = tx * d1y - ty * d1x;
  double sn, cs;
  sincos(a.q[a.edge_th[e]], &sn, &cs);
  double *o = a.ef;
  o[0 * NE + e] = tx;
  o[1 * NE + e] = ty;
  o[2 * NE + e] = tz;
  o[3 * NE + e] = il;
  o[4 * NE + e] = d1x;
  o[5 * NE + e] = d1y;
  o[6 * NE + e] = d1z;
  o[7 * NE + e] = cs * d1x + sn * d2x;   // m1
  o[8 * NE + e] = cs * d1y + sn * d2y;
  o[9 * NE + e] = cs * d1z + sn * d2z;
  o[10 * NE + e] = -sn * d1x + cs * d2x; // m2
  o[11 * NE + e] = -sn * d1y + cs * d2y;
  o[12 * NE + e] = -sn * d1z + cs * d2z;
  // stretching: dE/dx_b = EA (l/lbar - 1) t,
  // Hessian block K = EA/l t t^T + EA (1/lbar - 1/l) I
  const double EA = a.edge_EA[e], ilb = a.edge_ilbar[e];
  const double fm = EA * (l * ilb - 1.0);
  const double al = EA * (ilb - il), be = EA * il;
  double *w = a.es;
  w[0 * NE + e] = fm * tx;
  w[1 * NE + e] = fm * ty;
  w[2 * NE + e] = fm * tz;
  w[3 * NE + e] = fma(be * tx, tx, al);
  w[4 * NE + e] = be * tx * ty;
  w[5 * NE + e] = be * tx * tz;
  w[6 * NE + e] = fma(be * ty, ty, al);
  w[7 * NE + e] = be * ty * tz;
  w[8 * NE + e] = fma(be * tz, tz, al);
}

__global__ void k_edge(EdgeArgs a) {
  if (a.sys_res) {  // (a system that has stopped keeps its residual)
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    for (int s = t; s < a.nsys; s += gridDim.x * blockDim.x)
      if (a.sys_active[s]) a.sys_res[s] = 0ull;
    if (t == 0) a.ctrl[0] = a.ctrl[3] = 0;
  }
  // block-uniform grid-stride loop (count_units synchronises the block)
  for (int b0 = blockIdx.x * blockDim.x; b0 < a.ne; b0 += gridDim.x * blockDim.x)
    k_edge_one(a, b0 + threadIdx.x);
}

// ---------------------------------------------------------------------------
// small vector helpers (FP64)
// ---------------------------------------------------------------------------
struct v3 {
  double x, y, z;
};
__device__ __forceinline__ v3 mk(double x, double y, double z) { return {x, y, z}; }
__device__ __forceinline__ v3 operator+(v3 a, v3 b) { return {a.x + b.x, a.y + b.y, a.z + b.z}; }
__device__ __forceinline__ v3 operator-(v3 a, v3 b) { return {a.x - b.x, a.y - b.y, a.z - b.z}; }
__device__ __forceinline__ v3 operator*(double s, v3 a) { return {s * a.x, s * a.y, s * a.z}; }
__device__ __forceinline__ double dot(v3 a, v3 b) { return fma(a.x, b.x, fma(a.y, b.y, a.z * b.z)); }
__device__ __forceinline__ v3 cross(v3 a, v3 b) {
  return {fma(a.y, b.z, -a.z * b.y), fma(a.z, b.x, -a.x * b.z), fma(a.x, b.y, -a.y * b.x)};
}
__device__ __forceinline__ v3 axpy(double s, v3 x, v3 y) {  // s x + y
  return {fma(s, x.x, y.x), fma(s, x.y, y.y), fma(s, x.z, y.z)};
}
// component access by compile-time index
__device__ __forceinline__ double cmp(const v3 &a, int i) { return i == 0 ? a.x : (i == 1 ? a.y : a.z); }
// packed upper-triangle index of an n x n symmetric matrix (i <= j)
template <int n>
__host__ __device__ constexpr int up(int i, int j) {
  return i * n - i * (i - 1) / 2 + (j - i);
}

// s x for s = +-1 given as a sign word (0 or 0x80000000): the sign bit
// flipped on the integer pipe, the same value as the FP64 product
__device__ __forceinline__ double sgnmul(unsigned sw, double x) {
  return __hiloint2double(__double2hiint(x) ^ (int)sw, __double2loint(x));
}
__device__ __forceinline__ unsigned sign_word(int s) { return s < 0 ? 0x80000000u : 0u; }

// An edge's material frame (m1, m2, t), right-handed and orthonormal, in the
// stencil's orientation (a reversed edge: t and m2 flipped), and its 1/l.
struct Frame {
  v3 m1, m2, t;
  double il;
  __device__ __forceinline__ void load(const double *ef, int NE, int e, int sgn) {
    const unsigned sw = sign_word(sgn);
    t = mk(sgnmul(sw, ef[e]), sgnmul(sw, ef[NE + e]), sgnmul(sw, ef[2 * NE + e]));
    il = ef[3 * NE + e];
    m1 = mk(ef[7 * NE + e], ef[8 * NE + e], ef[9 * NE + e]);
    m2 = mk(sgnmul(sw, ef[10 * NE + e]), sgnmul(sw, ef[11 * NE + e]), sgnmul(sw, ef[12 * NE + e]));
  }
};

// Holonomy of the time-parallel transport: moving the edge's tangent t also
// rotates the director carried from the committed tangent t_n about t, by the
// holonomy chi of the geodesic triangle (t_n, t, t').  In the material frame,
// over tangent-plane displacements: grad chi = (r, -p), hess chi =
// -[r p, (r^2 - p^2)/2; ., -r p], with (p, r) = (t_n.m1, t_n.m2)/(1 + t_n.t).
__device__ __forceinline__ void holonomy(const double *tn, int NE, int e, int sgn, const Frame &f, double &p,
                                         double &r) {
  const unsigned sw = sign_word(sgn);
  const v3 n = mk(sgnmul(sw, tn[e]), sgnmul(sw, tn[NE + e]), sgnmul(sw, tn[2 * NE + e]));
  const double ic = rcp_int(1.0 + dot(n, f.t));  // k_edge: 1 + t_n.t > 1e-12
  const v3 d = n - f.t;                          // m.t = 0: the short difference loses nothing
  p = ic * dot(f.m1, d);
  r = ic * dot(f.m2, d);
}

// The holonomy's part in the Hessian block H (rows and columns: tangent plane
// 0, 1, angle 2): with E the energy's derivative in the angle, the angle
// shifts by -grad chi . phi - phi . hess chi phi / 2.
__device__ __forceinline__ void shift_block(double &h00, double &h01, double &h11, double &h02, double &h12,
                                            double h22, double E, double p, double r) {
  const double hh = 0.5 * h22;
  const double v0 = fma(-0.5 * E, p, fma(-hh, r, h02)), v1 = fma(-0.5 * E, r, fma(hh, p, h12));
  h00 = fma(-2.0 * r, v0, h00);
  h01 = fma(-r, v1, fma(p, v0, h01));
  h11 = fma(2.0 * p, v1, h11);
  h02 = fma(-r, h22, h02);
  h12 = fma(p, h22, h12);
}

// x m1 + y m2
__device__ __forceinline__ v3 span(double x, v3 m1, double y, v3 m2) {
  return mk(fma(x, m1.x, y * m2.x), fma(x, m1.y, y * m2.y), fma(x, m1.z, y * m2.z));
}

// 3 x 3 block of an edge in space: [h00 h01; h01 h11] in the (scaled) basis
// (m1, m2), and the terms -(g t^T + t g^T) of the angle's second order in the
// edge vector, into h at offset o
__device__ __forceinline__ void expand_block(double *h, int o, double h00, double h01, double h11, double g0,
                                             double g1, v3 m1, v3 m2, v3 t) {
  const v3 u = axpy(-g0, t, span(0.5 * h00, m1, h01, m2)), w = span(0.5 * h11, m2, -g1, t);
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = i; j < 3; ++j) {
      const double x = fma(cmp(m1, i), cmp(u, j), cmp(m2, i) * cmp(w, j));
      h[up<8>(o + i, o + j)] = i == j ? x + x : fma(cmp(u, i), cmp(m1, j), fma(cmp(w, i), cmp(m2, j), x));
    }
}

// atan2(v, u): for |v| <= u/8 by the Taylor series of atan (nine terms: the
// tenth is below 2^-56 of the sum), which costs a fifth of the general
// function's FP64 instructions.
__device__ __forceinline__ double twist_angle(double v, double u) {
  if (!(fabs(v) <= 0.125 * u && rcp64_in_range(u))) return atan2(v, u);
  const double x = v * rcp_int(u), y = x * x;
  double s = -1.0 / 19.0;
  s = fma(s, y, 1.0 / 17.0);
  s = fma(s, y, -1.0 / 15.0);
  s = fma(s, y, 1.0 / 13.0);
  s = fma(s, y, -1.0 / 11.0);
  s = fma(s, y, 1.0 / 9.0);
  s = fma(s, y, -1.0 / 7.0);
  s = fma(s, y, 1.0 / 5.0);
  s = fma(s, y, -1.0 / 3.0);
  return fma(x * y, s, x);
}

// Slot p of the 11 DOFs [x0 (0-2), th_a (3), x1 (4-6), th_b (7), x2 (8-10)]
// as a combination of the 8-space (e_a 0-2, e_b 3-5, A 6, B 7): x0 = -e_a,
// x1 = e_a - e_b, x2 = e_b, th_a = sa A, th_b = sb B.  Term t (0, 1) of
// slot p: its 8-space index (-1: none) and weight (1: +1, -1: -1, 2: sa,
// 3: sb).
__host__ __device__ constexpr int slot_index(int p, int t) {
  return p == 3 ? (t == 0 ? 6 : -1)
       : p == 7 ? (t == 0 ? 7 : -1)
       : p < 3  ? (t == 0 ? p : -1)
       : p < 7  ? (t == 0 ? p - 4 : p - 1)
                : (t == 0 ? p - 5 : -1);
}
__host__ __device__ constexpr int slot_weight(int p, int t) {
  return p == 3 ? 2 : p == 7 ? 3 : p < 3 ? -1 : p < 7 ? (t == 0 ? 1 : -1) : 1;
}

// Gradient of one stencil in its 11 DOFs: (e_a, e_b, A, B) -> [x0, th_a,
// x1, th_b, x2] with x0 = -e_a, x1 = e_a - e_b, x2 = e_b, A = sa th_a,
// B = sb th_b.
__device__ __forceinline__ void write_gradient(const StencilArgs &a, int k, const double *g8,
                                               int sa, int sb) {
  double *G = a.sg;
  const int NS = a.ns;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    G[(0 + c) * NS + k] = -g8[c];
    G[(4 + c) * NS + k] = g8[c] - g8[3 + c];
    G[(8 + c) * NS + k] = g8[3 + c];
  }
  G[3 * NS + k] = sgnmul(sign_word(sa), g8[6]);
  G[7 * NS + k] = sgnmul(sign_word(sb), g8[7]);
}

// The Hessian pass runs for a system only if the solver will factor its
// Jacobian this round: it is still iterating, its residual is above the
// tolerance (the solver's own convergence test on the same value), it has
// not failed, and the line search is not backtracking it.
__device__ __forceinline__ bool hess_due(const StencilArgs &a, int s) {
  if (a.sys_status[s] != 0) return false;
  if (a.ls_action && a.ls_action[s] == 1) return false;
  return !(__longlong_as_double((long long)a.sys_res[s]) <= a.tol);
}

// One bend-twist stencil (the work of one thread); returns early when
// inactive.  MODE 0: gradient and Hessian; 1: reference twist and gradient
// (the residual pass of a round); 2: Hessian of the systems the solver will
// factor, with the reference twist the gradient pass wrote (the Jacobian
// pass of a round).
template <int MODE>
__device__ __forceinline__ void k_stencil_one(StencilArgs a, const int k) {
  bool act = k < a.ns && a.sys_active[a.st_sys[k]];
  if (MODE == 2 && act) act = hess_due(a, a.st_sys[k]);
  count_units(a.units, act);
  if (!act) return;
  const int sys = a.st_sys[k];
  const int NS = a.ns, NE = a.ne;
  const int sg = a.st_sg[k];
  const int sa = (sg & 1) ? -1 : 1, sb = (sg & 2) ? -1 : 1;
  const int ea = a.st_ed[k], eb = a.st_ed[NS + k];
  Frame A, B;
  A.load(a.ef, NE, ea, sa);
  B.load(a.ef, NE, eb, sb);

  // frame b seen from frame a: C = [m1a m2a ta]^T [m1b m2b tb]; its last
  // column and row from tb - ta
  const double z = dot(A.t, B.t), chi = 1.0 + z;
  if (!(chi > 1e-12)) {
    if (MODE != 2) atomicMax(&a.sys_status[sys], (int)DM_ERR_DEGENERATE);
    return;
  }
  const double ic = rcp_int(chi);  // chi in (1e-12, 2]
  const v3 d = B.t - A.t;
  const double C11 = dot(A.m1, B.m1), C12 = dot(A.m1, B.m2), C21 = dot(A.m2, B.m1), C22 = dot(A.m2, B.m2);
  // Eq. 7: reference twist, continued from the committed value: the angle of
  // C's twist about the tangent less the difference of the material angles
  const double th = sgnmul(sign_word(sb), a.q[a.st_th[NS + k]]) - sgnmul(sign_word(sa), a.q[a.st_th[k]]);
  double beta;
  if (MODE == 2) {
    beta = a.beta_it[k];
  } else {
    const double ang = twist_angle(C21 - C12, C11 + C22) - th;
    const double bn = a.beta_n[k];
    double dd = ang - bn;
    dd -= 6.283185307179586 * rint(dd * 0.15915494309189535);
    beta = bn + dd;
    a.beta_it[k] = beta;
    if (a.frames_only) return;
  }
  // everything over chi from here on: C's last column (a, b, z), row (c, d, z)
  const double av = ic * dot(A.m1, d), bv = ic * dot(A.m2, d);
  const double cv = -ic * dot(B.m1, d), dv = -ic * dot(B.m2, d);
  const double zi = ic * z, C11i = ic * C11, C12i = ic * C12, C21i = ic * C21, C22i = ic * C22;
  // Eq. 4, 5: material curvatures
  const double k1 = av - cv, k2 = bv - dv;
  const double kbs = a.st_kb[k], kts = a.st_kt[k];
  const double c1 = kbs * (k1 - a.kbar[k]);
  const double c2 = kbs * (k2 - a.kbar[NS + k]);
  const double c3 = kts * (th + beta - a.taubar[k]);

  // gradients of kappa1, kappa2 and tau over (tangent plane of a, angle a,
  // tangent plane of b, angle b)
  const double zc1 = zi + C11i, zc2 = zi + C22i;
  const double x1[6] = {-fma(k1, av, zc1), -fma(k1, bv, C21i), bv, fma(-k1, cv, zc1), fma(-k1, dv, C12i), -dv};
  const double x2[6] = {-fma(k2, av, C12i), -fma(k2, bv, zc2), -av, fma(-k2, cv, C21i), fma(-k2, dv, zc2), cv};
  const double x3[6] = {-bv, av, -1.0, dv, -cv, 1.0};
  // the curvature energy's gradient, then the energy's
  double ck[6], g[6];
#pragma unroll
  for (int i = 0; i < 6; ++i) ck[i] = fma(c1, x1[i], c2 * x2[i]);
#pragma unroll
  for (int i = 0; i < 6; ++i) g[i] = fma(c3, x3[i], ck[i]);
  double pa, ra, pb, rb;  // holonomies of the two edges
  holonomy(a.tn, NE, ea, sa, A, pa, ra);
  holonomy(a.tn, NE, eb, sb, B, pb, rb);
  const double EA = g[2], EB = g[5], g0 = g[0], g1 = g[1];
  g[0] = fma(-ra, EA, g[0]);
  g[1] = fma(pa, EA, g[1]);
  g[3] = fma(-rb, EB, g[3]);
  g[4] = fma(pb, EB, g[4]);
  // the edges' bases over their lengths: tangent plane -> edge vector
  const v3 A1 = A.il * A.m1, A2 = A.il * A.m2, B1 = B.il * B.m1, B2 = B.il * B.m2;
  double g8[8];
  {
    const v3 x = span(g[0], A1, g[1], A2), y = span(g[3], B1, g[4], B2);
    g8[0] = x.x; g8[1] = x.y; g8[2] = x.z;
    g8[3] = y.x; g8[4] = y.y; g8[5] = y.z;
    g8[6] = EA;
    g8[7] = EB;
  }
  if (MODE == 1) {
    write_gradient(a, k, g8, sa, sb);
    return;
  }

  // Hessian over the six variables, upper triangle.  With k = c1 kappa1 + c2
  // kappa2 and N = chi k: Hess k = (Hess N - grad k grad chi^T - grad chi grad
  // k^T - k Hess chi)/chi, where N and chi are entries of C, whose second
  // derivatives under F -> F exp(phi) exp(theta t) are entries of C again.
  double H[21];
  {
    const double P = fma(c1, av, c2 * bv), Q = fma(c1, cv, c2 * dv), kk = P - Q;
    const double Sa = fma(kk, zi, Q), Sb = fma(kk, zi, -P);
    const double h1 = fma(0.5, fma(-c3, bv, c1), ck[0]), h2 = fma(0.5, fma(c3, av, c2), ck[1]);
    const double f1 = fma(0.5, fma(c3, dv, -c1), ck[3]), f2 = fma(-0.5, fma(c3, cv, c2), ck[4]);
    const double c1z = c1 * zi, c2z = c2 * zi;
    H[up<6>(0, 0)] = fma(-2.0 * av, h1, Sa);
    H[up<6>(0, 1)] = -fma(bv, h1, av * h2);
    H[up<6>(1, 1)] = fma(-2.0 * bv, h2, Sa);
    H[up<6>(0, 2)] = fma(-ck[2], av, c2z);
    H[up<6>(1, 2)] = fma(-ck[2], bv, -c1z);
    H[up<6>(2, 2)] = -P;
    H[up<6>(3, 3)] = fma(-2.0 * cv, f1, Sb);
    H[up<6>(3, 4)] = -fma(dv, f1, cv * f2);
    H[up<6>(4, 4)] = fma(-2.0 * dv, f2, Sb);
    H[up<6>(3, 5)] = fma(-ck[5], cv, -c2z);
    H[up<6>(4, 5)] = fma(-ck[5], dv, c1z);
    H[up<6>(5, 5)] = Q;
    H[up<6>(0, 3)] = fma(-c3, C21i, fma(-kk, C11i, fma(-ck[3], av, fma(-g0, cv, c1 * k1))));
    H[up<6>(0, 4)] = fma(-c3, C22i, fma(-kk, C12i, fma(-ck[4], av, fma(-g0, dv, fma(c2, av, -c1 * dv)))));
    H[up<6>(1, 3)] = fma(c3, C11i, fma(-kk, C21i, fma(-ck[3], bv, fma(-g1, cv, fma(c1, bv, -c2 * cv)))));
    H[up<6>(1, 4)] = fma(c3, C12i, fma(-kk, C22i, fma(-ck[4], bv, fma(-g1, dv, c2 * k2))));
    H[up<6>(0, 5)] = fma(-ck[5], av, fma(c2, C11i, -c1 * C12i));
    H[up<6>(1, 5)] = fma(-ck[5], bv, fma(c2, C21i, -c1 * C22i));
    H[up<6>(2, 3)] = fma(-ck[2], cv, fma(c1, C21i, -c2 * C11i));
    H[up<6>(2, 4)] = fma(-ck[2], dv, fma(c1, C22i, -c2 * C12i));
    H[up<6>(2, 5)] = 0.0;
    // outer products of the gradients
#pragma unroll
    for (int i = 0; i < 6; ++i) {
      const double y1 = kbs * x1[i], y2 = kbs * x2[i], y3 = i == 2 ? -kts : i == 5 ? kts : kts * x3[i];
#pragma unroll
      for (int j = i; j < 6; ++j) {
        const double t = j == 2 ? -y3 : j == 5 ? y3 : 0.0;  // y3 x3[j] for x3[j] = -+1
        const double v = i == 2 && j == 5 ? 0.0 : H[up<6>(i, j)];
        H[up<6>(i, j)] = fma(y1, x1[j], fma(y2, x2[j], j == 2 || j == 5 ? v + t : fma(y3, x3[j], v)));
      }
    }
  }
  // Exact derivatives of the energy with the reference frames carried from
  // the committed step by time-parallel transport (Eq. 9): the angles shift by
  // the holonomies, first a's, then b's.
  shift_block(H[up<6>(0, 0)], H[up<6>(0, 1)], H[up<6>(1, 1)], H[up<6>(0, 2)], H[up<6>(1, 2)], H[up<6>(2, 2)], EA, pa, ra);
#pragma unroll
  for (int j = 3; j < 6; ++j) {
    H[up<6>(0, j)] = fma(-ra, H[up<6>(2, j)], H[up<6>(0, j)]);
    H[up<6>(1, j)] = fma(pa, H[up<6>(2, j)], H[up<6>(1, j)]);
  }
  shift_block(H[up<6>(3, 3)], H[up<6>(3, 4)], H[up<6>(4, 4)], H[up<6>(3, 5)], H[up<6>(4, 5)], H[up<6>(5, 5)], EB, pb, rb);
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    H[up<6>(i, 3)] = fma(-rb, H[up<6>(i, 5)], H[up<6>(i, 3)]);
    H[up<6>(i, 4)] = fma(pb, H[up<6>(i, 5)], H[up<6>(i, 4)]);
  }
  // to edge vectors and angles
  double h[36];
  expand_block(h, 0, H[up<6>(0, 0)], H[up<6>(0, 1)], H[up<6>(1, 1)], g[0], g[1], A1, A2, A.il * A.t);
  expand_block(h, 3, H[up<6>(3, 3)], H[up<6>(3, 4)], H[up<6>(4, 4)], g[3], g[4], B1, B2, B.il * B.t);
  {
    const v3 x = span(H[up<6>(0, 3)], B1, H[up<6>(0, 4)], B2), y = span(H[up<6>(1, 3)], B1, H[up<6>(1, 4)], B2);
    const v3 aA = span(H[up<6>(0, 2)], A1, H[up<6>(1, 2)], A2), aB = span(H[up<6>(0, 5)], A1, H[up<6>(1, 5)], A2);
    const v3 bA = span(H[up<6>(2, 3)], B1, H[up<6>(2, 4)], B2), bB = span(H[up<6>(3, 5)], B1, H[up<6>(4, 5)], B2);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
#pragma unroll
      for (int j = 0; j < 3; ++j) h[up<8>(i, 3 + j)] = fma(cmp(A1, i), cmp(x, j), cmp(A2, i) * cmp(y, j));
      h[up<8>(i, 6)] = cmp(aA, i);
      h[up<8>(i, 7)] = cmp(aB, i);
      h[up<8>(3 + i, 6)] = cmp(bA, i);
      h[up<8>(3 + i, 7)] = cmp(bB, i);
    }
    h[up<8>(6, 6)] = H[up<6>(2, 2)];
    h[up<8>(6, 7)] = H[up<6>(2, 5)];
    h[up<8>(7, 7)] = H[up<6>(5, 5)];
  }
  if (a.dk) {
    // gradients of kappa1 and kappa2 as functions of the 11 DOFs (the same
    // shift of the angles), for the adjoint: d(grad E)/d(kappabar_c) =
    // -EI/V grad kappa_c
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const double *x = c == 0 ? x1 : x2;
      const v3 xa = span(fma(-ra, x[2], x[0]), A1, fma(pa, x[2], x[1]), A2);
      const v3 xb = span(fma(-rb, x[5], x[3]), B1, fma(pb, x[5], x[4]), B2);
      double *o = a.dk + (size_t)(11 * c) * NS + k;
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        o[(size_t)i * NS] = -cmp(xa, i);
        o[(size_t)(4 + i) * NS] = cmp(xa, i) - cmp(xb, i);
        o[(size_t)(8 + i) * NS] = cmp(xb, i);
      }
      o[(size_t)3 * NS] = sgnmul(sign_word(sa), x[2]);
      o[(size_t)7 * NS] = sgnmul(sign_word(sb), x[5]);
    }
  }

  if (MODE == 0) write_gradient(a, k, g8, sa, sb);

  // H11 = T^T H8 T written as packed upper triangle
  auto H8 = [&](int i, int j) -> double { return i <= j ? h[up<8>(i, j)] : h[up<8>(j, i)]; };
  // each entry a signed sum of H8 entries, from its first term (no add of
  // a zero), the signs sa, sb applied on the integer pipe
  double *Ho = a.sh;
  const unsigned swa = sign_word(sa), swb = sign_word(sb);
#pragma unroll
  for (int p = 0; p < 11; ++p)
#pragma unroll
    for (int q = p; q < 11; ++q) {
      double v = 0.0;
      bool first = true;
#pragma unroll
      for (int tp = 0; tp < 2; ++tp)
#pragma unroll
        for (int tq = 0; tq < 2; ++tq) {
          const int ip = slot_index(p, tp), iq = slot_index(q, tq);
          if (ip < 0 || iq < 0) continue;
          const int wp = slot_weight(p, tp), wq = slot_weight(q, tq);
          const bool neg = (wp == -1) != (wq == -1);
          const unsigned sw = (wp == 2 ? swa : wp == 3 ? swb : 0u) ^ (wq == 2 ? swa : wq == 3 ? swb : 0u);
          if (first) {
            v = sgnmul(sw ^ (neg ? 0x80000000u : 0u), H8(ip, iq));
            first = false;
          } else {
            const double x = sgnmul(sw, H8(ip, iq));
            v = neg ? v - x : v + x;
          }
        }
      Ho[up<11>(p, q) * NS + k] = v;
    }
}

// block-uniform grid-stride loops (count_units synchronises the block)
__global__ void __launch_bounds__(128) k_stencil(StencilArgs a) {
  for (int b0 = blockIdx.x * blockDim.x; b0 < a.ns; b0 += gridDim.x * blockDim.x)
    k_stencil_one<0>(a, b0 + threadIdx.x);
}
__global__ void __launch_bounds__(128) k_stencil_grad(StencilArgs a) {
  for (int b0 = blockIdx.x * blockDim.x; b0 < a.ns; b0 += gridDim.x * blockDim.x)
    k_stencil_one<1>(a, b0 + threadIdx.x);
}
__global__ void __launch_bounds__(128) k_stencil_hess(StencilArgs a) {
  for (int b0 = blockIdx.x * blockDim.x; b0 < a.ns; b0 += gridDim.x * blockDim.x)
    k_stencil_one<2>(a, b0 + threadIdx.x);
}

// Line search of batches with general systems: a cluster of four blocks per
// system.  The first decision is on the residual that the round's kernels left
// (the same sums as k_line_search); a small system that is pulled back is then
// evaluated here, again and again until it accepts -- edges, stencil gradients
// and nodes, rows, merit -- instead of a round for every trial point (most
// rounds of a batch of robots did nothing else: 75 us each for the chain of ten
// launches, 64 robots).  Each block decides for itself on the same numbers.
// Bound by the chain of a trial point's FP64 instructions (about 500 of 64
// cycles).  Larger systems (over kLoopDofs) keep a round per trial point: the
// whole chip's threads pay off there.
constexpr int kLoopDofs = 4096;
__global__ void __cluster_dims__(kLoopBlocks, 1, 1) __launch_bounds__(kLineSearchThreads)
    k_line_search_loop(LineSearchArgs a, LineLoopArgs b) {
  cooperative_groups::cluster_group cluster = cooperative_groups::this_cluster();
  __shared__ double part[kLineSearchThreads / 32];
  __shared__ unsigned long long most[kLineSearchThreads / 32];
  const int rank = (int)cluster.block_rank(), s = blockIdx.x / kLoopBlocks;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int t0 = rank * kLineSearchThreads + tid;
  constexpr int kT = kLoopBlocks * kLineSearchThreads;
  if (!a.sys_active[s]) return;  // the whole cluster
  const int d0 = a.sys_dof0[s], n = a.sys_ndof[s];
  const bool small = b.rows.sys_kind[s] == SOLVE_GENERAL && n <= kLoopDofs;
  LineState ls{a.trial[s], a.nback[s], a.wstry ? a.wstry[s] : 0, a.alpha[s], a.racc[s]};
  cluster.sync();  // every block has the state before the first block writes the new one
  const int e0 = b.edge_ptr[s], ne = b.edge_ptr[s + 1] - e0, v0 = b.node_ptr[s];
  const int nv = b.rows.nt ? b.node_ptr[s + 1] - v0 : 0, k0 = b.st_ptr[s], nk = b.st_ptr[s + 1] - k0;
  const int nk32 = (nk + 31) & ~31;
  double m = 0.0;
  unsigned long long res = 0;
  int action = 0;
  bool again = false;
  for (;;) {
    double acc = 0.0;
    res = 0;
#pragma unroll 4
    for (int i = tid; i < n; i += kLineSearchThreads) {
      const double v = a.f[d0 + i] * a.rscale[d0 + i];
      acc = fma(v, v, acc);
      res = max(res, (unsigned long long)__double_as_longlong(fabs(v)));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      acc += __shfl_xor_sync(0xffffffffu, acc, o);
      res = max(res, __shfl_xor_sync(0xffffffffu, res, o));
    }
    if (lane == 0) {
      part[warp] = acc;
      most[warp] = res;
    }
    __syncthreads();
    double tot = 0.0;
#pragma unroll
    for (int w = 0; w < kLineSearchThreads / 32; ++w) {
      tot += part[w];
      res = max(res, most[w]);
    }
    m = sqrt(tot);
    action = line_search_decide(m, ls);
    for (int i = d0 + t0; i < d0 + n; i += kT) {
      if (action == 1) a.q[i] = ls.alpha == 0.0 ? a.qacc[i] : 0.5 * (a.q[i] + a.qacc[i]);
      else a.qacc[i] = a.q[i];
    }
    if (!action || !small) break;
    again = true;
    cluster.sync();
    for (int i = t0; i < ne; i += kT) k_edge_one(b.edges, b.edge_list[e0 + i]);
    cluster.sync();
    for (int i = t0; i < nk32 + nv; i += kT) {  // other warps than the stencils' take the nodes
      if (i < nk) k_stencil_one<1>(b.stencils, b.st_list[k0 + i]);
      else if (i >= nk32) node_one(b.nodes, b.node_list[v0 + i - nk32]);
    }
    cluster.sync();
    for (int i = t0; i < n; i += kT) rows_gen_one(b.rows, d0 + i);
    cluster.sync();
  }
  if (rank == 0 && tid == 0) {
    a.merit[s] = m;
    if (a.wstry) a.wstry[s] = 0;
    a.trial[s] = ls.trial;
    a.nback[s] = ls.nback;
    a.racc[s] = ls.racc;
    a.action[s] = action;
    a.alpha[s] = ls.alpha;
    if (again) b.rows.sys_res[s] = res;
  }
}

}  // namespace dm
