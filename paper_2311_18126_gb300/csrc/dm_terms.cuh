// Terms of general systems (rods on the ground and joined at elastic joints)
// that several kernels evaluate: a node's contact and friction, a DOF's force
// balance; and the line search's decision.
#pragma once
#include "dm_internal.h"
#include "dm_kernels.cuh"

namespace dm {

// Node v's contact and friction terms.  Bound by their chain of FP64
// instructions: one exponential for the softplus and its derivatives,
// constants from the host, reciprocals of the integer pipe (20 k cycles a node
// before).
__device__ __forceinline__ void node_one(const NodeArgs &a, int v) {
  count_active(a.units);
  const int NN = a.nn;
  const int d = a.node_dof[v];
  const double z = a.q[d + 2] - a.ground_z;
  const double C = a.node_h[v], dl = a.delta, kc = a.node_kc[v];
  // Eq. 10 and its first two derivatives in D
  double dE = 0.0, d2E = 0.0;
  if (z <= C - dl) {
    dE = -2.0 * (C - z);
    d2E = 2.0;
  } else if (z < C + dl) {
    // softplus(s) = max(s, 0) + log(1 + e), its derivative the logistic sg
    const double s = a.K1 * (C - z), e = exp(-fabs(s)), r = rcp_any(1.0 + e), er = e * r;
    const double sp = fmax(s, 0.0) + log1p(e);
    const double sg = s >= 0.0 ? r : er, gs = s >= 0.0 ? er : r;  // gs = 1 - sg
    dE = -2.0 * sp * sg * a.iK1;
    d2E = 2.0 * sg * fma(sp, gs, sg);
  }
  const double Fn = -kc * dE;
  double F[3] = {0.0, 0.0, Fn};
  double J[9] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, kc * d2E};
  const double mu = a.node_mu[v];
  if (mu > 0.0 && Fn != 0.0) {
    const double K2 = a.K2, idt = a.idt;
    const double ux = (a.q[d] - a.qn[d]) * idt, uy = (a.q[d + 1] - a.qn[d + 1]) * idt;
    const double s = sqrt_any(ux * ux + uy * uy);
    const double fn = fabs(Fn);
    if (s == 0.0) {
      // limit of -mu |F_n| gamma(|u|) u/|u| at u = 0 (reading C14)
      const double c = mu * fn * 0.5 * K2 * idt;
      J[0] = c;
      J[4] = c;
    } else {
      const double th = tanh(0.5 * K2 * s);   // gamma of Eq. 12
      const double dth = 0.5 * K2 * (1.0 - th * th);
      const double is = rcp_any(s), hx = ux * is, hy = uy * is;
      F[0] = -mu * th * hx * fn;
      F[1] = -mu * th * hy * fn;
      // -dF/dx in the plane: mu |F_n| [g/s (I - u u^T) + g' u u^T] / dt
      const double a1 = mu * fn * th * is * idt, a2 = mu * fn * dth * idt;
      J[0] = a1 * (1.0 - hx * hx) + a2 * hx * hx;
      J[1] = (a2 - a1) * hx * hy;
      J[3] = J[1];
      J[4] = a1 * (1.0 - hy * hy) + a2 * hy * hy;
      // -dF/dz: |F_n| = -k_c E'(D) in contact, d|F_n|/dz = -k_c E''
      J[2] = -mu * th * hx * kc * d2E;
      J[5] = -mu * th * hy * kc * d2E;
    }
  }
#pragma unroll
  for (int c = 0; c < 3; ++c) a.nt[c * NN + v] = F[c];
#pragma unroll
  for (int k = 0; k < 9; ++k) a.nt[(3 + k) * NN + v] = J[k];
}

// Row i's force balance; the scaled residual's bits.
__device__ __forceinline__ unsigned long long rows_gen_one(const RowGenArgs &a, int i) {
  count_active(a.units);
  // sixteen terms at a time, loaded side by side (a joint node has dozens) and
  // summed in order
  double F = 0.0;
  const int k1 = a.gat_ptr[i + 1];
  for (int k = a.gat_ptr[i]; k < k1; k += 16) {
    int code[16];
    double x[16];
#pragma unroll
    for (int u = 0; u < 16; ++u) code[u] = k + u < k1 ? a.gat_ent[k + u] : -1;
#pragma unroll
    for (int u = 0; u < 16; ++u) {
      const int slot = code[u] & 15, idx = code[u] >> 5;
      x[u] = 0.0;
      if (code[u] < 0) continue;
      if (code[u] & 16) {
        const double v = a.es[(slot % 3) * a.ne + idx];
        x[u] = slot < 3 ? v : -v;
      } else {
        x[u] = -a.sg[slot * a.ns + idx];
      }
    }
#pragma unroll
    for (int u = 0; u < 16; ++u)
      if (k + u < k1) F += x[u];
  }
  const int c = a.dof_comp[i];
  const double m = a.mass[i], idt = a.idt;
  if (c < 3) {
    F += m * a.g[c];
    F -= a.damp[i] * (a.q[i] - a.qn[i]);
    if (a.nt) F += a.nt[c * a.nn + a.dof_node[i]];
  }
  double f = m * idt * idt * (a.q[i] - a.qn[i]) - m * idt * a.vn[i] - F;
  if (a.fixed[i]) f = 0.0;
  a.f[i] = f;
  return (unsigned long long)__double_as_longlong(fabs(f) * a.rscale[i]);
}

// A system's line search state.
struct LineState {
  int trial, nback, wstry;
  double alpha, racc;
};

// The decision at a point of merit m (block-uniform): 1: move back (halfway to
// the accepted iterate, or onto it when alpha comes out 0), 0: accepted.
__device__ __forceinline__ int line_search_decide(double m, LineState &t) {
  if (t.wstry) {
    // the learned guess is kept only if it lowers the merit below that of
    // the extrapolation; otherwise the iterate returns to the extrapolation
    t.wstry = 0;
    if (!(m <= (1.0 - 1e-4) * t.racc)) {
      t.alpha = 0.0;
      t.trial = t.nback = 0;
      return 1;
    }
  }
  if (t.trial && t.nback < 12 && !(m <= (1.0 - 1e-4 * t.alpha) * t.racc)) {
    t.alpha = 0.5 * t.alpha;
    t.nback += 1;
    return 1;
  }
  t.trial = t.nback = 0;
  t.racc = m;
  t.alpha = 1.0;
  return 0;
}

}  // namespace dm
