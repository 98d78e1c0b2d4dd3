// Residual, Jacobian assembly and line search of the backward-Euler Newton
// iteration (DisMech, arXiv 2311.18126, Sec. III-C, Eq. 15-16), FP64.
//
//  k_rows_rod   -- one thread per DOF row of a single-rod system: gathers the
//                  forces of the stencils/edges that touch the DOF (Eq. 9 plus
//                  gravity and damping), forms the residual
//                  f = M/dt^2 (q - q_n) - M/dt qdot_n - F, its scaled size
//                  |f| / (D l) (max-reduced per system), and the lower band
//                  row of J = M/dt^2 - dF/dq (half bandwidth 10 in the Eq. 1
//                  layout: a bend-twist stencil spans DOFs 4m-4 .. 4m+6).
//  k_line_search -- one block per system: Armijo test and backtracking.
#include "dm_internal.h"
#include "dm_kernels.cuh"
#include "dm_terms.cuh"

namespace dm {

template <int n>
__device__ __forceinline__ constexpr int upk(int i, int j) {
  return i * n - i * (i - 1) / 2 + (j - i);
}

__device__ __forceinline__ int ksym(int c, int cp) {  // packed 3x3 (xx,xy,xz,yy,yz,zz)
  int i = c < cp ? c : cp, j = c < cp ? cp : c;
  return 3 + (i == 0 ? j : (i == 1 ? 2 + j : 5));
}

// The band pass runs for a system only if the solver will factor its
// Jacobian this round (the test of the Hessian pass of the stencils).
__device__ __forceinline__ bool band_due(const RowArgs &a, int s) {
  if (a.sys_status[s] != 0) return false;
  if (a.ls_action && a.ls_action[s] == 1) return false;
  return !(__longlong_as_double((long long)a.sys_res[s]) <= a.tol);
}

// One DOF row (the work of one thread); returns early when inactive.
// MODE 0: residual and band row; 1: residual only (the residual pass of a
// round); 2: band row of the systems the solver will factor (the Jacobian
// pass).  Returns the row's scaled residual |f| / (D l) (as its bits; 0 where
// there is none) for the system in `sys` (-1: none).
template <int MODE>
__device__ __forceinline__ unsigned long long k_rows_rod_one(const RowArgs &a, const int i, int &sys) {
  sys = -1;
  bool act = i < a.nd && a.sys_active[a.dof_sys[i]] &&
             a.sys_kind[a.dof_sys[i]] != SOLVE_GENERAL;
  if (MODE == 2 && act) act = band_due(a, a.dof_sys[i]);
  count_units(a.units, act);
  if (!act) return 0;
  const int s = a.dof_sys[i];
  const int rod = a.dof_rod[i];
  const int base = a.rod_dof0[rod];
  const int r = i - base;
  const int n = a.rod_ndof[rod];
  const int N = (n + 1) >> 2;
  const int node = r >> 2, c = r & 3;
  const int st0 = a.rod_st0[rod], e0 = a.rod_edge0[rod];
  const int NS = a.ns, NE = a.ne;
  // G = minus the sum of the forces on DOF i (the residual adds it), so
  // that the sums start from their first term, not from an add to zero
  double G = 0.0;
  double brow[11];
  // stencils m (interior nodes 1..N-2) with 4m-4 <= r <= 4m+6
  int mlo = (r - 6 + 3) >= 0 ? (r - 6 + 3) / 4 : 0;
  if (mlo < 1) mlo = 1;
  int mhi = (r + 4) / 4;
  if (mhi > N - 2) mhi = N - 2;
  {
    const bool any = mlo <= mhi;
    const int lr = r - 4 * (mlo - 1);
    const int st = st0 + mlo - 1;
    if (MODE != 2 && any) G = a.sg[lr * NS + st];
#pragma unroll
    for (int d = 0; d < 11; ++d) {
      const int lc = lr - d;
      brow[d] = (MODE != 1 && any && lc >= 0) ? a.sh[upk<11>(lc, lr) * NS + st] : 0.0;
    }
  }
  for (int m = mlo + 1; m <= mhi; ++m) {
    const int lr = r - 4 * (m - 1);
    const int st = st0 + m - 1;
    if (MODE != 2) G += a.sg[lr * NS + st];
    if (MODE != 1) {
#pragma unroll
      for (int d = 0; d < 11; ++d) {
        const int lc = lr - d;
        if (lc >= 0) brow[d] += a.sh[upk<11>(lc, lr) * NS + st];
      }
    }
  }
  const double m_i = a.mass[i];
  const double idt = a.idt;
  if (c < 3) {
    // one copy per component, so that every index of brow is a constant
    // (brow stays in registers)
#pragma unroll
    for (int cc = 0; cc < 3; ++cc) {
      if (cc != c) continue;
      if (node <= N - 2) {  // edge `node` starts here
        const int e = e0 + node;
        if (MODE != 2) G -= a.es[cc * NE + e];
        if (MODE != 1) {
#pragma unroll
          for (int cp = 0; cp <= cc; ++cp) brow[cc - cp] += a.es[ksym(cc, cp) * NE + e];
        }
      }
      if (node >= 1) {  // edge `node-1` ends here
        const int e = e0 + node - 1;
        if (MODE != 2) G += a.es[cc * NE + e];
        if (MODE != 1) {
#pragma unroll
          for (int cp = 0; cp <= 2; ++cp) {
            const double kv = a.es[ksym(cc, cp) * NE + e];
            if (cp <= cc) brow[cc - cp] += kv;
            brow[4 + cc - cp] -= kv;
          }
        }
      }
    }
    const double cd = a.damp[i];
    if (MODE != 2) {
      G = fma(-m_i, a.g[c], G);
      G = fma(cd, a.q[i] - a.qn[i], G);
    }
    brow[0] += cd;
  }
  if (MODE != 1) {
    brow[0] += m_i * idt * idt;
    if (a.fixed[i]) {
      brow[0] = 1.0;
#pragma unroll
      for (int d = 1; d < 11; ++d) brow[d] = 0.0;
    } else {
#pragma unroll
      for (int d = 1; d < 11; ++d)
        if (r - d < 0 || a.fixed[i - d]) brow[d] = 0.0;
    }
#pragma unroll
    for (int d = 0; d < 11; ++d) a.band[(size_t)d * a.nd + i] = brow[d];
  }
  if (MODE != 2) {
    if (a.fc) G -= a.fc[i];
    double f = m_i * idt * idt * (a.q[i] - a.qn[i]) - m_i * idt * a.vn[i] + G;
    if (a.fixed[i]) f = 0.0;
    a.f[i] = f;
    sys = s;
    return (unsigned long long)__double_as_longlong(fabs(f) * a.rscale[i]);
  }
  return 0;
}

// block-uniform grid-stride loops (count_units synchronises the block)
__global__ void __launch_bounds__(256) k_rows_rod(RowArgs a) {
  for (int b0 = blockIdx.x * blockDim.x; b0 < a.nd; b0 += gridDim.x * blockDim.x) {
    int sys;
    const unsigned long long r = k_rows_rod_one<0>(a, b0 + threadIdx.x, sys);
    max_residual(a.sys_res, sys, r);
  }
}
__global__ void __launch_bounds__(256) k_rows_rod_res(RowArgs a) {
  for (int b0 = blockIdx.x * blockDim.x; b0 < a.nd; b0 += gridDim.x * blockDim.x) {
    int sys;
    const unsigned long long r = k_rows_rod_one<1>(a, b0 + threadIdx.x, sys);
    max_residual(a.sys_res, sys, r);
  }
}
__global__ void __launch_bounds__(256) k_rows_rod_band(RowArgs a) {
  for (int b0 = blockIdx.x * blockDim.x; b0 < a.nd; b0 += gridDim.x * blockDim.x) {
    int sys;
    k_rows_rod_one<2>(a, b0 + threadIdx.x, sys);
  }
}

// Line search (optional): Armijo test on the 2-norm of the scaled residual
// |f_i| / (D_i l_i) of each system (the Newton direction is a descent
// direction for it); a trial point without sufficient decrease is pulled
// halfway back to the last accepted iterate, at most 12 times.  One block
// of kLineSearchThreads per system: the merit in a fixed summation order
// (per-thread strided sums, then a fixed tree: deterministic), the decision
// by thread 0, then the move (or the new accepted iterate) over the
// system's DOFs.
__global__ void __launch_bounds__(kLineSearchThreads) k_line_search(LineSearchArgs a) {
  __shared__ double part[kLineSearchThreads / 32];
  __shared__ int s_action;
  __shared__ double s_alpha;
  const int s = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (s >= a.nsys || !a.sys_active[s]) return;  // block-uniform
  const int d0 = a.sys_dof0[s], n = a.sys_ndof[s];
  // the decision's inputs and the move's first DOFs on the way while the merit
  // is summed
  constexpr int U = 8;
  LineState ls{a.trial[s], a.nback[s], a.wstry ? a.wstry[s] : 0, a.alpha[s], a.racc[s]};
  double qv[U], qa[U];
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const int i = tid + u * kLineSearchThreads;
    qv[u] = i < n ? a.q[d0 + i] : 0.0;
    qa[u] = i < n ? a.qacc[d0 + i] : 0.0;
  }
  double acc = 0.0;
#pragma unroll 4
  for (int i = tid; i < n; i += kLineSearchThreads) {
    const double v = a.f[d0 + i] * a.rscale[d0 + i];
    acc = fma(v, v, acc);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if (lane == 0) part[warp] = acc;
  __syncthreads();
  if (tid == 0) {
    double tot = 0.0;
#pragma unroll
    for (int w = 0; w < kLineSearchThreads / 32; ++w) tot += part[w];
    const double m = sqrt(tot);
    a.merit[s] = m;
    const int action = line_search_decide(m, ls);
    if (a.wstry) a.wstry[s] = 0;
    a.trial[s] = ls.trial;
    a.nback[s] = ls.nback;
    a.racc[s] = ls.racc;
    a.action[s] = action;
    a.alpha[s] = ls.alpha;
    s_action = action;
    s_alpha = ls.alpha;
  }
  __syncthreads();
  const int action = s_action;
  const double alpha = s_alpha;
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const int i = tid + u * kLineSearchThreads;
    if (i >= n) break;
    if (action == 1) a.q[d0 + i] = alpha == 0.0 ? qa[u] : 0.5 * (qv[u] + qa[u]);
    else a.qacc[d0 + i] = qv[u];
  }
  for (int i = d0 + tid + U * kLineSearchThreads; i < d0 + n; i += kLineSearchThreads) {
    if (action == 1) a.q[i] = alpha == 0.0 ? a.qacc[i] : 0.5 * (a.q[i] + a.qacc[i]);
    else a.qacc[i] = a.q[i];
  }
}

}  // namespace dm
