// Residual, Jacobian assembly and line search of the backward-Euler Newton
// iteration (DisMech, arXiv 2311.18126, Sec. III-C, Eq. 15-16), FP64.
//
//  k_rows_rod   -- the DOF rows of single-rod systems: gathers the
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

__host__ __device__ constexpr int ksym(int c, int cp) {  // packed 3x3 (xx,xy,xz,yy,yz,zz)
  const int i = c < cp ? c : cp, j = c < cp ? cp : c;
  return 3 + (i == 0 ? j : (i == 1 ? 2 + j : 5));
}

// Rows of a rod, a block of T threads per T DOFs, in two steps.  First a thread
// sums the element terms of DOF b0 + 4 (t mod T/4) + t / (T/4): a quarter of the
// block has one component c of consecutive nodes (rods have 4 N - 1 DOFs, so c
// changes only where a rod ends), so that every index of the sums is a constant
// and the loads of a term are consecutive.  Then, through shared memory, a
// thread per DOF in order adds the diagonal, the masks and the residual and
// stores.  (One thread per DOF from the start: the four components of a node in
// one warp ran one after the other, 70 FP64 instructions a row, 240 us for the
// fused pass of 1828856 rows whose bytes take 59; now 154, the band pass 80 ->
// 63, the residual pass 56 -> 46.  Bound by the chain of loads, so four blocks
// per SM: two took 103 and 260.)
// MODE 0: residual and band row; 1: residual only (the residual pass of a
// round); 2: band row of the systems the solver will factor (the Jacobian
// pass).
constexpr int kRowThreads = 256;  // at most
__device__ __forceinline__ int row_pitch(int T) { return T / 4 + 4; }  // (conflict-free both ways)

// Loaded without a branch in between, so that system and rod arrive together
// (the kernel is a chain of dependent loads).
struct RowPlace {
  int sys, N, r, st0, e0;
  bool due;
  template <int MODE>
  __device__ __forceinline__ void load(const RowArgs &a, int i0) {
    const int i = min(i0, a.nd - 1), rod = a.dof_rod[i];
    sys = a.dof_sys[i];
    const int base = a.rod_dof0[rod], n = a.rod_ndof[rod], act = a.sys_active[sys], kind = a.sys_kind[sys];
    st0 = a.rod_st0[rod];
    e0 = a.rod_edge0[rod];
    due = act && kind != SOLVE_GENERAL && i0 < a.nd;
    if (MODE == 2) {  // only if the solver will factor its Jacobian this round (as the stencils' Hessian pass)
      const int st = a.sys_status[sys], act2 = a.ls_action ? a.ls_action[sys] : 0;
      const double res = __longlong_as_double((long long)a.sys_res[sys]);
      due = due && st == 0 && act2 != 1 && !(res <= a.tol);
    }
    r = i - base;
    N = (n + 1) >> 2;
  }
};

// Row C of `node` of a rod of N nodes: its band entries without the diagonal's
// mass and damping, and minus the sum of the elastic forces on it (the
// residual adds it), to out[0..10] and out[11], `plane` doubles apart.
template <int MODE, int C>
__device__ __forceinline__ void rod_row(const RowArgs &a, int N, int node, int st0, int e0, double *out, int plane) {
  constexpr int L0 = 8 + C, L1 = 4 + C, L2 = C;  // the row's place in the stencils of node - 1, node, node + 1
  const bool h0 = C < 3 && node >= 2, h1 = node >= 1 && node <= N - 2, h2 = node <= N - 3;
  const int st = st0 + node - 1, NS = a.ns, NE = a.ne;
  const bool es = C < 3 && node <= N - 2, ee = C < 3 && node >= 1;  // edges that start and end here
  if (MODE != 2) {
    double G = h0 ? a.sg[(size_t)(C < 3 ? L0 : 0) * NS + st - 1] : 0.0;
    const double g1 = h1 ? a.sg[(size_t)L1 * NS + st] : 0.0, g2 = h2 ? a.sg[(size_t)L2 * NS + st + 1] : 0.0;
    if (C < 3) {
      const double x = es ? a.es[(size_t)C * NE + e0 + node] : 0.0, y = ee ? a.es[(size_t)C * NE + e0 + node - 1] : 0.0;
      G = (((G + g1) + g2) - x) + y;
    } else {
      G = g1 + g2;
    }
    out[11 * plane] = G;
  }
  if (MODE != 1) {
    double v[11], v1[11], v2[11], x[3], y[3];
#pragma unroll
    for (int d = 0; d < 11; ++d) {
      v[d] = C < 3 && d <= L0 && h0 ? a.sh[(size_t)upk<11>(C < 3 ? L0 - d : 0, C < 3 ? L0 : 0) * NS + st - 1] : 0.0;
      v1[d] = d <= L1 && h1 ? a.sh[(size_t)upk<11>(d <= L1 ? L1 - d : 0, L1) * NS + st] : 0.0;
      v2[d] = d <= L2 && h2 ? a.sh[(size_t)upk<11>(d <= L2 ? L2 - d : 0, L2) * NS + st + 1] : 0.0;
    }
#pragma unroll
    for (int cp = 0; cp < 3; ++cp) {
      x[cp] = cp <= C && es ? a.es[(size_t)ksym(C < 3 ? C : 0, cp) * NE + e0 + node] : 0.0;
      y[cp] = ee ? a.es[(size_t)ksym(C < 3 ? C : 0, cp) * NE + e0 + node - 1] : 0.0;
    }
#pragma unroll
    for (int d = 0; d < 11; ++d) {
      double w = C < 3 ? v[d] : v1[d];
      if (C < 3 && d <= L1) w += v1[d];
      if (d <= L2) w += v2[d];
      if (C < 3) {
        if (d <= C) w += x[C - d < 0 ? 0 : C - d];
        if (d <= C) w += y[C - d < 0 ? 0 : C - d];
        if (d >= 2 + C && d <= 4 + C) w -= y[4 + C - d < 0 ? 0 : 4 + C - d > 2 ? 2 : 4 + C - d];
      }
      out[d * plane] = w;
    }
  }
}

template <int MODE>
__device__ __forceinline__ void rows_rod(const RowArgs &a, double *sm) {
  const int T = blockDim.x, t = threadIdx.x, pitch = row_pitch(T), plane = 4 * pitch, q = t / (T / 4);
  for (int b0 = blockIdx.x * T; b0 < a.nd; b0 += gridDim.x * T) {
    RowPlace pa, pb;
    pa.load<MODE>(a, b0 + 4 * (t - q * (T / 4)) + q);
    pb.load<MODE>(a, b0 + t);
    // the second step's inputs, on the way during the first
    const int i = min(b0 + t, a.nd - 1), c = pb.r & 3;
    const double m = a.mass[i], damp = a.damp[i];
    double dq = 0.0, vn = 0.0, rscale = 0.0, fc = 0.0;
    if (MODE != 2) {
      dq = a.q[i] - a.qn[i];
      vn = a.vn[i];
      rscale = a.rscale[i];
      if (a.fc) fc = a.fc[i];
    }
    unsigned fixed = a.fixed[i] != 0;  // bit d: row i - d is fixed
    if (MODE != 1) {
#pragma unroll
      for (int d = 1; d < 11; ++d) fixed |= a.fixed[max(i - d, 0)] ? 1u << d : 0u;
    }
    if (pa.due) {
      double *out = sm + q * pitch + t - q * (T / 4);
      const int node = pa.r >> 2;
      switch (pa.r & 3) {
        case 0: rod_row<MODE, 0>(a, pa.N, node, pa.st0, pa.e0, out, plane); break;
        case 1: rod_row<MODE, 1>(a, pa.N, node, pa.st0, pa.e0, out, plane); break;
        case 2: rod_row<MODE, 2>(a, pa.N, node, pa.st0, pa.e0, out, plane); break;
        default: rod_row<MODE, 3>(a, pa.N, node, pa.st0, pa.e0, out, plane); break;
      }
    }
    __syncthreads();
    count_units(a.units, pb.due);
    int sys = -1;
    unsigned long long res = 0;
    if (pb.due) {
      const double *in = sm + (t & 3) * pitch + (t >> 2);
      const double idt = a.idt, cd = c < 3 ? damp : 0.0;
      if (MODE != 1) {
        double row[11];
#pragma unroll
        for (int d = 0; d < 11; ++d) row[d] = in[d * plane];
        if (c < 3) row[0] += cd;
        row[0] += m * idt * idt;
#pragma unroll
        for (int d = 1; d < 11; ++d)
          if ((fixed & 1u) || pb.r < d || ((fixed >> d) & 1u)) row[d] = 0.0;
        if (fixed & 1u) row[0] = 1.0;
#pragma unroll
        for (int d = 0; d < 11; ++d) a.band[(size_t)d * a.nd + i] = row[d];
      }
      if (MODE != 2) {
        double G = in[11 * plane];
        if (c < 3) {
          G = fma(-m, a.g[c], G);
          G = fma(cd, dq, G);
        }
        if (a.fc) G -= fc;
        double f = m * idt * idt * dq - m * idt * vn + G;
        if (fixed & 1u) f = 0.0;
        a.f[i] = f;
        sys = pb.sys;
        res = (unsigned long long)__double_as_longlong(fabs(f) * rscale);
      }
    }
    if (MODE != 2) max_residual(a.sys_res, sys, res);
    __syncthreads();
  }
}

__global__ void __launch_bounds__(kRowThreads, 4) k_rows_rod(RowArgs a) {
  __shared__ double sm[12 * 4 * (kRowThreads / 4 + 4)];
  rows_rod<0>(a, sm);
}
__global__ void __launch_bounds__(kRowThreads) k_rows_rod_res(RowArgs a) {
  __shared__ double sm[12 * 4 * (kRowThreads / 4 + 4)];
  rows_rod<1>(a, sm);
}
__global__ void __launch_bounds__(kRowThreads, 4) k_rows_rod_band(RowArgs a) {
  __shared__ double sm[12 * 4 * (kRowThreads / 4 + 4)];
  rows_rod<2>(a, sm);
}

// Line search (optional): Armijo test on the 2-norm of the scaled residual
// |f_i| / (D_i l_i) of each system (the Newton direction is a descent
// direction for it); a trial point without sufficient decrease is pulled
// halfway back to the last accepted iterate, at most 12 times.  One block
// per system: the merit in a fixed summation order (per-thread strided sums,
// then a fixed tree: deterministic), the decision by thread 0, then the move
// (or the new accepted iterate) over the system's DOFs.  128 threads, 512 for
// contact systems of over 1024 DOFs (a coil of 1999: 22 us with 128, 8 with 512).
template <int T>
__device__ __forceinline__ void line_search(const LineSearchArgs &a) {
  __shared__ double part[T / 32];
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
    const int i = tid + u * T;
    qv[u] = i < n ? a.q[d0 + i] : 0.0;
    qa[u] = i < n ? a.qacc[d0 + i] : 0.0;
  }
  double acc = 0.0;
#pragma unroll 4
  for (int i = tid; i < n; i += T) {
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
    for (int w = 0; w < T / 32; ++w) tot += part[w];
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
    const int i = tid + u * T;
    if (i >= n) break;
    if (action == 1) a.q[d0 + i] = alpha == 0.0 ? qa[u] : 0.5 * (qv[u] + qa[u]);
    else a.qacc[d0 + i] = qv[u];
  }
  for (int i = d0 + tid + U * T; i < d0 + n; i += T) {
    if (action == 1) a.q[i] = alpha == 0.0 ? a.qacc[i] : 0.5 * (a.q[i] + a.qacc[i]);
    else a.qacc[i] = a.q[i];
  }
}

__global__ void __launch_bounds__(kLineSearchThreads) k_line_search(LineSearchArgs a) {
  line_search<kLineSearchThreads>(a);
}
__global__ void __launch_bounds__(kLineSearchWide) k_line_search_wide(LineSearchArgs a) {
  line_search<kLineSearchWide>(a);
}

}  // namespace dm
