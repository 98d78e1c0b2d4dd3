// Step bookkeeping kernels: predictor, commit and rollback (DisMech,
// arXiv 2311.18126, Sec. III-C: q_dot_{n+1} = (q_{n+1} - q_n)/dt; Sec. III:
// reference frames carried between steps by time-parallel transport).
#include "dm_internal.h"
#include "dm_kernels.cuh"

namespace dm {

// Start of a step: every system active, Newton guess q = q_n + dt qdot_n
// (reading C23), fixed DOFs keep q_n.
__global__ void k_begin_step(StepArgs a) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < a.nsys) {
    a.sys_active[i] = 1;
    a.sys_iters[i] = 0;
    a.sys_status[i] = 0;
    a.sys_res[i] = 0ull;
  }
  if (i < a.nd) a.q[i] = a.fixed[i] ? a.qn[i] : fma(a.dt, a.vn[i], a.qn[i]);
}

// Length-projected Newton guess (an option of the predictor): for each
// single-rod system, every edge of the guess in q is rescaled to its length
// in the committed state q_n, node positions rebuilt outward from the rod's
// first node along the guess's edge directions; a node with a fixed position
// DOF keeps its value.  The stiff stretching part of the guess's error goes,
// the soft bending part stays.  The rebuilt positions are a prefix sum of
// the rescaled edge vectors that restarts at node 0 and at every fixed node
// (a segmented scan; Eq. 1 layout: node k at DOFs 4k..4k+2): NT threads per
// system, each sums a run of consecutive nodes serially, the runs' totals are
// scanned over the threads, and the nodes before a run's first restart take
// the total before it.  A warp for the rods of a batch, 512 threads where the
// longest has more than 512 nodes (a warp's 160 passes over a rod of 5000
// nodes took 727 us, 87 us now).
// Implicit midpoint (q holds the midpoint guess y): the projection acts on
// the step's end guess 2y - q_n and y is rebuilt as its mean with q_n.
template <int NT>
__global__ void __launch_bounds__(NT) k_project_lengths(const int32_t *sys_kind, const int32_t *sys_dof0,
                                                        const int32_t *sys_ndof, const uint8_t *fixed,
                                                        const double *qn, double *q, int midpoint) {
  constexpr int kWarps = NT / 32;
  __shared__ double wsum[kWarps][3];
  __shared__ int whead[kWarps];
  const int s = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (sys_kind[s] != SOLVE_ROD_BAND) return;  // block-uniform
  const unsigned full = 0xffffffffu;
  const int d0 = sys_dof0[s], N = (sys_ndof[s] + 1) / 4;
  const int per = (N + NT - 1) / NT, k0 = min(N, tid * per), k1 = min(N, k0 + per);
  auto guess = [&](int o, double(&g)[3]) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      g[c] = q[o + c];
      if (midpoint) g[c] = 2.0 * g[c] - qn[o + c];
    }
  };
  double p[3] = {0.0, 0.0, 0.0};  // the guess of the node before the run
  if (k0 > 0 && k0 < k1) guess(d0 + 4 * (k0 - 1), p);
  __syncthreads();  // before any node is rewritten
  double v[3] = {0.0, 0.0, 0.0};  // sum since the run's start or its last restart
  int first = k1;                 // the run's first restart
  for (int k = k0; k < k1; ++k) {
    const int o = d0 + 4 * k;
    double g[3];
    guess(o, g);
    const bool keep = k == 0 || fixed[o] || fixed[o + 1] || fixed[o + 2];
    if (keep) {
      if (first == k1) first = k;
#pragma unroll
      for (int c = 0; c < 3; ++c) v[c] = g[c];
    } else {
      double e2 = 0.0, l2 = 0.0, e[3];
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        e[c] = g[c] - p[c];
        const double l = qn[o + c] - qn[o + c - 4];
        e2 += e[c] * e[c];
        l2 += l * l;
      }
      const double sc = e2 > 0.0 ? sqrt_any(l2 * rcp_any(e2)) : 1.0;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        v[c] = fma(sc, e[c], v[c]);
        // relative to the run's start before its first restart, else final
        q[o + c] = first < k1 && midpoint ? 0.5 * (qn[o + c] + v[c]) : v[c];
      }
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) p[c] = g[c];
  }
  // the totals before each run: inclusive segmented scan over the warp, then over the warps
  bool h = first < k1 || k0 >= k1;  // (an empty run has nothing after it)
  double t[3] = {v[0], v[1], v[2]};
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const bool uh = __shfl_up_sync(full, (int)h, d) != 0;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const double u = __shfl_up_sync(full, t[c], d);
      if (lane >= d && !h) t[c] += u;
    }
    if (lane >= d) h = h || uh;
  }
  if (lane == 31) {
    whead[warp] = h;
#pragma unroll
    for (int c = 0; c < 3; ++c) wsum[warp][c] = t[c];
  }
  double b[3];
  bool bh = __shfl_up_sync(full, (int)h, 1) != 0;
#pragma unroll
  for (int c = 0; c < 3; ++c) b[c] = __shfl_up_sync(full, t[c], 1);
  if (lane == 0) {
    bh = false;
    b[0] = b[1] = b[2] = 0.0;
  }
  if (kWarps > 1) {
    __syncthreads();
    for (int w = warp - 1; w >= 0 && !bh; --w) {
#pragma unroll
      for (int c = 0; c < 3; ++c) b[c] += wsum[w][c];
      bh = whead[w] != 0;
    }
  }
  for (int k = k0; k < first; ++k) {
    const int o = d0 + 4 * k;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const double x = q[o + c] + b[c];
      q[o + c] = midpoint ? 0.5 * (qn[o + c] + x) : x;
    }
  }
}

void project_lengths(int nsys, int max_nodes, const int32_t *sys_kind, const int32_t *sys_dof0,
                     const int32_t *sys_ndof, const uint8_t *fixed, const double *qn, double *q, int midpoint,
                     cudaStream_t st) {
  if (max_nodes > 512)
    k_project_lengths<512><<<nsys, 512, 0, st>>>(sys_kind, sys_dof0, sys_ndof, fixed, qn, q, midpoint);
  else
    k_project_lengths<32><<<nsys, 32, 0, st>>>(sys_kind, sys_dof0, sys_ndof, fixed, qn, q, midpoint);
}

// Commit the converged step: velocities, then q_n, the transported reference
// directors and tangents of every edge, and the reference twist of every
// stencil (all computed at the converged iterate).
__global__ void k_commit(StepArgs a) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const double idt = 1.0 / a.dt;
  if (i < a.nd) {
    const double q = a.q[i];
    a.vn[i] = a.vnew ? a.vnew[i] : (q - a.qn[i]) * idt;
    a.qn[i] = q;
  }
  if (i < a.ne) {
    const int NE = a.ne;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      a.tn[c * NE + i] = a.ef[c * NE + i];
      a.d1n[c * NE + i] = a.ef[(4 + c) * NE + i];
    }
  }
  if (i < a.ns) a.beta_n[i] = a.beta_it[i];
}

// Implicit midpoint, solved as backward Euler over dt/2 (a.dt) for the
// midpoint configuration y (held in q): with y = (q_n + q_{n+1})/2 the
// midpoint residual 2M/dt^2 (q_{n+1} - q_n - dt qdot_n) - F(y) is the
// backward-Euler residual 4M/dt^2 (y - q_n - (dt/2) qdot_n) - F(y), and the
// velocity of velocity-dependent forces (x_{n+1} - x_n)/dt = (y - x_n)/(dt/2).
// Here: q <- q_{n+1} = 2y - q_n and the staged velocity qdot_{n+1} =
// 2 (q_{n+1} - q_n)/dt - qdot_n = 2 (y - q_n)/(dt/2) - qdot_n (zero on fixed
// DOFs); every system is marked active so that the frames and the reference
// twist can be evaluated at q_{n+1} before the commit.
__global__ void k_midpoint_finish(StepArgs a, double *vnew) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < a.nd) {
    const double y = a.q[i], qn = a.qn[i];
    vnew[i] = a.fixed[i] ? 0.0 : 2.0 * (y - qn) / a.dt - a.vn[i];
    a.q[i] = a.fixed[i] ? qn : 2.0 * y - qn;
  }
  if (i < a.nsys) a.sys_active[i] = 1;
}

// Systems whose status was set outside the Newton bookkeeping (the frame
// evaluation at q_{n+1} of an implicit-midpoint step) count as failed.
__global__ void k_collect_failures(int nsys, const int32_t *sys_status, int32_t *ctrl) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= nsys || sys_status[s] == 0) return;
  atomicAdd(&ctrl[1], 1);
  atomicMin(&ctrl[2], s);
}

// Failed step: drop the iterate, the committed state is untouched.
__global__ void k_restore(StepArgs a) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < a.nd) a.q[i] = a.qn[i];
}

// End of one Newton round inside the round graph: counts the round and
// keeps the graph's while loop going while some system is still active and
// fewer than max_rounds rounds have run (ctrl[0] = systems still active,
// ctrl[4] = rounds of this step), so the loop always ends.
__global__ void k_round_continue(int32_t *ctrl, int max_rounds, cudaGraphConditionalHandle h) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  const int r = ++ctrl[4];
  cudaGraphSetConditional(h, (ctrl[0] > 0 && r < max_rounds) ? 1u : 0u);
}

// Counts a round run before the graph's while node (the fused first round).
__global__ void k_round_count(int32_t *ctrl) {
  if (threadIdx.x == 0 && blockIdx.x == 0) ++ctrl[4];
}

// Committed tangents recomputed from q (after a state is set).
__global__ void k_tangents(int ne, const int32_t *edge_a, const int32_t *edge_b,
                           const double *q, double *tn, int32_t *bad) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= ne) return;
  const int ia = edge_a[e], ib = edge_b[e];
  const double x = q[ib] - q[ia], y = q[ib + 1] - q[ia + 1], z = q[ib + 2] - q[ia + 2];
  const double l2 = x * x + y * y + z * z;
  if (!(l2 > 0.0)) {
    atomicExch(bad, 1);
    return;
  }
  const double il = rsqrt(l2);
  tn[e] = x * il;
  tn[ne + e] = y * il;
  tn[2 * ne + e] = z * il;
}

}  // namespace dm
