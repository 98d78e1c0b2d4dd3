// Edge-edge contact within a rod (DisMech, arXiv 2311.18126, Sec. III-B,
// Eq. 10-11) and the linear solve of systems that carry it.
//
//  k_cc_cells / k_cc_fill  -- uniform grid over edge midpoints, hashed into a
//                             table; cell size >= longest edge + C + delta,
//                             so two edges closer than C + delta lie in
//                             neighbouring cells.
//  k_cc_pairs              -- a warp per edge, a lane per candidate: the edges
//                             of the 27 neighbouring cells, minus the excluded
//                             pairs (sharing a node or at most two edges apart
//                             along the rod), whose segment distance D is
//                             below C + delta (C = sum of the radii).
//  k_cc_terms              -- a warp per active pair: D and its first and
//                             second derivatives with respect to the 12
//                             node coordinates (in closed form at the closest
//                             points, the 78 second ones spread over the
//                             lanes), k_c E(D) of Eq. 10 by the chain rule; -grad into the contact force vector,
//                             the Hessian into the system's dense matrix.
//  k_cc_band               -- adds the rod's own band (11 lower diagonals of
//                             the symmetric Jacobian) to the dense matrix.
//  k_lu* / k_cc_subst      -- blocked LU without pivoting over the nonzero
//                             32 x 32 tiles of the matrix (the rod band, the
//                             contacts and their fill), all systems at once,
//                             then the solve, q += dq.
#include <algorithm>
#include <cmath>

#include <cooperative_groups.h>

#include "dm_internal.h"
#include "dm_kernels.cuh"

namespace dm {

namespace {

constexpr int kNH = 78;  // packed upper 12x12
constexpr int kHP = 3;   // entries of it per lane

// The lane's entries: coordinates (i, j) of each, and its own coordinate.
struct HLane {
  int i[kHP], j[kHP], own;
  bool on[kHP];
  __device__ __forceinline__ void load(int lane) {
#pragma unroll
    for (int k = 0; k < kHP; ++k) {
      const int e = lane + 32 * k;
      on[k] = e < kNH;
      int r = 0, left = on[k] ? e : 0;
      while (left >= 12 - r) left -= 12 - r++;
      i[k] = r;
      j[k] = r + left;
    }
    own = lane < 12 ? lane : 0;
  }
};

// First-order dual number in the 12 coordinates of a pair (value in every
// lane, the derivative in coordinate l in lane l < 12), for the friction force
// whose Jacobian is not a Hessian.
struct D1 {
  double v, g;
};
__device__ __forceinline__ D1 d1_const(double v) { return {v, 0.0}; }
__device__ __forceinline__ D1 operator+(const D1 &a, const D1 &b) { return {a.v + b.v, a.g + b.g}; }
__device__ __forceinline__ D1 operator-(const D1 &a, const D1 &b) { return {a.v - b.v, a.g - b.g}; }
__device__ __forceinline__ D1 operator*(const D1 &a, const D1 &b) {
  return {a.v * b.v, fma(a.v, b.g, b.v * a.g)};
}
__device__ __forceinline__ D1 operator*(double c, const D1 &a) { return {c * a.v, c * a.g}; }
// f(a) with f(a.v) = f0, f'(a.v) = f1
__device__ __forceinline__ D1 d1_apply(const D1 &a, double f0, double f1) { return {f0, f1 * a.g}; }

// A pair's distance D and its derivatives, spread over a warp.  With f = D^2/2
// as a function of the 12 coordinates x and of (s, t), d = sum_n w_n x_n, w =
// (1 - s, s, t - 1, -t): at the closest points f's derivative in a free s or t
// is zero, so D's gradient is f_x / D and its Hessian comes from f_xx + f_xz z_x
// + (f_xz z_x)^T + z_x^T f_zz z_x, where z_x = (s_x, t_x) are the closest
// points' own derivatives (zero for a clamped one); for near-parallel segments
// f_t t_x and f_t t_xx come in.  Every lane has the values;
// lanes 0-11 the derivatives of their own coordinate, which the lanes' second
// derivatives fetch.  (Second-order dual numbers through the whole computation
// took 1400 FP64 instructions a pair, 94 us a launch for 897 pairs.)
struct Distance {
  double D, s, t, d[3];
  double sx, tx, Dx;  // of the lane's own coordinate
  double dx[3];       // d's, likewise
  double h[kHP], gi[kHP], gj[kHP];
};

// By the same closest-point rule as the plain distance below: s from the
// unconstrained minimiser clamped to [0, 1] (s = 0 for near-parallel
// segments), t for that s clamped, then s again for the clamped t, clamped.
__device__ __forceinline__ Distance pair_distance(const double *x, const HLane &ln) {
  constexpr unsigned full = 0xffffffffu;
  Distance q;
  double a[3], b[3], r[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    a[c] = x[3 + c] - x[c];
    b[c] = x[9 + c] - x[6 + c];
    r[c] = x[c] - x[6 + c];
  }
  const auto dot3 = [](const double *u, const double *v) { return fma(u[0], v[0], fma(u[1], v[1], u[2] * v[2])); };
  const double A = dot3(a, a), B = dot3(a, b), C = dot3(b, b), Dd = dot3(a, r), Ee = dot3(b, r);
  const double den = A * C - B * B, iA = rcp_any(A), iC = rcp_any(C), iden = rcp_any(den);
  const bool parallel = den < 1e-12 * A * C;
  const double s0 = parallel ? 0.0 : (B * Ee - C * Dd) * iden;
  const double s1 = fmin(fmax(s0, 0.0), 1.0);
  const double t0 = fma(B, s1, Ee) * iC;
  q.t = fmin(fmax(t0, 0.0), 1.0);
  const double s2 = fma(B, q.t, -Dd) * iA;
  q.s = fmin(fmax(s2, 0.0), 1.0);
  const bool joint = !parallel && s0 == s1, tfree = t0 == q.t, sfree = s2 == q.s;
  double d1[3];  // d at (s1, t)
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const double rt = fma(-q.t, b[c], r[c]);
    q.d[c] = fma(q.s, a[c], rt);
    d1[c] = fma(s1, a[c], rt);
  }
  const double u = dot3(q.d, q.d);
  q.D = sqrt_any(u);
  const double iD = rcp_any(q.D);
  // the lane's own coordinate: node m, component c
  const int m = ln.own / 3, c = ln.own - 3 * m;
  const auto pick = [&](const double *v) { return c == 0 ? v[0] : c == 1 ? v[1] : v[2]; };
  const double ac = pick(a), bc = pick(b), dc = pick(q.d);
  const double w = m == 0 ? 1.0 - q.s : m == 1 ? q.s : m == 2 ? q.t - 1.0 : -q.t;
  const double w1 = m == 0 ? 1.0 - s1 : m == 1 ? s1 : w;
  const double ms = m == 0 ? -1.0 : m == 1 ? 1.0 : 0.0, mt = m == 2 ? 1.0 : m == 3 ? -1.0 : 0.0;
  const double fs = fma(w, ac, ms * dc), ft = fma(-w, bc, mt * dc);
  q.tx = !tfree ? 0.0 : joint ? -fma(B, fs, A * ft) * iden : fma(w1, bc, -mt * pick(d1)) * iC;
  q.sx = !sfree ? 0.0 : fma(B, q.tx, -fs) * iA;
  // (the last term vanishes but for near-parallel segments, where t is the
  // closest point of s = 0 and f's derivative in t, -d b, is not zero)
  q.Dx = iD * fma(-dot3(q.d, b), q.tx, w * dc);
#pragma unroll
  for (int e = 0; e < 3; ++e) q.dx[e] = fma(a[e], q.sx, fma(-b[e], q.tx, e == c ? w : 0.0));
  const double ps = fma(0.5, fma(A, q.sx, -B * q.tx), fs), pt = fma(0.5, fma(C, q.tx, -B * q.sx), ft);
  // t's own second derivative for those: t = E / C, E = b r and C = b b, with b
  // = sum -mt_n x_n and r = sum rho_n x_n
  const bool curved = parallel && tfree;  // warp-uniform
  const double rho = m == 0 ? 1.0 : m == 2 ? -1.0 : 0.0, cx = -2.0 * mt * bc, ftC = -dot3(q.d, b) * iC;
#pragma unroll
  for (int k = 0; k < kHP; ++k) {
    const int i = ln.i[k], j = ln.j[k];
    const double wi = __shfl_sync(full, w, i), wj = __shfl_sync(full, w, j);
    double h = i % 3 == j % 3 ? wi * wj : 0.0;
    h = fma(__shfl_sync(full, ps, i), __shfl_sync(full, q.sx, j), h);
    h = fma(__shfl_sync(full, pt, i), __shfl_sync(full, q.tx, j), h);
    h = fma(__shfl_sync(full, q.sx, i), __shfl_sync(full, ps, j), h);
    h = fma(__shfl_sync(full, q.tx, i), __shfl_sync(full, pt, j), h);
    if (curved) {
      const double bi = -__shfl_sync(full, mt, i), bj = -__shfl_sync(full, mt, j);
      const double ri = __shfl_sync(full, rho, i), rj = __shfl_sync(full, rho, j);
      double tt = i % 3 == j % 3 ? fma(bi, rj, ri * bj) - 2.0 * q.t * bi * bj : 0.0;
      tt = fma(-__shfl_sync(full, q.tx, i), __shfl_sync(full, cx, j), tt);
      tt = fma(-__shfl_sync(full, cx, i), __shfl_sync(full, q.tx, j), tt);
      h = fma(ftC, tt, h);
    }
    q.gi[k] = __shfl_sync(full, q.Dx, i);
    q.gj[k] = __shfl_sync(full, q.Dx, j);
    q.h[k] = iD * fma(-q.gi[k], q.gj[k], h);
  }
  return q;
}

// Plain segment distance (same rule), for the candidate filter.
__device__ double segment_distance(const double *x) {
  double a[3], b[3], r[3];
  for (int c = 0; c < 3; ++c) {
    a[c] = x[3 + c] - x[c];
    b[c] = x[9 + c] - x[6 + c];
    r[c] = x[c] - x[6 + c];
  }
  const double A = a[0] * a[0] + a[1] * a[1] + a[2] * a[2];
  const double B = a[0] * b[0] + a[1] * b[1] + a[2] * b[2];
  const double Cc = b[0] * b[0] + b[1] * b[1] + b[2] * b[2];
  const double Dd = a[0] * r[0] + a[1] * r[1] + a[2] * r[2];
  const double Ee = b[0] * r[0] + b[1] * r[1] + b[2] * r[2];
  const double den = A * Cc - B * B;
  double s = den < 1e-12 * A * Cc ? 0.0 : fmin(fmax((B * Ee - Cc * Dd) / den, 0.0), 1.0);
  const double t = fmin(fmax((B * s + Ee) / Cc, 0.0), 1.0);
  s = fmin(fmax((B * t - Dd) / A, 0.0), 1.0);
  double dd = 0.0;
  for (int c = 0; c < 3; ++c) {
    const double d = r[c] + s * a[c] - t * b[c];
    dd += d * d;
  }
  return sqrt(dd);
}

// Eq. 10 with K1 = 15/delta: value and the first two derivatives in D.
__device__ void imc(double D, double C, double delta, double &e0, double &e1, double &e2) {
  if (D <= C - delta) {
    e0 = (C - D) * (C - D);
    e1 = -2.0 * (C - D);
    e2 = 2.0;
  } else if (D < C + delta) {
    const double K1 = 15.0 / delta;
    const double u = K1 * (C - D);
    const double sp = fmax(u, 0.0) + log1p(exp(-fabs(u)));
    const double sg = 1.0 / (1.0 + exp(-u));
    e0 = (sp / K1) * (sp / K1);
    e1 = -2.0 * sp * sg / K1;
    e2 = 2.0 * (sg * sg + sp * sg * (1.0 - sg));
  } else {
    e0 = e1 = e2 = 0.0;
  }
}

__device__ __forceinline__ unsigned long long cell_key(int cx, int cy, int cz) {
  return ((unsigned long long)(cx & 0x1fffff) << 42) | ((unsigned long long)(cy & 0x1fffff) << 21) |
         (unsigned long long)(cz & 0x1fffff);
}

__device__ __forceinline__ unsigned hash_key(unsigned long long k, unsigned mask) {
  k ^= k >> 33;
  k *= 0xff51afd7ed558ccdull;
  k ^= k >> 33;
  return (unsigned)k & mask;
}

__device__ __forceinline__ void edge_cell(const ContactArgs &a, int e, int c[3]) {
  const int ia = a.edge_a[e], ib = a.edge_b[e];
  for (int k = 0; k < 3; ++k) c[k] = (int)floor(0.5 * (a.q[ia + k] + a.q[ib + k]) * a.inv_cell);
}

}  // namespace

__global__ void k_cc_cells(ContactArgs a) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= a.ne) return;
  if (!a.sys_active[a.edge_sys[e]] || a.sys_kind[a.edge_sys[e]] != SOLVE_CONTACT) return;
  int c[3];
  edge_cell(a, e, c);
  const unsigned long long k = cell_key(c[0], c[1], c[2]);
  a.edge_key[e] = k;
  atomicAdd(a.bucket_count + hash_key(k, a.table_mask), 1);
}

// exclusive prefix sum of the bucket counts (one block of 1024 threads: a
// serial sum per thread, then a scan over the warps)
__global__ void __launch_bounds__(1024) k_cc_scan(ContactArgs a) {
  __shared__ int part[32];
  const int T = a.table_mask + 1, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int per = (T + blockDim.x - 1) / blockDim.x;
  const int b0 = min(T, tid * per), b1 = min(T, b0 + per);
  int sum = 0;
  for (int b = b0; b < b1; ++b) sum += a.bucket_count[b];
  int incl = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int v = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += v;
  }
  if (lane == 31) part[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    int w = part[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, w, o);
      if (lane >= o) w += v;
    }
    part[lane] = w;
  }
  __syncthreads();
  int run = incl - sum + (warp ? part[warp - 1] : 0);
  if (tid == (int)blockDim.x - 1) a.bucket_start[T] = run + sum;
  for (int b = b0; b < b1; ++b) {
    a.bucket_start[b] = run;
    a.bucket_fill[b] = run;
    run += a.bucket_count[b];
  }
}

__global__ void k_cc_fill(ContactArgs a) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= a.ne) return;
  if (!a.sys_active[a.edge_sys[e]] || a.sys_kind[a.edge_sys[e]] != SOLVE_CONTACT) return;
  const unsigned h = hash_key(a.edge_key[e], a.table_mask);
  a.bucket_edges[atomicAdd(a.bucket_fill + h, 1)] = e;
}

// A warp per edge: lanes 0-26 look up the neighbouring cells' buckets, then
// every lane takes candidates of the joint list (a segment distance is some
// 150 dependent FP64 instructions, so candidates side by side, not in turn).
__global__ void __launch_bounds__(128) k_cc_pairs(ContactArgs a) {
  const int e = (int)((blockIdx.x * (size_t)blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
  if (e >= a.ne) return;
  const int s = a.edge_sys[e];
  if (!a.sys_active[s] || a.sys_kind[s] != SOLVE_CONTACT) return;
  const unsigned full = 0xffffffffu;
  int c[3];
  edge_cell(a, e, c);
  double x[12];
  const int ia = a.edge_a[e], ib = a.edge_b[e];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    x[k] = a.q[ia + k];
    x[3 + k] = a.q[ib + k];
  }
  unsigned long long key = 0;
  int start = 0, cnt = 0;
  if (lane < 27) {
    key = cell_key(c[0] + lane % 3 - 1, c[1] + (lane / 3) % 3 - 1, c[2] + lane / 9 - 1);
    const unsigned h = hash_key(key, a.table_mask);
    start = a.bucket_start[h];
    cnt = a.bucket_start[h + 1] - start;
  }
  int incl = cnt;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int v = __shfl_up_sync(full, incl, o);
    if (lane >= o) incl += v;
  }
  const int total = __shfl_sync(full, incl, 31), excl = incl - cnt;
  for (int base = 0; base < total; base += 32) {
    // candidate base + lane: the cell whose range of the joint list holds it
    const int m = base + lane;
    int cell = 0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const int v = __shfl_sync(full, excl, min(cell + o, 31));
      if (cell + o < 32 && v <= m) cell += o;
    }
    const unsigned long long ck = __shfl_sync(full, key, cell);
    const int at = __shfl_sync(full, start, cell) + m - __shfl_sync(full, excl, cell);
    if (m >= total) continue;
    const int f = a.bucket_edges[at];
    if (f <= e || a.edge_key[f] != ck || a.edge_sys[f] != s) continue;
    if (abs(a.edge_idx[f] - a.edge_idx[e]) <= 2) continue;  // excluded pairs
    const int ja = a.edge_a[f], jb = a.edge_b[f];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      x[6 + k] = a.q[ja + k];
      x[9 + k] = a.q[jb + k];
    }
    const double C = a.edge_h[e] + a.edge_h[f];
    const double D = segment_distance(x);
    if (!(D > 0.0)) {  // Eq. 10 undefined: interpenetration
      atomicCAS(a.sys_status + s, 0, (int)DM_ERR_PENETRATION);
      continue;
    }
    if (D < C + a.delta) {
      const int p = atomicAdd(a.npairs, 1);
      if (p < a.pair_cap) {
        a.pairs[2 * p] = e;
        a.pairs[2 * p + 1] = f;
      } else {
        atomicCAS(a.sys_status + s, 0, (int)DM_ERR_DEGENERATE);
      }
    }
  }
}

// The tiles of entries (r, c) and (c, r) of a contact system's matrix are in use.
__device__ __forceinline__ void mark_tile(const ContactArgs &a, int s, int n, int r, int c) {
  const int nt = (n + kNB - 1) / kNB, I = r / kNB, J = c / kNB;
  uint8_t *nz = a.nz + a.sys_nz0[s];
  nz[(size_t)I * nt + J] = 1;
  nz[(size_t)J * nt + I] = 1;
}

// A warp per pair; the launch's warps stride over the pairs found.
__global__ void __launch_bounds__(64) k_cc_terms(ContactArgs a) {
  const int np = min(*a.npairs, a.pair_cap), lane = threadIdx.x & 31;
  const int nwarp = (int)(gridDim.x * (blockDim.x >> 5));
  HLane ln;
  ln.load(lane);
  for (int p = (int)(blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)); p < np; p += nwarp) {
    const int e = a.pairs[2 * p], f = a.pairs[2 * p + 1];
    const int s = a.edge_sys[e];
    const int nodes[4] = {a.edge_a[e], a.edge_b[e], a.edge_a[f], a.edge_b[f]};
    double x[12];
#pragma unroll
    for (int n = 0; n < 4; ++n)
#pragma unroll
      for (int k = 0; k < 3; ++k) x[3 * n + k] = a.q[nodes[n] + k];
    auto dof = [&](int i) { return (i < 6 ? (i < 3 ? nodes[0] : nodes[1]) : (i < 9 ? nodes[2] : nodes[3])) + i % 3; };
    const Distance q = pair_distance(x, ln);
    const double C = a.edge_h[e] + a.edge_h[f];
    double e0, e1, e2;
    imc(q.D, C, a.delta, e0, e1, e2);
    const double kc = a.kc;
    const int d0 = a.sys_dof0[s], n = a.sys_ndof[s];
    double *M = a.dense + a.sys_dense0[s];
    const bool mine = lane < 12 && !a.fixed[dof(ln.own)];
    if (mine) atomicAdd(a.fc + dof(ln.own), -kc * e1 * q.Dx);  // F = -dE/dq (Eq. 11)
#pragma unroll
    for (int k = 0; k < kHP; ++k) {
      const int di = dof(ln.i[k]), dj = dof(ln.j[k]);
      if (!ln.on[k] || a.fixed[di] || a.fixed[dj]) continue;
      const double hv = kc * (e1 * q.h[k] + e2 * q.gi[k] * q.gj[k]);
      const int r = di - d0, c = dj - d0;
      atomicAdd(M + (size_t)r * n + c, hv);
      if (r != c) atomicAdd(M + (size_t)c * n + r, hv);
      mark_tile(a, s, n, r, c);
    }
    if (a.mu == 0.0) continue;
    // Friction at the closest points (Eq. 12-13): u = tangential relative
    // velocity of the closest points with the implicit velocities
    // (x - x_n)/dt; F_a = -mu gamma(|u|) u/|u| |F_con| on edge a, -F_a on
    // edge b, spread by the closest-point weights; |F_con| = k_c |dE/dD|.
    // Derivatives by first-order dual numbers; at |u| = 0 the limit
    // gamma/|u| -> K2/2 of the smooth law.
    const D1 sD = {q.s, q.sx}, tD = {q.t, q.tx}, Dd = {q.D, q.Dx}, one = d1_const(1.0);
    const D1 iD = d1_apply(Dd, 1.0 / Dd.v, -1.0 / (Dd.v * Dd.v));
    const double idt = 1.0 / a.dt;
    D1 nrm[3], ur[3], u[3], Fa[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      nrm[c] = D1{q.d[c], q.dx[c]} * iD;
      D1 v[4];
#pragma unroll
      for (int m = 0; m < 4; ++m)
        v[m] = {idt * (x[3 * m + c] - a.qn[nodes[m] + c]), ln.own == 3 * m + c ? idt : 0.0};
      ur[c] = ((one - sD) * v[0] + sD * v[1]) - ((one - tD) * v[2] + tD * v[3]);
    }
    const D1 vn = ur[0] * nrm[0] + ur[1] * nrm[1] + ur[2] * nrm[2];
#pragma unroll
    for (int c = 0; c < 3; ++c) u[c] = ur[c] - vn * nrm[c];
    const D1 s2 = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
    // |F_con| = -k_c e1 (e1 <= 0 in contact), derivative -k_c e2 grad D
    const D1 fn = d1_apply(Dd, -kc * e1, -kc * e2);
    D1 coef;
    if (s2.v > 0.0) {
      const double sg = sqrt(s2.v);
      const D1 sig = d1_apply(s2, sg, 0.5 / sg);
      const double ex = exp(-a.K2 * sg);
      const double gam = 2.0 / (1.0 + ex) - 1.0;
      const double dgam = 2.0 * a.K2 * ex / ((1.0 + ex) * (1.0 + ex));
      // gamma(sigma) / sigma
      const D1 gs = d1_apply(sig, gam / sg, (dgam * sg - gam) / (sg * sg));
      coef = (-a.mu) * (fn * gs);
    } else {
      coef = (-0.5 * a.mu * a.K2) * fn;
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) Fa[c] = coef * u[c];
    const D1 wgt[4] = {one - sD, sD, tD - one, d1_const(0.0) - tD};
#pragma unroll
    for (int m = 0; m < 4; ++m)
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const int i = nodes[m] + c;
        if (a.fixed[i]) continue;
        const D1 F = wgt[m] * Fa[c];
        if (lane == 0) atomicAdd(a.fc + i, F.v);
        // J = -dF/dq, one column per lane (its tile is marked above)
        if (mine && F.g != 0.0) atomicAdd(M + (size_t)(i - d0) * n + (dof(ln.own) - d0), -F.g);
      }
  }
}

// Ground contact and friction of the nodes of contact systems (Eq. 10-13,
// the node terms of k_nodes: force F and -dF/dx, nonsymmetric with friction)
// into their contact force and dense matrix, one thread per node; after
// k_cc_terms in stream order (no concurrent writer to these entries).
__global__ void k_cc_ground(ContactArgs a, const int32_t *node_dof, const int32_t *node_sys,
                            const double *nt) {
  const int v = blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= a.nn) return;
  const int s = node_sys[v];
  // residual phase of the round: the line search has not decided yet (an
  // earlier round's backtracking decision must not drop the force)
  if (!a.sys_active[s] || a.sys_kind[s] != SOLVE_CONTACT) return;
  const int d = node_dof[v], d0 = a.sys_dof0[s], n = a.sys_ndof[s], NN = a.nn;
  double *M = a.dense + a.sys_dense0[s];
#pragma unroll
  for (int r = 0; r < 3; ++r) {
    if (a.fixed[d + r]) continue;
    a.fc[d + r] += nt[r * NN + v];
#pragma unroll
    for (int c = 0; c < 3; ++c)
      if (!a.fixed[d + c]) {
        M[(size_t)(d + r - d0) * n + (d + c - d0)] += nt[(3 + 3 * r + c) * NN + v];
        mark_tile(a, s, n, d + r - d0, d + c - d0);
      }
  }
}

// The rod's band (lower, symmetric) into the dense matrix of each contact
// system, one thread per DOF row, and the right-hand side y = -f.
__global__ void k_cc_band(ContactArgs a, const double *f, double *y) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= a.nd) return;
  const int s = a.dof_sys[i];
  if (!a.sys_active[s] || a.sys_kind[s] != SOLVE_CONTACT) return;
  if (a.ls_action && a.ls_action[s] == 1) return;
  const int d0 = a.sys_dof0[s], n = a.sys_ndof[s], r = i - d0;
  double *M = a.dense + a.sys_dense0[s];
  y[i] = -f[i];
  // the row's entries, then what is there already, all loads side by side (one
  // after the other a launch of 1999 rows took 18 us, now 8)
  double v[11], lo[11], up[11];
#pragma unroll
  for (int d = 0; d < 11; ++d) v[d] = d <= r ? a.band[(size_t)d * a.nd + i] : 0.0;
#pragma unroll
  for (int d = 0; d < 11; ++d)
    if (d == 0 || v[d] != 0.0) {
      lo[d] = M[(size_t)r * n + (r - d)];
      up[d] = M[(size_t)(r - d) * n + r];
    }
  int reach = 0;  // the farthest nonzero diagonal: no tile is marked beyond it
#pragma unroll
  for (int d = 0; d < 11; ++d)
    if (d == 0 || v[d] != 0.0) {
      M[(size_t)r * n + (r - d)] = lo[d] + v[d];
      if (d > 0) M[(size_t)(r - d) * n + r] = up[d] + v[d];
      reach = d;
    }
  mark_tile(a, s, n, r, r);
  if ((r - reach) / kNB != r / kNB) mark_tile(a, s, n, r, r - reach);
}

// Zeroes the tiles that the last factorisation of each contact system used,
// and their marks: a block per tile row.
__global__ void __launch_bounds__(256) k_cc_clear(ContactArgs a) {
  const int s = a.contact_sys[blockIdx.x];
  const int n = a.sys_ndof[s], nt = (n + kNB - 1) / kNB, I = blockIdx.y;
  if (I >= nt) return;
  uint8_t *nz = a.nz + a.sys_nz0[s] + (size_t)I * nt;
  double *M = a.dense + a.sys_dense0[s];
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  for (int b = 0; b < nt; b += 32)
    for (unsigned on = __ballot_sync(0xffffffffu, b + tx < nt && nz[b + tx] != 0); on; on &= on - 1) {
      const int c = (b + __ffs(on) - 1) * kNB + tx;
#pragma unroll
      for (int r = ty; r < kNB; r += 8)
        if (I * kNB + r < n && c < n) M[(size_t)(I * kNB + r) * n + c] = 0.0;
    }
  __syncthreads();
  for (int J = threadIdx.x; J < nt; J += blockDim.x) nz[J] = 0;
}

// --- blocked LU of the contact systems (no pivoting), spread over the GPU ---
//
// The rods' Jacobian with the contact blocks is sparse in 32 x 32 tiles: the
// band along each rod, the tiles that touching edges couple, and the fill
// between them (its pattern is symmetric).  `nz` marks the tiles in use.
//   k_lu_order   orders the elimination by levels from the pattern alone, a
//                block per system: a level takes up to eight tile columns
//                (fronts) of the fewest neighbours (one more allowed), no two
//                of them coupled, the outermost first; it lists each front's
//                remaining neighbours and marks the fill.  Rods eliminate from
//                both ends, separate rods side by side.
//   k_lu         all levels in one launch, the chip's blocks shared among the
//                systems, which each meet at their own counter twice a level:
//                panel -- the fronts' diagonal tiles are factored (in every
//                block, which saves a meeting; a front's first block keeps its
//                tile in `lud`) and the tiles below (L = A U^-1) and right of
//                it (U = L^-1 A) and the right-hand side solved, a warp per row
//                or column: 32 steps of a shuffle and one FMA, the pivots'
//                reciprocals moved out of the chain into the rows of U;
//                update -- L(I,k) U(k,J) subtracted from the tiles (I, J) of a
//                front's neighbours, in quarters of 16 x 16 (an SM's FP64 pipe
//                takes 9 us for a whole tile), and the right-hand side's part.
// k_cc_decide takes the Newton decision of each contact system first;
// k_cc_subst runs the backward substitution, level by level, and updates q.
// Bound by the chain of levels: a 500-node coil (63 tile columns, up to 12
// neighbours) has 24, a gripper of five 60-node fingers (38) has 8.  The
// diagonal tile's 32 dependent columns run on four warps (one per SM
// partition).
// Measured (GB300): a level 42 k cycles and up -- the diagonal tile 23 k, its
// solves 7 k, the two meetings 3 k each, the update from 6 k (few tiles) to 85 k
// (2400 quarters: the FP64 pipes' rate); factorisation and solve of the coil 2.8
// -> 1.0 ms, of four grippers 1.8 -> 0.4 ms (before: tile columns in their
// order, two launches for each; before that, the full bandwidth: 9 and 21 ms).

__global__ void k_cc_decide(ContactArgs a, SolveArgs v) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= a.n_contact) return;
  const int s = a.contact_sys[c];
  int go = 0;
  if (v.sys_active[s] && v.ls_action && v.ls_action[s] == 1) {
    atomicAdd(&v.ctrl[0], 1);  // backtracking: no solve this round
  } else if (v.sys_active[s]) {
    const double res = __longlong_as_double((long long)v.sys_res[s]);
    int st = v.sys_status[s];
    if (st == 0 && isnan(res)) st = DM_ERR_NONFINITE;
    if (st == 0 && res <= v.tol) {
      v.sys_active[s] = 0;
    } else {
      if (st == 0 && v.sys_iters[s] >= v.max_iter) st = DM_ERR_NOT_CONVERGED;
      if (st != 0) {
        v.sys_status[s] = st;
        v.sys_active[s] = 0;
        atomicAdd(&v.ctrl[1], 1);
        atomicMin(&v.ctrl[2], s);
      } else {
        go = 1;
      }
    }
  }
  a.cgo[c] = go;
  a.cbad[c] = 0;
}

constexpr int kMaxTiles = 1024;  // tile columns of a system (its matrix is at most 8 GB)
constexpr int kFronts = 8;       // tile columns eliminated at once
constexpr unsigned kDegreeSlack = 1;
static_assert(kLevelInts > 1 + 2 * kFronts + 1, "a level's record");
// a level's record: number of fronts, their tile columns, their neighbours'
// counts (zero fronts: past the last level); the first one ends with the
// number of levels

struct Level {
  int nf, k[kFronts], m[kFronts];
};

// Bit rows of the pattern in shared memory, word w of tile i at row[w nt + i];
// a thread per tile.
__global__ void __launch_bounds__(1024) k_lu_order(ContactArgs a) {
  const int c = blockIdx.x;
  if (!a.cgo[c]) return;
  const int s = a.contact_sys[c], n = a.sys_ndof[s], nt = (n + kNB - 1) / kNB, W = (nt + 31) / 32;
  extern __shared__ unsigned row[];
  __shared__ unsigned rem[kMaxTiles / 32], best[2][kFronts][32];
  __shared__ int levels;
  int32_t *lev = a.lu_level + (size_t)c * a.max_tiles * kLevelInts;
  uint8_t *nz = a.nz + a.sys_nz0[s];
  uint16_t *adj = a.lu_adj + a.sys_nz0[s];
  const int i = threadIdx.x, lane = i & 31;
#pragma unroll 4
  for (int e = i >> 5; e < nt * W; e += blockDim.x >> 5) {
    const int r = e / W, J = (e - r * W) * 32 + lane;
    const unsigned bits = __ballot_sync(0xffffffffu, J < nt && J != r && nz[(size_t)r * nt + J] != 0);
    if (lane == 0) row[(e - r * W) * nt + r] = bits;
  }
  if (i < W) rem[i] = i == W - 1 && (nt & 31) ? (1u << (nt & 31)) - 1u : 0xffffffffu;
  if (i == 0) a.lu_bar[c] = 0;
  __syncthreads();
  int l = 0;
  if (i < 32 * W) {  // (the other warps wait at the end)
    const auto meet = [&] { asm volatile("bar.sync 1, %0;" ::"r"(32 * W) : "memory"); };
    const auto bit = [&](int p) { return i < nt && ((row[(p >> 5) * nt + i] >> (p & 31)) & 1u); };  // i ~ p
    for (;; ++l) {
      // fewest remaining neighbours, then farthest from the middle, then first
      unsigned key = 0xffffffffu;
      const bool alive = i < nt && ((rem[i >> 5] >> lane) & 1u);
      if (alive) {
        unsigned deg = 0;
        for (int w = 0; w < W; ++w) deg += __popc(row[w * nt + i] & rem[w]);
        key = (deg << 21) | ((unsigned)(1024 - abs(2 * i - (nt - 1))) << 10) | (unsigned)i;
      }
      int nf = 0, pick[kFronts];
      unsigned lim = 0;
#pragma unroll
      for (int f = 0; f < kFronts; ++f) {
        if (nf < f) break;
        unsigned b = __reduce_min_sync(0xffffffffu, key);
        if (lane == 0) best[l & 1][f][i >> 5] = b;
        meet();
        for (int w = 0; w < W; ++w) b = min(b, best[l & 1][f][w]);
        if (f == 0) lim = (b >> 21) + kDegreeSlack;
        if (b == 0xffffffffu || (b >> 21) > lim) break;
        pick[f] = (int)(b & 1023u);
        nf = f + 1;
        if (i == pick[f] || bit(pick[f])) key = 0xffffffffu;
      }
      if (nf == 0) break;
      meet();  // (rem read)
#pragma unroll
      for (int f = 0; f < kFronts; ++f)
        if (f < nf && i == pick[f]) atomicAnd(&rem[i >> 5], ~(1u << lane));
      meet();
      const bool left = alive && ((rem[i >> 5] >> lane) & 1u);
#pragma unroll
      for (int f = 0; f < kFronts; ++f) {
        if (f >= nf) break;
        const int p = pick[f];
        if (i == p) {
          int m = 0;
          for (int w = 0; w < W; ++w) m += __popc(row[w * nt + p] & rem[w]);
          lev[l * kLevelInts + 1 + f] = p;
          lev[l * kLevelInts + 1 + kFronts + f] = m;
        }
        if (left && bit(p)) {
          int rank = 0;
          for (int w = 0; w < W; ++w) {
            const unsigned x = row[w * nt + p] & rem[w];
            if (w < i >> 5) rank += __popc(x);
            if (w == i >> 5) rank += __popc(x & ((1u << lane) - 1u));
            row[w * nt + i] |= w == i >> 5 ? x & ~(1u << lane) : x;  // fill (own row only)
          }
          adj[(size_t)p * nt + rank] = (uint16_t)i;
        }
      }
      if (i == 0) lev[l * kLevelInts] = nf;
      meet();
    }
  }
  if (i == 0) levels = l;
  __syncthreads();
  l = levels;
  if (i == 0) lev[kLevelInts - 1] = l;
  for (int x = l + i; x < a.max_tiles; x += blockDim.x) lev[x * kLevelInts] = 0;
  for (int e = i >> 5; e < nt * W; e += blockDim.x >> 5) {
    const int r = e / W, J = (e - r * W) * 32 + lane;
    if ((row[(e - r * W) * nt + r] >> lane) & 1u) nz[(size_t)r * nt + J] = 1;
  }
}

// LU of the 32 x 32 tile D (shared memory; four zero rows behind it) by warps
// 0-3; every thread of the block calls it.  Leaves the unit factors (L below
// the diagonal, U over its pivots above it) in D and the pivots' reciprocals in
// R.  Column j: rows j + 1 + warp, + 4, ..., a lane per column; no branches (the
// zero rows take what is too much, and reciprocals are those of the integer
// pipe): 705 cycles a column, 496 of them the chain of product, first row,
// exchange, reciprocal and barrier.  False if a pivot was outside the
// reciprocal's range; `exact`: any pivot, by division (thrice the time).
template <bool exact>
__device__ __forceinline__ bool factor_tile(double (*D)[kNB + 1], double *R) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (warp < 4) {
    double r = exact ? 1.0 / D[0][0] : rcp_int(D[0][0]);
    if (warp == 0 && lane == 0) R[0] = r;
#pragma unroll
    for (int p = 0; p < 8; ++p) {
      const int NT = 8 - p;  // rows of a warp in columns 4 p .. 4 p + 3
#pragma unroll 1
      for (int j = 4 * p; j < (p < 7 ? 4 * p + 4 : kNB - 1); ++j) {
        const int i0 = j + 1 + warp;
        double m[8], d[8];
#pragma unroll
        for (int t = 0; t < NT; ++t) {
          m[t] = D[i0 + 4 * t][j];
          d[t] = D[i0 + 4 * t][lane];
        }
        const double x = D[j][lane] * r, u = lane > j ? x : 0.0;
        d[0] = fma(-m[0], u, d[0]);
        const double piv = __shfl_sync(0xffffffffu, d[0], j + 1);  // (warp 0's)
        const double rn = exact ? 1.0 / piv : rcp_int(piv);
#pragma unroll
        for (int t = 1; t < NT; ++t) d[t] = fma(-m[t], u, d[t]);
#pragma unroll
        for (int t = 0; t < NT; ++t) D[i0 + 4 * t][lane] = d[t];
        if (warp == 0 && lane == 0) R[j + 1] = rn;
        asm volatile("bar.sync 1, 128;" ::: "memory");
        r = R[j + 1];
      }
    }
  }
  __syncthreads();
  return exact || !__syncthreads_or(warp == 0 && !rcp64_in_range(D[lane][lane]));
}

// Why a system's factorisation stopped (cbad): a pivot that is zero or not
// finite, or a wait between its blocks that ran out, which goes before.
constexpr int kLuZeroPivot = 1, kLuTimeout = 2;

// The blocks of a system meet (all of them are resident: a cooperative launch
// when there are several): a release by thread 0 after the block's barrier, an
// acquire before the next; work between the two calls needs nothing of the
// other blocks.  lu_wait: false if a wait ran out, or (`check`) at a zero pivot.
constexpr int kSpinLimit = 1 << 22;  // a few seconds
__device__ __forceinline__ void lu_arrive(int32_t *bar, int blocks, int &target) {
  __syncthreads();
  target += blocks;
  if (threadIdx.x == 0 && blocks > 1) asm volatile("red.release.gpu.global.add.s32 [%0], 1;" ::"l"(bar) : "memory");
}
__device__ __forceinline__ bool lu_wait(int32_t *bar, int32_t *bad, int blocks, int target, bool check) {
  __shared__ int ok;
  if (threadIdx.x == 0) {
    int fine = 1;
    if (blocks > 1) {
      int seen = 0, spins = 0;
      do {
        asm volatile("ld.acquire.gpu.s32 %0, [%1];" : "=r"(seen) : "l"(bar) : "memory");
      } while (seen < target && ++spins < kSpinLimit);
      if (seen < target) {
        atomicMax(bad, kLuTimeout);
        fine = 0;
      }
    }
    // (a zero pivot is written before the barrier that follows its panel, and
    // none while any block is between that barrier and the next)
    if (check && *reinterpret_cast<volatile int32_t *>(bad)) fine = 0;
    ok = fine;
  }
  __syncthreads();
  return ok != 0;
}

// Factorisation of all levels: gridDim.y blocks per system (a grid takes more
// systems along x than along y: 65535).
constexpr int kLuThreads = 512;
__global__ void __launch_bounds__(kLuThreads, 1) k_lu(ContactArgs a, double *yall) {
  const int c = blockIdx.x, block = blockIdx.y;
  if (!a.cgo[c]) return;
  const int s = a.contact_sys[c];
  const int n = a.sys_ndof[s], nt = (n + kNB - 1) / kNB;
  __shared__ Level lv;
  __shared__ double D[kNB + 4][kNB + 1], R[kNB];
  __shared__ double Lh[2][16][kNB + 1];
  __shared__ double Uh[2][kNB][16 + 1];
  __shared__ uint16_t list[kFronts][kMaxTiles];
  __shared__ unsigned reach[kMaxTiles / 4];  // per tile, a byte: the fronts it neighbours
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int half = tid >> 8, ty = (tid & 255) >> 4, tx = tid & 15;  // of the update
  double (*Ls)[kNB + 1] = Lh[half], (*Us)[16 + 1] = Uh[half];
  double *A = a.dense + a.sys_dense0[s], *y = yall + a.sys_dof0[s];
  const uint16_t *adj = a.lu_adj + a.sys_nz0[s];
  const int32_t *lev = a.lu_level + (size_t)c * a.max_tiles * kLevelInts;
  const int levels = lev[kLevelInts - 1];
  const auto fronts = [&](int I) { return (reach[I >> 2] >> (8 * (I & 3))) & 0xffu; };
  const int blocks = gridDim.y;
  int target = 0, items = 0, vecs = 0;
  // level l's record, its fronts' neighbours and who neighbours whom
  const auto load_level = [&](int l) {
    if (tid < 1 + 2 * kFronts) reinterpret_cast<int *>(&lv)[tid] = lev[l * kLevelInts + tid];
    for (int e = tid; e < (nt + 3) / 4; e += kLuThreads) reach[e] = 0;
    __syncthreads();
    items = vecs = 0;
    for (int f = 0; f < lv.nf; ++f) {
      const uint16_t *src = adj + (size_t)lv.k[f] * nt;
      for (int e = tid; e < lv.m[f]; e += kLuThreads) {
        const int I = src[e];
        list[f][e] = (uint16_t)I;
        atomicOr(&reach[I >> 2], 1u << (8 * (I & 3) + f));
      }
      items += 4 * lv.m[f] * lv.m[f];
      vecs += lv.m[f];
    }
    __syncthreads();
  };
  load_level(0);
  for (int l = 0; l < levels; ++l) {
    const int nf = lv.nf;

    // panel: the blocks are dealt to the fronts by their vectors (rows of L,
    // columns of U, the right-hand side: a warp each), so that a block factors
    // one diagonal tile; fronts in turn when there are fewer blocks
    for (int f = 0, start = 0; f < nf; ++f) {
      const int k = lv.k[f], m = lv.m[f], k0 = k * kNB, nb = min(kNB, n - k0), vec = 2 * kNB * m + 1;
      int part = 0, parts = 1;
      if (blocks >= nf) {
        parts += (blocks - nf) * vec / (2 * kNB * vecs + nf);
        part = block - start;
        start += parts;
        if (part < 0 || part >= parts) continue;
      } else if (f % blocks != block) {
        continue;
      }
      const int each = min((vec + parts - 1) / parts, kLuThreads / 32);  // vectors of a block at a time
      if (part * each >= vec) continue;
      const auto load = [&] {  // the identity beyond the matrix
        __syncthreads();
#pragma unroll
        for (int t = 0; t < kNB * 32 / kLuThreads; ++t) {
          const int i = warp + kLuThreads / 32 * t;
          D[i][lane] = i < nb && lane < nb ? A[(size_t)(k0 + i) * n + k0 + lane] : i == lane ? 1.0 : 0.0;
        }
        if (warp < 4) D[kNB + warp][lane] = 0.0;
        __syncthreads();
      };
      load();
      if (!factor_tile<false>(D, R)) {
        load();
        factor_tile<true>(D, R);
        if (warp == 0 && zero_or_nonfinite(D[lane][lane])) atomicMax(a.cbad + c, kLuZeroPivot);
        __syncthreads();
      }
      const double rl = R[lane];
#pragma unroll
      for (int t = 0; t < kNB * 32 / kLuThreads; ++t) {
        const int i = warp + kLuThreads / 32 * t;
        D[i][lane] = lane == i ? 1.0 : D[i][lane] * (lane < i ? rl : R[i]);
      }
      __syncthreads();
      if (part == 0) {
        double *out = a.lud + (size_t)(a.sys_dof0[s] + k0) * kNB;
#pragma unroll
        for (int t = 0; t < kNB * 32 / kLuThreads; ++t) {
          const int i = warp + kLuThreads / 32 * t;
          if (i < nb) out[i * kNB + lane] = i == lane ? R[i] : D[i][lane];
        }
      }
      for (int g = part * each + warp; g < vec && warp < each; g += parts * each) {
        if (g < kNB * m) {  // a row of L: x U = a, w_j = x_j d_j
          const int row = list[f][g / kNB] * kNB + g % kNB;
          if (row >= n) continue;
          double *p = A + (size_t)row * n + k0 + lane;
          double w = lane < nb ? *p : 0.0;
#pragma unroll
          for (int j = 0; j < kNB - 1; ++j) {
            const double wj = __shfl_sync(0xffffffffu, w, j);
            if (lane > j) w = fma(-wj, D[j][lane], w);
          }
          if (lane < nb) *p = w * R[lane];
        } else {  // a column of U, or the right-hand side: L x = a (unit lower)
          const int h = g - kNB * m;
          const bool rhs = h == kNB * m;
          const int col = rhs ? 0 : list[f][h / kNB] * kNB + h % kNB;
          if (col >= n) continue;
          double *p = rhs ? y + k0 + lane : A + (size_t)(k0 + lane) * n + col;
          double w = lane < nb ? *p : 0.0;
#pragma unroll
          for (int j = 0; j < kNB - 1; ++j) {
            const double wj = __shfl_sync(0xffffffffu, w, j);
            if (lane > j) w = fma(-wj, D[lane][j], w);
          }
          if (lane < nb) *p = w;
        }
      }
    }
    if (l + 1 == levels) return;  // (the last level has no neighbours left)
    lu_arrive(a.lu_bar + c, blocks, target);
    if (!lu_wait(a.lu_bar + c, a.cbad + c, blocks, target, true)) return;

    // update, by half a block: quarter items (16 x 16 of a tile), front by front,
    // then the right-hand side's rows; a tile or row of several fronts belongs to the
    // first, which takes the others' parts along
    for (int f = 0, base = 0, it = block + half * blocks; it < items + vecs; it += 2 * blocks) {
      if (it >= items) {  // right-hand side: a lane per term
        int g = it - items, fv = 0;
        while (g >= lv.m[fv]) g -= lv.m[fv++];
        const int I = list[fv][g];
        const unsigned on = fronts(I);
        if (__ffs(on) - 1 != fv) continue;
        for (int r = warp & 7; r < kNB; r += 8) {
          const int row = I * kNB + r;
          if (row >= n) break;
          double v = 0.0;
          for (unsigned q = on; q; q &= q - 1) {
            const int k0 = lv.k[__ffs(q) - 1] * kNB;
            if (lane < n - k0) v = fma(A[(size_t)row * n + k0 + lane], y[k0 + lane], v);
          }
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
          if (lane == 0) y[row] -= v;
        }
        continue;
      }
      while (it >= base + 4 * lv.m[f] * lv.m[f]) base += 4 * lv.m[f] * lv.m[f], ++f;
      const int q = (it - base) & 3, t = (it - base) >> 2, ti = t / lv.m[f], tj = t - ti * lv.m[f];
      const int I = list[f][ti], J = list[f][tj];
      const int r0 = I * kNB + 16 * (q >> 1), c0 = J * kNB + 16 * (q & 1);
      const unsigned on = fronts(I) & fronts(J);
      if (__ffs(on) - 1 != f || r0 >= n || c0 >= n) continue;
      if (a.lu_flops && (tid & 255) == 0)
        atomicAdd(a.lu_flops, 2ull * (unsigned long long)(min(16, n - r0) * min(16, n - c0) * kNB * __popc(on)));
      const bool in = r0 + ty < n && c0 + tx < n;
      double *p = A + (size_t)(r0 + ty) * n + c0 + tx;
      const double old = in ? *p : 0.0;
      double acc = 0.0;
      for (unsigned qf = on; qf; qf &= qf - 1) {
        const int k0 = lv.k[__ffs(qf) - 1] * kNB, nb = min(kNB, n - k0);
        asm volatile("bar.sync %0, 256;" ::"r"(2 + half) : "memory");
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const int i = (warp & 7) + 8 * e, mm = lane;
          Ls[i][mm] = r0 + i < n && mm < nb ? A[(size_t)(r0 + i) * n + k0 + mm] : 0.0;
          const int u = ty + 16 * e;
          Us[u][tx] = c0 + tx < n && u < nb ? A[(size_t)(k0 + u) * n + c0 + tx] : 0.0;
        }
        asm volatile("bar.sync %0, 256;" ::"r"(2 + half) : "memory");
#pragma unroll
        for (int mm = 0; mm < kNB; ++mm) acc = fma(Ls[ty][mm], Us[mm][tx], acc);
      }
      if (in) *p = old - acc;
    }
    lu_arrive(a.lu_bar + c, blocks, target);
    load_level(l + 1);  // (its own shared memory only)
    if (!lu_wait(a.lu_bar + c, a.cbad + c, blocks, target, false)) return;
  }
}

// In-place transpose of the contact systems' matrices (for the adjoint's
// J^T solve): a block per tile row, the tiles on and right of the diagonal.
__global__ void __launch_bounds__(256) k_cc_transpose(ContactArgs a) {
  const int s = a.contact_sys[blockIdx.x];
  const int n = a.sys_ndof[s], nt = (n + kNB - 1) / kNB, I = blockIdx.y;
  if (I >= nt) return;
  const uint8_t *nz = a.nz + a.sys_nz0[s] + (size_t)I * nt;
  double *A = a.dense + a.sys_dense0[s];
  for (int J = I; J < nt; ++J) {
    if (!nz[J]) continue;
    for (int e = threadIdx.x; e < kNB * kNB; e += blockDim.x) {
      const int i = I * kNB + e / kNB, j = J * kNB + e % kNB;
      if (i >= j || i >= n || j >= n) continue;
      const double x = A[(size_t)i * n + j];
      A[(size_t)i * n + j] = A[(size_t)j * n + i];
      A[(size_t)j * n + i] = x;
    }
  }
}

// Backward substitution U x = z of each contact system, q += x: a cluster of
// blocks per system, levels from the last one up; the level's fronts are dealt
// to a block's warps, a front's tiles to the blocks (eight columns at a time,
// lane = row); a front's own block adds the blocks' sums and solves the
// diagonal tile.
constexpr int kSubstWarps = 16;
__global__ void __launch_bounds__(32 * kSubstWarps) k_cc_subst(ContactArgs a, SolveArgs v) {
  cooperative_groups::cluster_group cluster = cooperative_groups::this_cluster();
  const int blocks = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  const int c = blockIdx.x / blocks;
  const int s = a.contact_sys[c];
  if (!a.cgo[c]) return;
  if (a.cbad[c]) {
    if (rank == 0 && threadIdx.x == 0) {
      v.sys_status[s] = a.cbad[c] == kLuTimeout ? DM_ERR_CUDA : DM_ERR_DEGENERATE;
      v.sys_active[s] = 0;
      atomicAdd(&v.ctrl[1], 1);
      atomicMin(&v.ctrl[2], s);
    }
    return;
  }
  const int d0 = v.sys_dof0[s], n = v.sys_ndof[s], nt = (n + kNB - 1) / kNB;
  const double *A = a.dense + a.sys_dense0[s];
  const uint16_t *adj = a.lu_adj + a.sys_nz0[s];
  const int32_t *lev = a.lu_level + (size_t)c * a.max_tiles * kLevelInts;
  double *y = v.dq + d0;
  __shared__ double part[kSubstWarps][kNB + 1], tot[kFronts][kNB];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int l = lev[kLevelInts - 1] - 1; l >= 0; --l) {
    const int32_t *rec = lev + l * kLevelInts;
    const int nf = rec[0], sh = nf <= 1 ? 0 : 32 - __clz(nf - 1);  // fronts, rounded up to 2^sh
    const int per = kSubstWarps >> sh, f = warp / per, slot = warp - f * per;
    const bool on = f < nf, first = on && slot == 0, own = first && f % blocks == rank;
    const int k = on ? rec[1 + f] : 0, m = on ? rec[1 + kFronts + f] : 0;
    const int k0 = k * kNB, nb = min(kNB, n - k0);
    double sum = 0.0;
    for (int t = rank + blocks * slot; t < 4 * m; t += blocks * per) {
      const int j0 = adj[(size_t)k * nt + (t >> 2)] * kNB + 8 * (t & 3);
      double x[8], z[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const bool in = lane < nb && j0 + j < n;
        x[j] = in ? A[(size_t)(k0 + lane) * n + j0 + j] : 0.0;
        z[j] = in ? y[j0 + j] : 0.0;
      }
#pragma unroll
      for (int j = 0; j < 8; ++j) sum = fma(x[j], z[j], sum);
    }
    part[warp][lane] = sum;
    // the lane's row of U over its pivot
    const double *Dk = a.lud + (size_t)(d0 + k0) * kNB;
    double urow[kNB], r = 0.0, z = 0.0;
    if (own) {
#pragma unroll
      for (int j = 0; j < kNB; ++j) urow[j] = lane < nb && j > lane && j < nb ? Dk[lane * kNB + j] : 0.0;
      r = lane < nb ? Dk[lane * kNB + lane] : 1.0;
      z = lane < nb ? y[k0 + lane] : 0.0;
    }
    __syncthreads();
    if (first) {
      const int got = min(per, (4 * m - rank + blocks - 1) / blocks);  // slots with tiles
      for (int w = 1; w < got; ++w) sum += part[warp + w][lane];
      tot[f][lane] = sum;
    }
    cluster.sync();
    if (own) {
      for (int b = 0; b < min(blocks, 4 * m); ++b) z -= cluster.map_shared_rank(&tot[f][0], b)[lane];
      double x = z * r;
#pragma unroll
      for (int j = kNB - 1; j > 0; --j) x = fma(-urow[j], __shfl_sync(0xffffffffu, x, j), x);
      if (lane < nb) {
        y[k0 + lane] = x;
        atomicAdd(v.q + d0 + k0 + lane, x);
      }
    }
    cluster.sync();
  }
  if (rank == 0 && threadIdx.x == 0) {
    v.sys_iters[s] += 1;
    if (v.ls_trial) v.ls_trial[s] = 1;
    atomicAdd(&v.ctrl[0], 1);
    if (v.units) atomicAdd(v.units, (unsigned long long)n);
  }
}

// The whole factorisation and solve: right-hand side in v.dq (k_cc_band).
cudaError_t lu_solve(const ContactArgs &a, const SolveArgs &v, int sms, cudaStream_t st) {
  const int nt = a.max_tiles, nc = a.n_contact;
  if (nc == 0) return cudaSuccess;
  const int words = nt * ((nt + 31) / 32), threads = std::max(512, (nt + 31) / 32 * 32);
  k_lu_order<<<nc, threads, 4 * words, st>>>(a);
  // the chip shared among the systems; several blocks of a system wait for one
  // another, so all of them must be resident (one per SM), which a cooperative
  // launch guarantees; without such launches, and under MPS, where CUDA takes
  // none inside the round's graph, one block per system
  int dev = 0, coop = 0, mps = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&mps, cudaDevAttrMpsEnabled, dev);
  if (e != cudaSuccess) return e;
  cudaLaunchAttribute at[1];
  cudaLaunchConfig_t cfg{};
  cfg.attrs = at;
  cfg.numAttrs = 1;
  cfg.stream = st;
  const int share = coop && !mps ? std::max(1, std::min(sms / nc, 4 * nt * nt)) : 1;
  cfg.gridDim = dim3(nc, share);
  cfg.blockDim = dim3(kLuThreads);
  at[0].id = cudaLaunchAttributeCooperative;
  at[0].val.cooperative = share > 1 ? 1 : 0;
  e = cudaLaunchKernelEx(&cfg, k_lu, a, v.dq);
  if (e != cudaSuccess) return e;
  // a cluster of up to eight blocks while the systems leave SMs idle
  int cs = 8;
  while (cs > 1 && cs * nc > sms) cs >>= 1;
  cfg.gridDim = dim3(nc * cs);
  cfg.blockDim = dim3(32 * kSubstWarps);
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = cs;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  e = cudaLaunchKernelEx(&cfg, k_cc_subst, a, v);
  return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace dm
