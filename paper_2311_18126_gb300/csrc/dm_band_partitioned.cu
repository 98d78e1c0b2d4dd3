// Partitioned solve of long symmetric banded systems (half bandwidth 10, the
// single-rod Jacobian of Sec. III-C, Eq. 16) that removes the sequential
// chain over the whole rod: the DOFs of a system are cut into interiors of
// m - 10 rows separated by 10-row separators, so that interiors do not
// couple (|i - j| > 10 across a separator):
//
//   1. k_part_factor, a warp per interior: L D L^T from its first row to its
//      last, the separator above carried along as ten more rows (and its own
//      Schur complement in registers), so that what is left in the window at
//      the end is the separator below with its coupling to the one above;
//   2. k_part_separators, a block per system: the block-tridiagonal system of
//      the separators (10 x 10 blocks, Gauss-Jordan without pivoting: a Schur
//      complement of the symmetric matrix, positive definite whenever the rod
//      Jacobian is), then x on the separators;
//   3. k_part_back, a warp per interior: x_i = z_i - L^T x - (the upper
//      separator's multipliers) x_top.
//
// A column costs 230 (full band) or on average 202 (a rod's envelope: ENV)
// updates against 65 or 49 without the carried separator, but the sequential
// depth is m rows plus one block elimination per separator instead of n rows.
// Bound by the FP64 pipe (64 cycles per warp instruction and SM partition):
// the updates of a column are dealt evenly over the 32 lanes, its multipliers
// formed once (one instruction, exchanged through shared memory), 7.75 FP64
// slots per column of a rod; the reciprocal runs on the integer pipe.
// Measured (GB300): the solves of one step of 64 rods of 4000-6000 nodes (1.3 M
// DOFs, interiors of 502 rows) 12.5 -> 2.7 ms against a warp per interior that
// factored the band, solved for the carried columns and formed the Schur
// products one after another, with two barriers and a division per column.
#include <algorithm>
#include <cmath>
#include <string>
#include <vector>

#include "dm_internal.h"
#include "dm_kernels.cuh"

namespace dm {

namespace {

constexpr int PW = 10;  // half bandwidth = separator width

// Pivots smaller than this fraction of their row's original diagonal entry
// are treated as zero (DM_ERR_DEGENERATE): without pivoting they would
// amplify rounding errors without bound.
constexpr double kTinyPivot = 1e-13;

constexpr int kRecW = 24;   // a column's record: z, l_1..l_10, 0, the ten carried rows' multipliers, 0, 0
constexpr int kRowW = 22;   // a window row: 11 diagonals, right-hand side, coupling to the separator above
constexpr int kPB = 12;     // columns per block (4-periodic like the envelope)
constexpr int kPWin = 2 * kPB * kRowW;  // doubles of a window buffer
constexpr int kPCell = 2;               // a fixed cell (the 65th separator sum)
constexpr int kPSmem = 2 * kPWin + kPB * kRecW + kPCell;

struct PartArgs {
  int64_t ntot;
  int nparts, nsep;
  const int32_t *p_a, *p_mm, *p_top, *p_bot;  // interior rows [a, a+mm), separator ids or -1
  const int32_t *s_a;                          // separator rows [s_a, s_a + 10)
  const int32_t *sys_sep0, *sys_nsep;          // per system: first separator, count
  const double *band, *rhs;
  double *x;
  double *q;                   // NULL, or q -= x
  double *rec;                 // [ntot][kRecW]
  double *wb, *tt, *xo;        // [nparts][110]: what is left of the separator below (10x10, 10), the
                               // Schur terms of the one above (10x10, 10), their coupling (10x10)
  double *Xs;                  // [nsep][110]: T'^{-1} [To | g']
  const int32_t *p_sys;        // interior -> system (index into go / bad)
  const int32_t *go;           // per system: solve it (NULL: all)
  int *bad;                    // per system: zero or non-finite pivot
};

// Window tasks of a column with R rows below it, in order: row i = 1..R,
// columns q = 1..i, the right-hand side, the ten carried rows; task t is lane
// t mod 32's slot t / 32 (the next pivot (1, 1): lane 0's first).  Spare slots
// repeat the lane's first task, except lane 31's last one (spare for every
// R), which takes the 65th of the carried rows' own 65 sums (55 and ten of
// the right-hand side; the other 64 are registers, two per lane).
__host__ __device__ constexpr int win_tasks(int R) { return R * (R + 1) / 2 + 11 * R; }
__host__ __device__ constexpr int win_slots(int R) { return (win_tasks(R) + 31) / 32; }
static_assert(win_slots(10) == 6 && win_slots(9) == 5 && win_slots(8) == 4 && win_slots(7) == 4);
static_assert(win_tasks(10) <= 191 && win_tasks(9) <= 159 && win_tasks(8) <= 127 && win_tasks(7) <= 127,
              "lane 31's last slot is spare");

extern __shared__ __align__(16) char g_psm[];
__device__ __forceinline__ double &psm(int off) { return *reinterpret_cast<double *>(g_psm + off); }

template <bool ENV>
struct PartLane {
  static constexpr int T = ENV ? 4 : 1, K = win_slots(10);
  int to[T][K], uo[T][K], lo[T][K];  // byte offsets: target, column entry, multiplier (in the record)
  int su[2], sl[2];                  // the lane's two register sums: column entry, multiplier
  int mo, ro;                        // the lane's multiplier: source, record word
  int adj;                           // lane 31: -1 (its last task's target does not move)
  __device__ __forceinline__ void load(int lane, int rec, int cell) {
    adj = lane == 31 ? -8 * kRowW : 0;
#pragma unroll
    for (int t = 0; t < T; ++t) {
      const int R = 10 - t, n = win_tasks(R);
#pragma unroll
      for (int k = 0; k < K; ++k) {
        if (k >= win_slots(R)) continue;
        int e = lane + 32 * k;
        if (e >= n) e = lane;
        int i = 1;
        while (e >= i + 11) e -= i++ + 11;
        // e < i: column q = e + 1; e == i: right-hand side; beyond: carried row e - i - 1
        const int c = e < i ? 0 : e == i ? 11 : 12 + e - i - 1;
        to[t][k] = 8 * (kRowW * i + (e < i ? i - e - 1 : c));
        uo[t][k] = 8 * (e < i ? (kRowW + 1) * (e + 1) : c);
        lo[t][k] = rec + 8 * i;
        if (lane == 31 && k == win_slots(R) - 1) {
          to[t][k] = cell;
          uo[t][k] = 8 * 11;
          lo[t][k] = rec + 8 * 21;
        }
      }
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      int e = lane + 32 * h, k = 0;
      while (e >= k + 2) e -= k++ + 2;
      su[h] = 8 * (e <= k ? 12 + e : 11);
      sl[h] = rec + 8 * (12 + k);
    }
    // lanes 0-9: l_1..l_10; 10-19: the carried rows; 20: z; the others repeat z
    mo = lane < 10 ? 8 * (kRowW + 1) * (lane + 1) : lane < 20 ? 8 * (12 + lane - 10) : 8 * 11;
    ro = rec + 8 * (lane < 10 ? lane + 1 : lane < 20 ? lane + 2 : 0);
  }
  // which sum (row k, column e <= k or the right-hand side) register h of the lane is
  __device__ __forceinline__ int sum_index(int lane, int h) const {
    int e = lane + 32 * h, k = 0;
    while (e >= k + 2) e -= k++ + 2;
    return e <= k ? k * PW + e : 100 + k;
  }
};

// Column u of a block at window offset w (bytes): rj its pivot's reciprocal
// (in), the next column's (out).
template <bool ENV>
__device__ __forceinline__ void part_column(const PartLane<ENV> &ln, const int t, const int u, int w, double &rj,
                                            double (&sum)[2], bool act) {
  constexpr int K = PartLane<ENV>::K;
  const int NK = win_slots(10 - t);
  const int wu = w + 8 * kRowW * u, ru = 8 * kRecW * u;
  psm(ln.ro + ru) = psm(ln.mo + wu) * rj;
  double uq[K], dv[K], v[K];
#pragma unroll
  for (int k = 0; k < K; ++k)
    if (k < NK) {
      uq[k] = psm(ln.uo[t][k] + wu);
      dv[k] = psm(ln.to[t][k] + (k == NK - 1 && ln.adj ? 0 : wu));
    }
  const double s0 = psm(ln.su[0] + wu), s1 = psm(ln.su[1] + wu);
  __syncwarp();
#pragma unroll
  for (int k = 0; k < K; ++k)
    if (k < NK) v[k] = fma(-psm(ln.lo[t][k] + ru), uq[k], dv[k]);
  rj = rcp_any(__shfl_sync(0xffffffffu, v[0], 0));
  const double p0 = fma(-psm(ln.sl[0] + ru), s0, sum[0]), p1 = fma(-psm(ln.sl[1] + ru), s1, sum[1]);
  if (act) {
    sum[0] = p0;
    sum[1] = p1;
#pragma unroll
    for (int k = 0; k < K; ++k)
      if (k < NK) psm(ln.to[t][k] + (k == NK - 1 && ln.adj ? 0 : wu)) = v[k];
  }
  __syncwarp();
}

__device__ __forceinline__ void part_cp8(double *dst, const double *src, bool on) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n" ::"r"(d), "l"(src), "r"(on ? 8 : 0) : "memory");
}

// Interior rows row0 .. row0 + 11 (and beyond its end the separator's) into
// the window at `buf`, zero past `rows`; the coupling to the separator above
// (rows 0-9, J[r][k - 10]) where `top`.
__device__ __forceinline__ void part_stage(const PartArgs &a, int r0, double *buf, int row0, int rows, bool top,
                                           int lane) {
#pragma unroll
  for (int e = lane; e < kPB * kRowW; e += 32) {
    const int d = e / kPB, s = e - d * kPB, r = row0 + s;
    bool on = r < rows;
    const double *src = a.rhs;
    if (d < 11) {
      on = on && d <= r;
      src = a.band + (size_t)d * a.ntot + r0 + r;
    } else if (d == 11) {
      src = a.rhs + r0 + r;
    } else {
      const int k = d - 12;
      on = on && top && k >= r;
      src = a.band + (size_t)(r + PW - k) * a.ntot + r0 + r;
    }
    part_cp8(buf + s * kRowW + d, on ? src : a.rhs, on);
  }
}

template <bool ENV>
__global__ void __launch_bounds__(32) k_part_factor(PartArgs a) {
  const int p = blockIdx.x, lane = threadIdx.x;
  const int sys = a.p_sys[p];
  if (a.go && !a.go[sys]) return;
  const int r0 = a.p_a[p], mm = a.p_mm[p];
  const bool top = a.p_top[p] >= 0, bot = a.p_bot[p] >= 0;
  const int rows = mm + (bot ? PW : 0);
  double *W = reinterpret_cast<double *>(g_psm);
  double *R = W + 2 * kPWin, *cell = R + kPB * kRecW;
  PartLane<ENV> ln;
  ln.load(lane, 8 * (2 * kPWin), 8 * (2 * kPWin + kPB * kRecW));
  // record words that no lane writes stay zero; rows outside the envelope too
  for (int i = lane; i < kPB * kRecW + kPCell; i += 32) R[i] = 0.0;
  part_stage(a, r0, W, 0, rows, top, lane);
  part_stage(a, r0, W + kPB * kRowW, kPB, rows, false, lane);
  cp_async_commit();
  cp_async_wait_all();
  __syncwarp();
  double rj = rcp_any(W[0]), sum[2] = {0.0, 0.0};
  bool bad = false;
  const int nblk = (mm + kPB - 1) / kPB;
  for (int b = 0; b < nblk; ++b) {
    const int j0 = b * kPB, w = b & 1 ? 8 * kPWin : 0;
    double *cur = W + (b & 1 ? kPWin : 0), *nxt = W + (b & 1 ? 0 : kPWin);
    const bool more = b + 1 < nblk;
    if (more) part_stage(a, r0, nxt + kPB * kRowW, j0 + 2 * kPB, rows, false, lane);
    cp_async_commit();
    // the original diagonal entries of the block's rows, for the pivot test
    const bool mine = lane < kPB && j0 + lane < mm;
    const double diag = mine ? a.band[r0 + j0 + lane] : 0.0;
#pragma unroll
    for (int u = 0; u < kPB; ++u) part_column<ENV>(ln, ENV ? (u & 3) : 0, u, w, rj, sum, j0 + u < mm);
    if (mine) {
      const double d = cur[kRowW * lane];
      if (!(fabs(d) > 0.0) || !isfinite(d) || fabs(diag) * kTinyPivot > fabs(d)) bad = true;
    }
    // the block's records (12 words each of the two halves' 16-byte parts)
    for (int e = lane; e < kPB * (kRecW / 2); e += 32) {
      const int u = e / (kRecW / 2), h = e - u * (kRecW / 2);
      if (j0 + u < mm)
        *reinterpret_cast<double2 *>(a.rec + (size_t)(r0 + j0 + u) * kRecW + 2 * h) =
            *reinterpret_cast<const double2 *>(R + u * kRecW + 2 * h);
    }
    cp_async_wait_all();
    __syncwarp();  // the staged rows and this block's last columns, by every lane
    if (more)
      for (int e = lane; e < kPB * kRowW; e += 32) nxt[e] = cur[kPB * kRowW + e];
    __syncwarp();
  }
  if (__any_sync(0xffffffffu, bad)) {
    if (lane == 0) atomicExch(a.bad + sys, 1);
    return;
  }
  // what is left: the separator below and its coupling to the one above
  if (bot) {
    const double *F = W + (nblk & 1 ? 0 : kPWin) + kRowW * (mm - kPB * (nblk - 1));
    for (int e = lane; e < 210; e += 32) {
      if (e < 100) {
        const int i = e / PW, j = e - i * PW, hi = i > j ? i : j, d = i > j ? i - j : j - i;
        a.wb[(size_t)p * 110 + e] = F[kRowW * hi + d];
      } else if (e < 110) {
        a.wb[(size_t)p * 110 + e] = F[kRowW * (e - 100) + 11];
      } else {
        const int k = (e - 110) / PW, i = (e - 110) - k * PW;
        a.xo[(size_t)p * 100 + (e - 110)] = F[kRowW * i + 12 + k];
      }
    }
  }
  if (top) {
    double *T = a.tt + (size_t)p * 110;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int e = ln.sum_index(lane, h);
      T[e] = sum[h];
      if (e < 100) T[(e % PW) * PW + e / PW] = sum[h];
    }
    if (lane == 31) T[109] = cell[0];
  }
}

// Block-tridiagonal elimination over a system's separators, four warps:
// separator s couples to s + 1 through interior s + 1.  The block [T' | To |
// g'] (10 x 21) is reduced by Gauss-Jordan, warp w on rows w, w + 4, w + 8,
// lane j on column j; the next separator's terms are fetched meanwhile.
constexpr int kSepThreads = 128;
__global__ void __launch_bounds__(kSepThreads) k_part_separators(PartArgs a) {
  __shared__ double M[2][PW][22];        // by pivot parity: a column is read while it is rewritten
  __shared__ double Tp[PW][PW + 1], Xp[PW][PW + 1];  // To and T'^{-1} [To | g'] of the one before
  __shared__ int fail;
  const int sys = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int s0 = a.sys_sep0[sys], ns = a.sys_nsep[sys];
  if (ns == 0 || (a.go && !a.go[sys]) || a.bad[sys]) return;
  if (tid == 0) fail = 0;
  // this thread's entry of [T | To | g]: T and g from the interior above
  // (wb) and below (tt), To from the one below
  auto fetch = [&](int s) -> double {
    const int pu = s0 + s + sys, pd = pu + 1;
    double v = 0.0;
    if (s < ns && tid < 110) {
      v = a.wb[(size_t)pu * 110 + tid] + a.tt[(size_t)pd * 110 + tid];
    }
    return v;
  };
  auto fetch_to = [&](int s) -> double {
    return s + 1 < ns && tid < 100 ? a.xo[(size_t)(s0 + s + sys + 1) * 100 + tid] : 0.0;
  };
  double nt = fetch(0), no = fetch_to(0);
  for (int s = 0; s < ns; ++s) {
    const int i = tid < 100 ? tid / PW : tid - 100, j = tid < 100 ? tid % PW : 2 * PW;
    if (tid < 110) {
      double v = nt;
      if (s > 0) {  // T'_s = T_s - To^T X, g'_s = g_s - To^T y of the separator before
#pragma unroll
        for (int k = 0; k < PW; ++k) v = fma(-Tp[k][i], Xp[k][tid < 100 ? j : PW], v);
      }
      M[0][i][j] = v;
    }
    __syncthreads();
    if (tid < 100) {
      M[0][i][PW + j] = no;
      Tp[i][j] = no;
    }
    nt = fetch(s + 1);
    no = fetch_to(s + 1);
    __syncthreads();
    double d0 = tid < PW ? M[0][tid][tid] : 1.0;  // starting diagonal, for the pivot test
    double piv = 0.0;
#pragma unroll
    for (int k = 0; k < PW; ++k) {
      const double(*A)[22] = M[k & 1];
      double(*B)[22] = M[(k + 1) & 1];
      const double pk = A[k][k], r = rcp_any(pk);
      if (tid == k) piv = pk;
      if (lane < 2 * PW + 1) {
        const double mk = A[k][lane] * r;
#pragma unroll
        for (int t = 0; t < 3; ++t) {
          const int row = warp + 4 * t;
          if (row < PW) B[row][lane] = row == k ? mk : fma(-A[row][k], mk, A[row][lane]);
        }
      }
      __syncthreads();
    }
    if (tid < PW && (!(fabs(piv) > 0.0) || !isfinite(piv) || fabs(piv) < kTinyPivot * fabs(d0))) fail = 1;
    if (tid < 110) {  // PW is even: the result is in M[0]
      const double v = tid < 100 ? M[0][i][PW + j] : M[0][i][2 * PW];
      Xp[i][tid < 100 ? j : PW] = v;
      a.Xs[(size_t)(s0 + s) * 110 + tid] = v;
    }
    __syncthreads();
    if (fail) {  // uniform
      if (tid == 0) atomicExch(a.bad + sys, 1);
      return;
    }
  }
  // back substitution by one warp: x_s = y_s - X_s x_{s+1}, lane i < 10 the row
  if (warp) return;
  __syncwarp();
  double xn = 0.0;
  double row[PW], yn = 0.0;
  auto load = [&](int s) {
    if (lane < PW && s >= 0) {
      const double *X = a.Xs + (size_t)(s0 + s) * 110;
#pragma unroll
      for (int k = 0; k < PW; ++k) row[k] = X[lane * PW + k];
      yn = X[100 + lane];
    }
  };
  load(ns - 1);
  for (int s = ns - 1; s >= 0; --s) {
    double xv = yn, c[PW];
#pragma unroll
    for (int k = 0; k < PW; ++k) c[k] = s + 1 < ns ? row[k] : 0.0;
    load(s - 1);
    double even = xv, odd = 0.0;
#pragma unroll
    for (int k = 0; k < PW; k += 2) {
      even = fma(-c[k], __shfl_sync(0xffffffffu, xn, k), even);
      odd = fma(-c[k + 1], __shfl_sync(0xffffffffu, xn, k + 1), odd);
    }
    xn = even + odd;
    if (lane < PW) {
      const int at = a.s_a[s0 + s] + lane;
      a.x[at] = xn;
      if (a.q) a.q[at] -= xn;
    }
  }
}

// x of an interior, from its last row up: the row of step t is pending in
// lane t mod 32; a step takes its x by a shuffle and subtracts its part from
// the next ten rows.  The separator below feeds the first ten steps, the one
// above enters a row's start value with its record's carried multipliers.
// Each lane stages the record of its own next row.
__global__ void __launch_bounds__(32) k_part_back(PartArgs a) {
  constexpr int kRing = 3;
  __shared__ __align__(16) double ring[32][kRing * kRecW + 2];
  const int p = blockIdx.x, lane = threadIdx.x;
  if ((a.go && !a.go[a.p_sys[p]]) || a.bad[a.p_sys[p]]) return;
  const int r0 = a.p_a[p], mm = a.p_mm[p];
  const int st = a.p_top[p], sb = a.p_bot[p];
  const unsigned full = 0xffffffffu;
  double xt = 0.0, xb = 0.0;  // lane c < 10: separator values
  if (lane < PW) {
    if (st >= 0) xt = a.x[a.s_a[st] + lane];
    if (sb >= 0) xb = a.x[a.s_a[sb] + lane];
  }
  // step t < 10: separator row 9 - t; step t >= 10: interior row mm + 9 - t
  const int R0 = mm + 9;
  auto fetch = [&](int g) {
    const int r = R0 - (32 * g + lane);
    double *dst = &ring[lane][kRecW * (g % kRing)];
    if (r >= 0 && r < mm) {
      const double *src = a.rec + (size_t)(r0 + r) * kRecW;
#pragma unroll
      for (int e = 0; e < kRecW; e += 2) {
        const unsigned d = (unsigned)__cvta_generic_to_shared(dst + e);
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(src + e) : "memory");
      }
    } else {
#pragma unroll
      for (int e = 0; e < kRecW; ++e) dst[e] = 0.0;
    }
  };
  auto start = [&](int g) -> double {  // z - (carried multipliers) x_top
    const double *rc = &ring[lane][kRecW * (g % kRing)];
    double even = rc[0], odd = 0.0;
    if (st >= 0) {  // warp-uniform
#pragma unroll
      for (int k = 0; k < PW; k += 2) {
        even = fma(-rc[12 + k], __shfl_sync(full, xt, k), even);
        odd = fma(-rc[13 + k], __shfl_sync(full, xt, k + 1), odd);
      }
    }
    return even + odd;
  };
#pragma unroll
  for (int g = 0; g < kRing; ++g) fetch(g);
  cp_async_commit();
  cp_async_wait_all();
  int idx[32];
#pragma unroll
  for (int u = 0; u < 32; ++u) {
    const int d = (lane - u) & 31;
    idx[u] = d == 0 || d > 11 ? 11 : d;  // word 11 is zero
  }
  double v = start(0);
  const int groups = (R0 + 1 + 31) / 32;
  for (int g = 0; g < groups; ++g) {
    const double *ra = &ring[lane][kRecW * (g % kRing)], *rb = &ring[lane][kRecW * ((g + 1) % kRing)];
    const double zn = start(g + 1);
    double x_own = 0.0;
#pragma unroll
    for (int u = 0; u < 32; ++u) {
      double x = __shfl_sync(full, v, u);
      if (g == 0 && u < PW) x = __shfl_sync(full, xb, 9 - u);
      if (lane == u) {
        x_own = x;
        v = zn;
      }
      v = fma(-(lane <= u ? rb : ra)[idx[u]], x, v);
    }
    const int r = R0 - (32 * g + lane);
    if (r >= 0 && r < mm) {
      if (a.q) a.q[r0 + r] -= x_own;
      else a.x[r0 + r] = x_own;
    }
    fetch(g + kRing);
    cp_async_commit();
    asm volatile("cp.async.wait_group 1;\n" ::: "memory");
  }
  cp_async_wait_all();
}

// Newton rounds of long rods (the partitioned path of dm_step): the
// bookkeeping of the rod solver (converged, failed or solving this round;
// the solve itself takes q -= J^-1 f).
struct LongArgs {
  int nlong;
  const int32_t *sys;                 // long system -> system index
  double tol;
  int max_iter;
  int32_t *sys_active, *sys_iters, *sys_status;
  const unsigned long long *sys_res;
  int32_t *ctrl;
  const int32_t *ls_action;
  int32_t *ls_trial;
  int32_t *go;
  int *bad;
};

__global__ void k_long_decide(LongArgs a) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= a.nlong) return;
  const int s = a.sys[k];
  int go = 0;
  a.bad[k] = 0;
  if (a.sys_active[s]) {
    if (a.ls_action && a.ls_action[s] == 1) {  // backtracking: no solve this round
      atomicAdd(&a.ctrl[0], 1);
    } else {
      const double res = __longlong_as_double((long long)a.sys_res[s]);
      int st = a.sys_status[s];
      if (st == 0 && isnan(res)) st = DM_ERR_NONFINITE;
      if (st == 0 && res <= a.tol) {
        a.sys_active[s] = 0;
      } else {
        if (st == 0 && a.sys_iters[s] >= a.max_iter) st = DM_ERR_NOT_CONVERGED;
        if (st != 0) {
          a.sys_status[s] = st;
          a.sys_active[s] = 0;
          atomicAdd(&a.ctrl[1], 1);
          atomicMin(&a.ctrl[2], s);
        } else {
          go = 1;
        }
      }
    }
  }
  a.go[k] = go;
}

__global__ void k_long_finish(LongArgs a) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= a.nlong || !a.go[k]) return;
  const int s = a.sys[k];
  if (a.bad[k]) {
    a.sys_status[s] = DM_ERR_DEGENERATE;
    a.sys_active[s] = 0;
    atomicAdd(&a.ctrl[1], 1);
    atomicMin(&a.ctrl[2], s);
    return;
  }
  a.sys_iters[s] += 1;
  if (a.ls_trial) a.ls_trial[s] = 1;
  atomicAdd(&a.ctrl[0], 1);
}

}  // namespace

// Host plan of a partitioned solve: interiors, separators and scratch for
// a fixed set of systems.
struct PartPlan {
  int np = 0, nsep = 0, nsys = 0;
  char *scr = nullptr;
  PartArgs A{};
};

static void part_plan_free(PartPlan &P) {
  if (P.scr) cudaFree(P.scr);
  P.scr = nullptr;
}

// layout: interiors [k m, k m + m - 10), separators [k m + m - 10, (k+1) m),
// the last interior [(P-1) m, n) with at least 11 rows
static dm_status part_plan_build(int nsys, const int32_t *sys_dof0, const int32_t *sys_ndof,
                                 int64_t ntot, int m, PartPlan &P, cudaStream_t st) {
  std::vector<int32_t> pa, pmm, ptop, pbot, psys, sa, s0(nsys), nsp(nsys);
  for (int k = 0; k < nsys; ++k) {
    const int n = sys_ndof[k], d0 = sys_dof0[k];
    if (n <= 0 || d0 < 0 || (int64_t)d0 + n > ntot) {
      set_error("partitioned band solve: system outside the vectors");
      return DM_ERR_INVALID_ARG;
    }
    int np = (n - 1) / m + 1;
    while (np > 1 && n - (np - 1) * m < PW + 1) --np;
    s0[k] = (int32_t)sa.size();
    nsp[k] = np - 1;
    for (int p = 0; p < np; ++p) {
      const int a = p * m, b = p + 1 < np ? a + m - PW : n;
      pa.push_back(d0 + a);
      pmm.push_back(b - a);
      psys.push_back(k);
      // the top separator of interior p > 0 is the bottom one of p - 1
      ptop.push_back(p > 0 ? pbot.back() : -1);
      if (p + 1 < np) sa.push_back(d0 + b);
      pbot.push_back(p + 1 < np ? (int32_t)sa.size() - 1 : -1);
    }
  }
  const int np = (int)pa.size(), nsep = (int)sa.size();
  P.np = np;
  P.nsep = nsep;
  P.nsys = nsys;
  size_t bytes = 0;
  auto take = [&](size_t n, size_t elt) {
    const size_t o = bytes;
    bytes += (n * elt + 255) / 256 * 256;
    return o;
  };
  const size_t orec = take((size_t)ntot * kRecW, 8), owb = take((size_t)np * 110, 8), ott = take((size_t)np * 110, 8),
               oxo = take((size_t)np * 100, 8), oX = take((size_t)std::max(nsep, 1) * 110, 8),
               oI = take(5 * (size_t)np + (size_t)nsep + 3 * (size_t)nsys + 1, 4);
  if (cudaMalloc(&P.scr, bytes) != cudaSuccess) {
    set_error("partitioned band solve: cudaMalloc");
    return DM_ERR_OOM;
  }
  std::vector<int32_t> ints;
  for (auto *v : {&pa, &pmm, &ptop, &pbot, &psys, &sa, &s0, &nsp}) ints.insert(ints.end(), v->begin(), v->end());
  ints.resize(ints.size() + nsys, 0);  // bad flags
  int32_t *ib = reinterpret_cast<int32_t *>(P.scr + oI);
  PartArgs &A = P.A;
  A.ntot = ntot;
  A.nparts = np;
  A.nsep = nsep;
  A.p_a = ib;
  A.p_mm = ib + np;
  A.p_top = ib + 2 * np;
  A.p_bot = ib + 3 * np;
  A.p_sys = ib + 4 * np;
  A.s_a = ib + 5 * np;
  A.sys_sep0 = ib + 5 * np + nsep;
  A.sys_nsep = ib + 5 * np + nsep + nsys;
  A.bad = ib + 5 * np + nsep + 2 * nsys;
  A.rec = reinterpret_cast<double *>(P.scr + orec);
  A.wb = reinterpret_cast<double *>(P.scr + owb);
  A.tt = reinterpret_cast<double *>(P.scr + ott);
  A.xo = reinterpret_cast<double *>(P.scr + oxo);
  A.Xs = reinterpret_cast<double *>(P.scr + oX);
  cudaError_t e = cudaMemcpyAsync(ib, ints.data(), ints.size() * sizeof(int32_t),
                                  cudaMemcpyHostToDevice, st);
  if (e != cudaSuccess) {
    part_plan_free(P);
    set_error(std::string("partitioned band solve: ") + cudaGetErrorString(e));
    return DM_ERR_CUDA;
  }
  return DM_OK;
}

// env: the matrices have the envelope of a rod's Jacobian and every interior
// starts at a node (part_rows a multiple of four).
static cudaError_t part_launch(const PartPlan &P, const double *band, const double *rhs,
                               double *x, double *q, const int32_t *go, bool env, cudaStream_t st) {
  PartArgs A = P.A;
  A.band = band;
  A.rhs = rhs;
  A.x = x;
  A.q = q;
  A.go = go;
  constexpr size_t smem = kPSmem * sizeof(double);
  static_assert(smem <= 48 * 1024, "within the default limit");
  if (env) k_part_factor<true><<<P.np, 32, smem, st>>>(A);
  else k_part_factor<false><<<P.np, 32, smem, st>>>(A);
  if (P.nsep > 0) k_part_separators<<<P.nsys, kSepThreads, 0, st>>>(A);
  k_part_back<<<P.np, 32, 0, st>>>(A);
  return cudaGetLastError();
}

struct LongRods {
  PartPlan plan;
  LongArgs la{};
  std::vector<void *> allocs;
};

// Rows per interior (a multiple of four, for the envelope): a column takes
// about 550 cycles, a separator of the sequential elimination about 14000, so
// for one rod of n rows the two chains m + 25 n / m are shortest at
// m = 5 sqrt(n), and half of that costs little more in separators;
// a large batch takes interiors that still come in several waves, which the
// block scheduler balances: 64 rods of 20000 rows factor in 0.95 ms with 512
// rows, in 1.29 ms with 1060 (one uneven wave), while the separators shrink
// from 0.28 to 0.15 ms.
static int long_part_rows(int64_t total, int n_max, int sms) {
  const int64_t m = std::max<int64_t>((int64_t)(2.5 * std::sqrt((double)n_max)), total / (16 * sms));
  return (int)std::min<int64_t>(2048, std::max<int64_t>(128, m)) / 4 * 4;
}

dm_status long_rods_create(dm_system *s, const std::vector<int32_t> &sys, LongRods **out) {
  *out = nullptr;
  if (sys.empty()) return DM_OK;
  const HostTopology &T = s->T;
  auto *L = new LongRods();
  const int nl = (int)sys.size();
  std::vector<int32_t> d0(nl), nd(nl);
  int64_t total = 0;
  int n_max = 0, dev = 0, sms = 1;
  for (int k = 0; k < nl; ++k) {
    d0[k] = T.sys_dof0[sys[k]];
    nd[k] = T.sys_ndof[sys[k]];
    total += nd[k];
    n_max = std::max(n_max, nd[k]);
  }
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int part_rows = long_part_rows(total, n_max, sms);
  dm_status r = part_plan_build(nl, d0.data(), nd.data(), T.n_dofs, part_rows, L->plan, s->stream);
  auto dal = [&](void **p, size_t bytes) {
    if (cudaMalloc(p, bytes) != cudaSuccess) return false;
    L->allocs.push_back(*p);
    return true;
  };
  int32_t *dsys = nullptr, *dgo = nullptr;
  if (r == DM_OK && (!dal((void **)&dsys, nl * 4) || !dal((void **)&dgo, nl * 4))) {
    set_error("long rods: cudaMalloc");
    r = DM_ERR_OOM;
  }
  if (r == DM_OK && cudaMemcpy(dsys, sys.data(), nl * 4, cudaMemcpyHostToDevice) != cudaSuccess)
    r = DM_ERR_CUDA;
  if (r != DM_OK) {
    long_rods_free(L);
    return r;
  }
  L->la.nlong = nl;
  L->la.sys = dsys;
  L->la.go = dgo;
  L->la.bad = L->plan.A.bad;
  *out = L;
  return DM_OK;
}

void long_rods_free(LongRods *L) {
  if (!L) return;
  part_plan_free(L->plan);
  for (void *p : L->allocs) cudaFree(p);
  delete L;
}

int long_rods_count(const LongRods *L) { return L ? L->la.nlong : 0; }

cudaError_t long_rods_round(LongRods *L, const SolveArgs &v, cudaStream_t st) {
  LongArgs a = L->la;
  a.tol = v.tol;
  a.max_iter = v.max_iter;
  a.sys_active = v.sys_active;
  a.sys_iters = v.sys_iters;
  a.sys_status = v.sys_status;
  a.sys_res = v.sys_res;
  a.ctrl = v.ctrl;
  a.ls_action = v.ls_action;
  a.ls_trial = v.ls_trial;
  const int nb = (a.nlong + 127) / 128;
  k_long_decide<<<nb, 128, 0, st>>>(a);
  cudaError_t e = part_launch(L->plan, v.band, v.f, v.dq, v.q, a.go, true, st);
  if (e != cudaSuccess) return e;
  k_long_finish<<<nb, 128, 0, st>>>(a);
  return cudaGetLastError();
}

}  // namespace dm

namespace dm {
bool check_band_batch(int32_t nsys, const int32_t *dof0, const int32_t *ndof, int64_t ntot,
                      const double *band, const double *rhs, const double *x);
}  // namespace dm

using namespace dm;

extern "C" dm_status dm_solve_band_partitioned(int32_t nsys, const int32_t *sys_dof0,
                                               const int32_t *sys_ndof, int64_t ntot,
                                               const double *band, const double *rhs, double *x,
                                               int32_t part_rows, void *stream) {
  // the same batch rules as dm_solve_band (systems in range, no shared
  // rows, x apart from band and rhs)
  if (!check_band_batch(nsys, sys_dof0, sys_ndof, ntot, band, rhs, x)) return DM_ERR_INVALID_ARG;
  const int m = part_rows > 0 ? part_rows : 512;
  if (m < 2 * PW + 1 || m > 1024) {
    set_error("dm_solve_band_partitioned: part_rows must be in [21, 1024]");
    return DM_ERR_INVALID_ARG;
  }
  if (nsys == 0) return DM_OK;
  cudaStream_t st = (cudaStream_t)stream;
  PartPlan P;
  dm_status r = part_plan_build(nsys, sys_dof0, sys_ndof, ntot, m, P, st);
  if (r != DM_OK) return r;
  cudaError_t e = part_launch(P, band, rhs, x, nullptr, nullptr, false, st);
  std::vector<int> bad(nsys, 0);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(bad.data(), P.A.bad, nsys * sizeof(int), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  part_plan_free(P);
  if (e != cudaSuccess) {
    set_error(std::string("dm_solve_band_partitioned: ") + cudaGetErrorString(e));
    return DM_ERR_CUDA;
  }
  for (int k = 0; k < nsys; ++k)
    if (bad[k]) {
      set_error("dm_solve_band_partitioned: zero or non-finite pivot in system " +
                std::to_string(k));
      return DM_ERR_DEGENERATE;
    }
  return DM_OK;
}
