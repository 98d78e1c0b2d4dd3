// Banded LDL^T solve of J dq = -f for single rods (DisMech, arXiv 2311.18126,
// Sec. III-C, Eq. 16; half bandwidth 10 in the Eq. 1 layout), FP64.
//
// What bounds it: an SM partition retires one FP64 warp instruction per 64
// cycles whatever the active mask (76 with all four partitions busy: 1.68
// FMA per clock and SM; a dependent FMA waits the same 64 cycles), and a
// column of the elimination is a short chain of dependent steps.  So the
// FP64 instructions of a column are what counts, and everything else is kept
// off that pipe:
//  - each rod is factored from both ends at once (a twisted factorisation):
//    a top chain eliminates columns 0..m-1 downwards, a bottom chain columns
//    n-1..m+10 upwards, and the 10-row separator between them is combined
//    from both windows and eliminated as ten more columns of the top chain;
//  - the Jacobian of a rod fills only an envelope: in the order of either
//    chain the columns have 10, 9, 8 and 7 rows below them in turn (the three
//    position components of a node, then a twist angle: a bend-twist stencil
//    couples DOFs 4m-4 .. 4m+6), and elimination fills nothing outside it, so
//    a rod's column costs 164 instead of 220 updates per node (ENV); the
//    caller's matrices of dm_solve_band take the full band (not ENV);
//  - a chain is run by L lanes: 16 (a warp per rod: 6, 5, 4, 3 updates and
//    one multiplier per lane and column, 5.5 FP64 slots on average) while the
//    batch has few rods, where a column's latency counts, and 8 (two rods
//    per warp, 8.75 slots for twice the chains) when it fills the chip;
//  - the pivot's reciprocal runs on the integer pipe (rcp_int): three
//    dependent FP64 instructions less on the column's critical path;
//  - rows arrive by asynchronous copies a block of 12 columns ahead of their
//    use, the multipliers of a column leave as one record of 12 doubles, and
//    the back substitution keeps the pending rows in registers (one update
//    per row and a shuffle), each lane staging its own records.
// The pivot tests run once per block of columns on the integer pipe.
// Measured (GB300): the solves of one step of 4096 uneven rods (4.3 M DOFs
// in four rounds) 3.31 -> 1.59 ms against the kernel before (eight lanes per
// chain, full band, FP64 reciprocal, rows loaded in the column that uses
// them, one warp per SM partition), its first round 0.43 ms with the FP64
// pipe 64 % and the shared-memory pipe 65 % busy; of one 50-node rod 142 ->
// 58 us; of 301 rods 348 -> 136 us.
#include <algorithm>

#include "dm_internal.h"
#include "dm_kernels.cuh"

namespace dm {
namespace {

constexpr int kBlk = 12;                 // columns per block, 4-periodic like the envelope
constexpr int kWinRows = 2 * kBlk;       // rows of a window buffer: the block's columns and 12 more
constexpr int kWin = kWinRows * 12;      // doubles: 11 diagonals J[r][r-d], then the right-hand side
constexpr int kWindow = 2 * kWin + 2;    // two buffers (the next block arrives in one); +2: banks
constexpr int kRec = 12 * kBlk;          // records of a block's columns
constexpr int kChain = kWindow + kRec;   // doubles of a chain
static_assert(kChain % 2 == 0 && kWindow % 2 == 0, "records move by 16 bytes");
// per warp, behind the chains: where lanes store what nobody needs (kRec)

// Update tasks of a column with R rows below it, split over the L lanes of a
// chain: window row i = 1..R has the columns q = 1..i and the right-hand side
// (q = i + 1); a lane takes up to two runs (row, first q, count).  Packed
// per lane: i0 | q0 << 4 | n0 << 8, and the second run from bit 12 on; i = 0
// with n = 0 is the pivot row's right-hand side, whose product with the
// reciprocal is z_j.  The lane of task (1, 1) -- the next pivot -- has it
// first.
__host__ __device__ constexpr unsigned run(int i, int q, int n) {
  return (unsigned)(i | (q << 4) | (n << 8));
}
__host__ __device__ constexpr unsigned two(unsigned a, unsigned b) { return a | (b << 12); }
constexpr unsigned kNone = 15;  // no run

template <int L>
struct Split;

template <>
struct Split<16> {
  static constexpr int M = 1;  // multipliers per lane
  __host__ __device__ static constexpr int tasks(int R) { return R == 10 ? 6 : R == 9 ? 5 : R == 8 ? 4 : 3; }
  __host__ __device__ static constexpr unsigned lane(int R, int p) {
    constexpr unsigned t10[16] = {run(1, 1, 2), run(2, 1, 3), run(3, 1, 4), run(4, 1, 5),
                                  run(5, 1, 6), run(6, 1, 6), run(6, 7, 1), run(7, 1, 6),
                                  run(7, 7, 2), run(8, 1, 6), run(8, 7, 3), run(9, 1, 6),
                                  run(9, 7, 4), run(10, 1, 6), run(10, 7, 5), run(0, 0, 0)};
    constexpr unsigned t9[16] = {run(1, 1, 2), run(2, 1, 3), run(3, 1, 4), run(4, 1, 5),
                                 run(5, 1, 5), run(5, 6, 1), run(6, 1, 5), run(6, 6, 2),
                                 run(7, 1, 5), run(7, 6, 3), run(8, 1, 5), run(8, 6, 4),
                                 run(9, 1, 5), run(9, 6, 5), kNone, run(0, 0, 0)};
    constexpr unsigned t8[16] = {run(1, 1, 2), run(2, 1, 3), run(3, 1, 4), run(4, 1, 4),
                                 run(4, 5, 1), run(5, 1, 4), run(5, 5, 2), run(6, 1, 4),
                                 run(6, 5, 3), run(7, 1, 4), run(7, 5, 4), run(8, 1, 4),
                                 run(8, 5, 4), run(8, 9, 1), kNone, run(0, 0, 0)};
    constexpr unsigned t7[16] = {run(1, 1, 2), run(2, 1, 3), run(3, 1, 3), run(3, 4, 1),
                                 run(4, 1, 3), run(4, 4, 2), run(5, 1, 3), run(5, 4, 3),
                                 run(6, 1, 3), run(6, 4, 3), run(6, 7, 1), run(7, 1, 3),
                                 run(7, 4, 3), run(7, 7, 2), kNone, run(0, 0, 0)};
    return two(R == 10 ? t10[p] : R == 9 ? t9[p] : R == 8 ? t8[p] : t7[p], kNone);
  }
};

template <>
struct Split<8> {
  static constexpr int M = 2;
  __host__ __device__ static constexpr int tasks(int R) { return R == 10 ? 9 : R == 9 ? 7 : R == 8 ? 6 : 5; }
  __host__ __device__ static constexpr unsigned lane(int R, int p) {
    constexpr unsigned t10[8] = {
        two(run(1, 1, 2), run(2, 1, 3)),   two(run(10, 1, 9), kNone),
        two(run(10, 10, 2), run(5, 1, 6)), two(run(9, 1, 9), kNone),
        two(run(9, 10, 1), run(7, 1, 8)),  two(run(8, 1, 9), run(0, 0, 0)),
        two(run(3, 1, 4), run(4, 1, 5)),   two(run(6, 1, 7), kNone)};
    constexpr unsigned t9[8] = {
        two(run(1, 1, 2), run(3, 1, 4)), two(run(4, 1, 5), run(9, 1, 2)),
        two(run(9, 3, 7), run(0, 0, 0)), two(run(9, 10, 1), run(7, 1, 6)),
        two(run(7, 7, 2), run(6, 1, 5)), two(run(6, 6, 2), run(8, 1, 5)),
        two(run(8, 6, 4), run(5, 1, 3)), two(run(5, 4, 3), run(2, 1, 3))};
    constexpr unsigned t8[8] = {
        two(run(1, 1, 2), run(3, 3, 2)), two(run(5, 1, 6), run(0, 0, 0)),
        two(run(2, 1, 3), run(6, 1, 3)), two(run(6, 4, 4), run(3, 1, 2)),
        two(run(4, 1, 5), run(8, 1, 1)), two(run(8, 2, 6), kNone),
        two(run(8, 8, 2), run(7, 1, 4)), two(run(7, 5, 4), kNone)};
    constexpr unsigned t7[8] = {
        two(run(1, 1, 2), run(2, 1, 3)), two(run(5, 1, 5), kNone),
        two(run(5, 6, 1), run(3, 1, 4)), two(run(6, 1, 5), kNone),
        two(run(6, 6, 2), run(4, 1, 3)), two(run(4, 4, 2), run(7, 1, 3)),
        two(run(7, 4, 5), kNone),        two(run(0, 0, 0), kNone)};
    return R == 10 ? t10[p] : R == 9 ? t9[p] : R == 8 ? t8[p] : t7[p];
  }
};

// Every update (row i = 1..R, column q = 1..i + 1) exactly once, no lane over
// its task count, one lane for z, and the next pivot first in lane 0.
template <int L>
__host__ __device__ constexpr bool split_covers(int R) {
  int seen[12][13] = {};
  int z = 0;
  for (int p = 0; p < L; ++p) {
    int n = 0;
    for (int r = 0; r < 2; ++r) {
      const unsigned s = (Split<L>::lane(R, p) >> (12 * r)) & 0xFFFu;
      if (s == kNone) continue;
      const int i = s & 15, q0 = (s >> 4) & 15, c = s >> 8;
      if (r >= Split<L>::M) return false;
      if (i == 0) {
        if (c) return false;
        ++z;
        continue;
      }
      if (i > R) return false;
      for (int q = q0; q < q0 + c; ++q) {
        if (q < 1 || q > i + 1) return false;
        ++seen[i][q];
      }
      n += c;
    }
    if (n > Split<L>::tasks(R)) return false;
  }
  for (int i = 1; i <= R; ++i)
    for (int q = 1; q <= i + 1; ++q)
      if (seen[i][q] != 1) return false;
  return z == 1 && (Split<L>::lane(R, 0) & 0xFFu) == (1u | (1u << 4));
}
static_assert(split_covers<16>(10) && split_covers<16>(9) && split_covers<16>(8) && split_covers<16>(7));
static_assert(split_covers<8>(10) && split_covers<8>(9) && split_covers<8>(8) && split_covers<8>(7));

// A pivot smaller than 2^-43 (1.1e-13) times the original diagonal entry of
// its row counts as zero: J = M/dt^2 - dF/dq need not be positive definite
// (large steps, compressed or buckling rods), and without pivoting such a
// pivot would amplify rounding errors without bound.  So do pivots outside
// [2^-126, 2^126) (physical Jacobians stay many decades inside), infinite or
// NaN ones.  The test compares the upper 32 bits of |D| (exponent and 20
// leading mantissa bits, whose integer order is the order of the magnitudes)
// with a per-row threshold: the upper word of |J_jj| with 43 subtracted from
// its exponent field, at least that of 2^-126.  Exact but for ties in those
// 32 bits.
constexpr int kTinyPivotExp = 43;
constexpr int kPivotFloorHi = (1023 - 126) << 20;  // upper word of 2^-126
constexpr int kPivotCeilHi = (1023 + 126) << 20;   // upper word of 2^126
__device__ __forceinline__ bool pivot_bad(double d, double jjj) {
  const int thr = max((__double2hiint(jjj) & 0x7FFFFFFF) - (kTinyPivotExp << 20), kPivotFloorHi);
  const int h = __double2hiint(d) & 0x7FFFFFFF;
  return h < thr || h >= kPivotCeilHi;
}

__device__ __forceinline__ void cp_async8z(double *dst, const double *src, bool on) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n" ::"r"(d), "l"(src), "r"(on ? 8 : 0) : "memory");
}
__device__ __forceinline__ void cp_async16(double *dst, const double *src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(src) : "memory");
}

// One elimination direction of a rod: row r of the chain is the rod's row r
// (dir > 0) or n - 1 - r.
struct Chain {
  const double *band, *f;
  double *rec;
  size_t nd, base;
  int n, dir;
  __device__ __forceinline__ size_t at(int r) const { return base + (dir > 0 ? r : n - 1 - r); }
};

// The lane's tasks of the four (ENV) or one column types, as byte offsets in
// shared memory for the pivot row at the start of the chain's first buffer:
// update targets 12 i + (i - q) (or 12 i + 11) doubles on, column entries
// 13 q (or 11), multiplier sources 13 i (or 11 for z), and where the
// multipliers go in the record (lanes without one: the spare area).
template <int L, bool ENV>
struct Lane {
  static constexpr int T = ENV ? 4 : 1, M = Split<L>::M, K = Split<L>::tasks(10);
  int to[T][K], uo[T][K], mo[T][M], ro[T][M];
  unsigned sel[T][K];   // M > 1: all ones if the task's row is the second run's
  unsigned busy;        // bit t: the lane has tasks in column type t
  __device__ __forceinline__ void load(int p, int chain, int rec, int spare) {
    busy = 0;
#pragma unroll
    for (int t = 0; t < T; ++t) {
      unsigned s = 0;
#pragma unroll
      for (int pp = 0; pp < L; ++pp)
        if (p == pp) s = Split<L>::lane(10 - t, pp);
      const unsigned s0 = s & 0xFFFu, s1 = (s >> 12) & 0xFFFu;
      const int i0 = s0 & 15, q0 = (s0 >> 4) & 15, n0 = s0 == kNone ? 0 : (int)(s0 >> 8);
      const int i1 = s1 & 15, q1 = (s1 >> 4) & 15, n1 = s1 == kNone ? 0 : (int)(s1 >> 8);
      const bool on0 = s0 != kNone, on1 = s1 != kNone, idle = n0 + n1 == 0;
      mo[t][0] = chain + 8 * (on0 && i0 ? 13 * i0 : 11);
      ro[t][0] = !on0 ? spare : i0 == 0 ? rec : q0 == 1 ? rec + 8 * i0 : spare;
      if (M > 1) {
        mo[t][M - 1] = chain + 8 * (on1 && i1 ? 13 * i1 : 11);
        ro[t][M - 1] = !on1 ? spare : i1 == 0 ? rec : q1 == 1 ? rec + 8 * i1 : spare;
      }
      if (!idle) busy |= 1u << t;
#pragma unroll
      for (int k = 0; k < Split<L>::tasks(10 - t); ++k) {
        // beyond the lane's tasks: its last one again (the same value stored twice)
        const int kk = min(k, n0 + n1 - 1);
        const bool second = kk >= n0;
        const int i = second ? i1 : i0, q = second ? q1 + kk - n0 : q0 + kk;
        to[t][k] = chain + (idle ? 0 : 8 * (12 * i + (q == i + 1 ? 11 : i - q)));
        uo[t][k] = chain + 8 * (idle || q == i + 1 ? 11 : 13 * q);
        sel[t][k] = second && !idle ? ~0u : 0u;
      }
    }
  }
  // the offsets of the other buffer
  __device__ __forceinline__ void shift(int bytes) {
#pragma unroll
    for (int t = 0; t < T; ++t) {
#pragma unroll
      for (int k = 0; k < Split<L>::tasks(10 - t); ++k) {
        to[t][k] += bytes;
        uo[t][k] += bytes;
      }
#pragma unroll
      for (int m = 0; m < M; ++m) mo[t][m] += bytes;
    }
  }
};

__device__ __forceinline__ double pick(double a, double b, unsigned m) {  // m ? b : a, m = 0 or ~0
  const unsigned alo = (unsigned)__double2loint(a), ahi = (unsigned)__double2hiint(a);
  const unsigned blo = (unsigned)__double2loint(b), bhi = (unsigned)__double2hiint(b);
  return __hiloint2double((int)((ahi & ~m) | (bhi & m)), (int)((alo & ~m) | (blo & m)));
}

extern __shared__ __align__(16) char g_sm[];
__device__ __forceinline__ double &sm(int off) { return *reinterpret_cast<double *>(g_sm + off); }

// Column u of a block, of type t (10 - t rows below it): rj its pivot's
// reciprocal (in: this column's, out: the next one's), `move` bytes from the
// lane's offsets to the buffer, `rmove` to the records.
template <int L, bool ENV>
__device__ __forceinline__ void column(const Lane<L, ENV> &ln, const int t, const int u, int move, int rmove,
                                       double &rj, bool act, int cb) {
  constexpr int M = Lane<L, ENV>::M, K = Split<L>::tasks(10);
  const int NT = Split<L>::tasks(10 - t);
  double l[M], uq[K], dv[K], v[K];
#pragma unroll
  for (int m = 0; m < M; ++m) l[m] = sm(ln.mo[t][m] + move + 96 * u) * rj;
#pragma unroll
  for (int k = 0; k < K; ++k)
    if (k < NT) {
      uq[k] = sm(ln.uo[t][k] + move + 96 * u);
      dv[k] = sm(ln.to[t][k] + move + 96 * u);
    }
#pragma unroll
  for (int k = 0; k < K; ++k)
    if (k < NT) v[k] = fma(-(M > 1 ? pick(l[0], l[M - 1], ln.sel[t][k]) : l[0]), uq[k], dv[k]);
  rj = rcp_int(__shfl_sync(0xffffffffu, v[0], cb));  // lane 0 of the chain has the next pivot
#pragma unroll
  for (int m = 0; m < M; ++m) sm(ln.ro[t][m] + rmove + 96 * u) = l[m];
  if (act && ((ln.busy >> t) & 1u)) {
#pragma unroll
    for (int k = 0; k < K; ++k)
      if (k < NT) sm(ln.to[t][k] + move + 96 * u) = v[k];
  }
  __syncwarp();
}

// Chain rows row0 .. row0 + 11 into the window at `buf`; zero beyond row
// `rows` and before diagonal 0.  L / 4 groups of four lanes share the 12
// diagonals (the last one is the right-hand side), a lane takes three rows.
template <int L>
__device__ __forceinline__ void stage_rows(const Chain &c, double *buf, int row0, int rows, int p) {
  constexpr int W = 48 / L;
  const int g = p >> 2;
#pragma unroll
  for (int t = 0; t < 3; ++t) {
    const int s = (p & 3) + 4 * t, r = row0 + s;
    const bool in = r < rows;
    const size_t at = in ? c.at(r) : 0;
#pragma unroll
    for (int k = 0; k < W; ++k) {
      const int d = g * W + k;
      const bool on = in && (d == 11 || d <= r);
      // row r's entry of diagonal d is J[r][r-d]: stored with the larger index
      const double *src = d == 11 ? c.f + at : c.band + d * c.nd + at + (c.dir > 0 ? 0 : d);
      cp_async8z(buf + s * 12 + d, on ? src : c.f, on);
    }
  }
}

// The records of chain columns j0 .. j0 + count - 1 from shared memory to the
// global ones (their last word zero: the back substitution reads it as the
// multiplier of rows beyond the tenth).
template <int L>
__device__ __forceinline__ void store_records(const Chain &c, const double *rec, int j0, int count, int p) {
#pragma unroll
  for (int k = 0; k < (6 * kBlk + L - 1) / L; ++k) {
    const int e = p + L * k, u = e / 6, h = e - 6 * u;
    if (u < count) {
      double2 v = *reinterpret_cast<const double2 *>(rec + 12 * u + 2 * h);
      if (h == 5) v.y = 0.0;
      *reinterpret_cast<double2 *>(c.rec + 12 * c.at(j0 + u) + 2 * h) = v;
    }
  }
}

template <int L, bool ENV>
__global__ void __launch_bounds__(128, L == 16 ? 3 : 2) k_solve_rod(SolveArgs a) {
  constexpr int kChains = 32 / L, kRods = kChains / 2;
  const int lane = threadIdx.x & 31;
  const int chain = lane / L, unit = chain >> 1, half = chain & 1, p = lane & (L - 1);
  const int cb = chain * L, tb = (chain & ~1) * L;  // first lane of the chain, of the rod's top chain
  double *wsm = reinterpret_cast<double *>(g_sm) + (size_t)(threadIdx.x >> 5) * (kChains * kChain + kRec);
  double *W = wsm + chain * kChain, *R = W + kWindow;
  const int w_off = (int)(reinterpret_cast<char *>(W) - g_sm), r_off = w_off + 8 * kWindow;
  const unsigned full = 0xffffffffu;
  const bool head = lane == tb;  // bookkeeping lane of the rod
  const unsigned rod_mask = (kRods == 1 ? full : 0xFFFFu << (unit * 16));
  Lane<L, ENV> ln;
  ln.load(p, w_off, r_off, (int)(reinterpret_cast<char *>(wsm + kChains * kChain) - g_sm));
  // records: rows outside the envelope are never written and stay zero
  for (int i = p; i < kRec; i += L) R[i] = 0.0;

  // The warp takes consecutive rods of the size-sorted queue at a time and
  // factors them in lockstep.
  while (true) {
    int t0 = 0;
    if (lane == 0) t0 = atomicAdd(&a.ctrl[3], kRods);
    t0 = __shfl_sync(full, t0, 0);
    if (t0 >= a.nsys) break;
    const int my = t0 + unit;
    const int s = my < a.nsys ? a.order[my] : -1;
    // Newton bookkeeping of this rod: go = a solve is due this round
    bool go = false;
    if (s >= 0 && a.sys_active[s]) {
      if (a.ls_action && a.ls_action[s] == 1) {  // backtracking: no solve this round
        if (head) atomicAdd(&a.ctrl[0], 1);
      } else {
        const double res = __longlong_as_double((long long)a.sys_res[s]);
        int st = a.sys_status[s];
        if (st == 0 && isnan(res)) st = DM_ERR_NONFINITE;
        if (st == 0 && res <= a.tol) {  // converged at this iterate
          if (head) a.sys_active[s] = 0;
        } else {
          if (st == 0 && a.sys_iters[s] >= a.max_iter) st = DM_ERR_NOT_CONVERGED;
          if (st != 0) {
            if (head) {
              a.sys_status[s] = st;
              a.sys_active[s] = 0;
              atomicAdd(&a.ctrl[1], 1);
              atomicMin(&a.ctrl[2], s);
            }
          } else {
            go = true;
          }
        }
      }
    }
    __syncwarp();
    if (!__any_sync(full, go)) continue;
    const int n = go ? a.sys_ndof[s] : 0;
    Chain c{a.band, a.f, a.rec, (size_t)a.nd, go ? (size_t)a.sys_dof0[s] : 0, n, half ? -1 : 1};
    // split: top eliminates [0, m), bottom [m + 10, n), separator [m, m + 10)
    const bool twist = n >= 32;
    const int m = twist ? (n - 10) / 2 : n;
    const int ncol = !go ? 0 : (half ? (twist ? n - m - 10 : 0) : m);
    const int rows = ncol ? min(ncol + 10, n) : 0;  // the chain's columns and the window below the last
    const int nblk = (ncol + kBlk - 1) / kBlk;
    const int nwarp = (int)__reduce_max_sync(full, (unsigned)nblk);
    bool bad = false;
    stage_rows<L>(c, W, 0, rows, p);
    stage_rows<L>(c, W + 12 * kBlk, kBlk, rows, p);
    cp_async_commit();
    cp_async_wait_all();
    __syncwarp();
    double rj = rcp_int(W[0]);
    for (int b = 0; b < nwarp; ++b) {
      const int j0 = b * kBlk;
      double *cur = W + (b & 1 ? kWin : 0), *nxt = W + (b & 1 ? 0 : kWin);
      const bool more = j0 + kBlk < ncol;  // another block of this chain
      if (more) stage_rows<L>(c, nxt + 12 * kBlk, j0 + 2 * kBlk, rows, p);
      cp_async_commit();
      // the original diagonal entries of the block's rows, for the pivot test
      double diag[2] = {0.0, 0.0};
#pragma unroll
      for (int h = 0; h < (L == 16 ? 1 : 2); ++h)
        if (p + L * h < kBlk && j0 + p + L * h < ncol) diag[h] = c.band[c.at(j0 + p + L * h)];
#pragma unroll
      for (int u = 0; u < kBlk; ++u) column<L, ENV>(ln, ENV ? (u & 3) : 0, u, 0, 0, rj, j0 + u < ncol, cb);
      ln.shift(b & 1 ? -8 * kWin : 8 * kWin);
#pragma unroll
      for (int h = 0; h < (L == 16 ? 1 : 2); ++h)
        if (p + L * h < kBlk && j0 + p + L * h < ncol && pivot_bad(cur[12 * (p + L * h)], diag[h])) bad = true;
      store_records<L>(c, R, j0, min(kBlk, ncol - j0), p);
      cp_async_wait_all();
      if (more) {
#pragma unroll
        for (int e = 0; e < 12 * kBlk; e += L) nxt[e + p] = cur[12 * kBlk + e + p];
      }
      __syncwarp();
    }
    if (nwarp & 1) ln.shift(-8 * kWin);
    // a rod is bad if either of its chains met a zero pivot
    bad = (__ballot_sync(full, bad) & rod_mask) != 0;
    if (bad && go) {
      if (head) {
        a.sys_status[s] = DM_ERR_DEGENERATE;
        a.sys_active[s] = 0;
        atomicAdd(&a.ctrl[1], 1);
        atomicMin(&a.ctrl[2], s);
      }
      go = false;
    }
    // separator: S = top window + bottom window - original (10 x 10, lower),
    // right-hand side likewise, in the top chain's other buffer; then ten
    // more columns of the top chain, with the full band
    const bool sep = go && twist && half == 0;
    const int s_buf = nblk & 1 ? kWin : 0, f_buf = kWin - s_buf;
    double *S = W + s_buf;
    if (sep) {
      const double *Wb = W + kChain;
      const int mb = n - m - 10, nbb = (mb + kBlk - 1) / kBlk;
      const double *ft = W + f_buf + 12 * (m - kBlk * (nblk - 1));
      const double *fb = Wb + (nbb & 1 ? 0 : kWin) + 12 * (mb - kBlk * (nbb - 1));
      for (int e = p; e < 20 * 12; e += L) {
        const int i = e / 12, d = e - 12 * i;
        double v = 0.0;
        if (i < 10) {
          if (d == 11) v = ft[e] + fb[(9 - i) * 12 + 11] - a.f[c.base + m + i];
          else if (d <= i) v = ft[e] + fb[(9 - i + d) * 12 + d] - a.band[d * (size_t)a.nd + c.base + m + i];
        }
        S[e] = v;
      }
    }
    __syncwarp();
    if (__any_sync(full, sep)) {
      rj = rcp_int(S[0]);
#pragma unroll 2
      for (int u = 0; u < 10; ++u) column<L, ENV>(ln, 0, 0, 8 * s_buf + 96 * u, 96 * u, rj, sep, cb);
      bool sbad = false;
      if (sep) {
        for (int u = p; u < 10; u += L) {  // zero, subnormal, infinite, NaN, or of subnormal reciprocal
          const unsigned h = ((unsigned)__double2hiint(S[12 * u]) & 0x7FFFFFFFu) >> 20;
          if (h - 1u >= 2044u) sbad = true;
        }
        store_records<L>(c, R, m, 10, p);
      }
      if ((__ballot_sync(full, sbad) & rod_mask) != 0 && go) {
        if (head) {
          a.sys_status[s] = DM_ERR_DEGENERATE;
          a.sys_active[s] = 0;
          atomicAdd(&a.ctrl[1], 1);
          atomicMin(&a.ctrl[2], s);
        }
        go = false;
      }
    }
    __syncwarp();
    // Back substitution x_k = z_k - sum_d L[k+d][k] x_{k+d}, one row per
    // step t: the top chain takes row m + 9 - t (the separator first), the
    // bottom chain follows 20 steps behind its end: in steps 10..19 it takes
    // the separator's x in its own order from shared memory, from step 20 on its rows.
    // The row of step t is pending in lane t mod L of the chain; the step
    // takes its x by a shuffle and subtracts its part from the rows of the
    // next ten steps (record word d = 1..10; word 11 is zero, for the lanes
    // with a row further on).  With eight lanes a lane holds two of these
    // rows.  Each lane stages its own records, two groups of L steps ahead.
    constexpr int kSlots = 16 / L, kRing = 2 + kSlots;
    const int nrow = !go ? 0 : (half ? ncol : (twist ? m + 10 : n));
    const int R0 = half ? nrow + 19 : nrow - 1;  // the row of step t is R0 - t
    double *ring = W + 12 * kRing * p;
    static_assert(kRing * 12 * L <= kWindow, "ring");
    auto fetch = [&](int g) {  // the lane's record of step group g
      const int r = R0 - (L * g + p);
      double *dst = ring + 12 * (g % kRing);
      if (r >= 0 && r < nrow) {
        const double *src = c.rec + 12 * c.at(r);
#pragma unroll
        for (int e = 0; e < 12; e += 2) cp_async16(dst + e, src + e);
      } else {  // no such row: nothing of it may be infinite or NaN
#pragma unroll
        for (int e = 0; e < 12; e += 2) *reinterpret_cast<double2 *>(dst + e) = make_double2(0.0, 0.0);
      }
    };
#pragma unroll
    for (int g = 0; g < kRing; ++g) fetch(g);
    cp_async_commit();
    cp_async_wait_all();
    const int steps = nrow == 0 ? 0 : R0 + 1;
    const int groups = (int)__reduce_max_sync(full, (unsigned)((steps + L - 1) / L));
    double *xs = wsm + (chain & ~1) * kChain + kWindow;  // the top chain's record area: separator x
    double v[kSlots];
#pragma unroll
    for (int k = 0; k < kSlots; ++k) v[k] = ring[12 * k];
    int idx[L], idy[L];
#pragma unroll
    for (int u = 0; u < L; ++u) {
      const int d = (p - u) & (L - 1);  // 0: this step's own lane, whose next row is L steps on
      idx[u] = L == 16 ? (d == 0 || d > 11 ? 11 : d) : (d == 0 ? 8 : d);
      idy[u] = min(idx[u] + 8, 11);
    }
    double *qx = a.q + c.base;
    for (int g = 0; g < groups; ++g) {
      double x_own = 0.0;
      const double *ra = ring + 12 * (g % kRing), *rb = ring + 12 * ((g + 1) % kRing);
      const double *rc = ring + 12 * ((g + kSlots) % kRing);
      const double zn = rc[0];
#pragma unroll
      for (int u = 0; u < L; ++u) {
        double x = __shfl_sync(full, v[0], cb + u);
        const int t = L * g + u;
        if (t < 20 && t >= 10) {  // the separator's x, known since step 9
          if (half && twist) x = xs[19 - t];
        }
        const bool own = p == u;
        if (own) {
          x_own = x;
          if (kSlots > 1) v[0] = v[kSlots - 1];
          v[kSlots - 1] = zn;
        }
        const double ca = (own || p < u ? rb : ra)[idx[u]];
        v[0] = fma(-ca, x, v[0]);
        if (kSlots > 1) {
          const double cc = (own || p < u ? rc : rb)[idy[u]];
          v[kSlots - 1] = fma(-cc, x, v[kSlots - 1]);
        }
        if (t == 9 || (t < 9 && u == L - 1)) {  // the top chain's x of the steps so far
          if (!half && L * g + p <= t) xs[L * g + p] = x_own;
          __syncwarp();
        }
      }
      const int r = R0 - (L * g + p);
      if (r >= 0 && r < nrow) {
        const int o = c.dir > 0 ? r : n - 1 - r;
        if (a.direct) qx[o] = x_own;
        else atomicAdd(qx + o, -x_own);
      }
      fetch(g + kRing);
      cp_async_commit();
      asm volatile("cp.async.wait_group 1;\n" ::: "memory");
    }
    cp_async_wait_all();
    if (go && head) {
      a.sys_iters[s] += 1;
      if (a.ls_trial) a.ls_trial[s] = 1;
      atomicAdd(&a.ctrl[0], 1);
      if (a.units) atomicAdd(a.units, (unsigned long long)n);
    }
    __syncwarp();
    // the separator's records and x lay over the records' zero rows
    for (int i = p; i < kRec; i += L) R[i] = 0.0;
    __syncwarp();
  }
}

template <int L, bool ENV>
cudaError_t launch(const SolveArgs &a, int blocks, int warps, cudaStream_t st) {
  const size_t smem = rod_solve_smem(L, warps);
  // the largest block of this instance, so that no caller's smaller one lowers the limit
  cudaError_t e = cudaFuncSetAttribute(k_solve_rod<L, ENV>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)rod_solve_smem(L, 4));
  if (e != cudaSuccess) return e;
  k_solve_rod<L, ENV><<<blocks, 32 * warps, smem, st>>>(a);
  return cudaGetLastError();
}

template <int L, bool ENV>
cudaError_t occupancy(int warps, int *per_sm) {
  cudaError_t e = cudaFuncSetAttribute(k_solve_rod<L, ENV>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)rod_solve_smem(L, 4));
  if (e != cudaSuccess) return e;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(per_sm, k_solve_rod<L, ENV>, 32 * warps,
                                                       rod_solve_smem(L, warps));
}

}  // namespace

// Sixteen lanes per chain while that leaves at most two warps per SM
// partition: fewer instructions per column on the longest rods' chains
// (301 rods: see above); beyond it the eight-lane split, which spends 10.75
// FP64 slots per row on four chains instead of 6.5 on two.
int rod_solve_lanes(int nrods, int sms) { return nrods <= 8 * sms ? 16 : 8; }

size_t rod_solve_smem(int lanes, int warps) {
  return (size_t)warps * ((32 / lanes) * kChain + kRec) * sizeof(double);
}

cudaError_t rod_solve_occupancy(int lanes, bool env, int warps, int *per_sm) {
  if (lanes == 16) return env ? occupancy<16, true>(warps, per_sm) : occupancy<16, false>(warps, per_sm);
  return env ? occupancy<8, true>(warps, per_sm) : occupancy<8, false>(warps, per_sm);
}

cudaError_t rod_solve_launch(const SolveArgs &a, int lanes, bool env, int blocks, int warps,
                             cudaStream_t st) {
  if (lanes == 16)
    return env ? launch<16, true>(a, blocks, warps, st) : launch<16, false>(a, blocks, warps, st);
  return env ? launch<8, true>(a, blocks, warps, st) : launch<8, false>(a, blocks, warps, st);
}

}  // namespace dm
