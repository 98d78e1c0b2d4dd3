// Condensation solve of the Newton system J dq = -f for general systems
// whose limbs couple to the border only through the rows at one end (rods
// attached at one end: star robots; single rods on the ground).
//
//   1. k_gen_limb_factor (one warp per limb): forms the limb's band of the
//      Jacobian in shared memory straight from the stencil, edge and node
//      terms (the row formula of a single rod), and eliminates it without
//      pivoting from the free end, with the right-hand side alongside.  What
//      remains is the dense m x m block A_m of the rows next to the border;
//      [A_m C_m y_m; R_m 0 0] is eliminated further, and the limb's Schur
//      complement -R_m A_m^{-1} [C_m | y_m], which that leaves, goes to the
//      border system (atomics on the system's matrix).
//   2. k_gen_border (a block per system): Newton bookkeeping for the system
//      and the dense LU of the border system (in order, partial pivoting
//      where a pivot is tiny).
//   3. k_gen_limb_back (one warp per limb): back substitution from the border
//      values towards the free end; q += dq.
//
// Late Newton rounds carry few systems, so a round costs the length of one
// limb's elimination chain; full rounds cost FP64 slots (64 cycles per warp
// instruction and SM partition).  Per column: the multipliers, the scaled row
// of U and y in one instruction (exchanged through shared memory), the R (R +
// 1) updates dealt evenly over the lanes -- R = 10, 9, 8, 7 in turn, the
// envelope of a rod's Jacobian: 4 slots a column instead of 8 --, the pivot's
// reciprocal on the integer pipe; a pivot outside [2^-126, 2^126) (zero and
// non-finite included) fails the system.  The back substitution keeps the
// pending rows in lane registers: one update and one shuffle per row.
// Measured, 1024 star robots of 3 to 8 limbs of 112 rows, every robot active:
// factor 424 -> 330 us, border 81 -> 69 us, back substitution 102 -> 60 us,
// assembly of the couplings 352 -> 86 us (the limbs' bands are no longer
// stored); a round of few robots: a limb 89 k cycles, 58 k of them its 104
// columns (560 each), 12 k the coupled block, 10 k forming the rows.
//
// The Jacobian is that of Sec. III-C (M/dt^2 - dF/dq, with the contact and
// friction terms of Sec. III-B), not symmetric when friction acts, hence LU.
#include "dm_internal.h"
#include "dm_kernels.cuh"

namespace dm {

namespace {
constexpr int kRow = 22;        // 21 band entries (p, p + k) at k + 10, then the right-hand side
constexpr int kLBlk = 12;       // columns per block, 4-periodic like the envelope
constexpr int kLRec = 12;       // record of an eliminated row: y / d, U(p, p + 1..10) / d, 0
// small block: [A_m C_m y_m; R_m 0 0]; with pivoting instead [A_m | C_m | y_m],
// R_m and the small LU's scratch
constexpr int kSmall = (kFastMaxM + kFastMaxBC) * (kFastMaxM + kFastMaxBC + 1);
static_assert(kSmall >= kFastMaxM * (kFastMaxM + kFastMaxBC + 1) + kFastMaxBC * kFastMaxM + 2 * kFastMaxM, "small");
static_assert(kLimbExtra == 11 * kRow + kLBlk * kLRec + 12 + kSmall && kLimbExtra % 2 == 0, "limb smem layout");
static_assert(kFastMaxRows <= 32 * 2 * kLBlk * kLRec, "a bit per row fits the records");
constexpr unsigned kFull = 0xffffffffu;

// Pivots of an elimination in order smaller than 2^-43 of their starting
// diagonal entry, or not finite, send it to partial pivoting; the test compares
// the upper words (exponent and 20 mantissa bits), off the FP64 pipe.
__device__ __forceinline__ int pivot_floor(double d) {
  return max((__double2hiint(d) & 0x7FFFFFFF) - (43 << 20), 1 << 20);
}
__device__ __forceinline__ bool pivot_ok(double v, int floor) {
  const int h = __double2hiint(v) & 0x7FFFFFFF;
  return h >= floor && h < 0x7FF00000;
}

__device__ __forceinline__ double limb_recip(double d) { return rcp_any(d); }

// The border kernel's decision for system s, without its side effects.
__device__ __forceinline__ bool wants_solve(const SolveGenArgs &a, int s) {
  if (!a.sys_active[s]) return false;
  if (a.ls_action && a.ls_action[s] == 1) return false;
  if (a.sys_status[s] != 0) return false;
  const double res = __longlong_as_double((long long)a.sys_res[s]);
  if (isnan(res) || res <= a.tol) return false;
  return a.sys_iters[s] < a.max_iter;
}

// [A | B] <- [U | A^{-1} B] for a dense n x n matrix A with nrhs
// right-hand sides B beside it (row-major, leading dimension ld >= n + nrhs)
// in shared memory, by one warp: Gaussian elimination with partial
// pivoting, reciprocal pivots, the multipliers of a column by one lane per
// row, the trailing update and the back substitution spread over (row,
// column) pairs -- no lane works through a whole row.  lm and dinv: n
// doubles of scratch each.  Returns false (uniformly) on a zero or
// non-finite pivot.
__device__ bool warp_lu_solve(double *M, int n, int ld, int nrhs, double *lm, double *dinv,
                              int lane) {
  for (int j = 0; j < n; ++j) {
    double best = -1.0;
    int bi = j;
    for (int i = j + lane; i < n; i += 32) {
      const double v = fabs(M[i * ld + j]);
      if (v > best) {
        best = v;
        bi = i;
      }
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) {
      const double ob = __shfl_xor_sync(kFull, best, o);
      const int oi = __shfl_xor_sync(kFull, bi, o);
      if (ob > best || (ob == best && oi < bi)) {
        best = ob;
        bi = oi;
      }
    }
    if (!(best > 0.0) || !isfinite(best)) return false;
    if (bi != j)
      for (int c = j + lane; c < n + nrhs; c += 32) {
        const double t = M[j * ld + c];
        M[j * ld + c] = M[bi * ld + c];
        M[bi * ld + c] = t;
      }
    __syncwarp();
    const double rp = limb_recip(M[j * ld + j]);
    if (lane == 0) dinv[j] = rp;
    for (int i = j + 1 + lane; i < n; i += 32) lm[i] = M[i * ld + j] * rp;
    __syncwarp();
    // rows j+1.., columns j+1 .. n+nrhs-1; the row of pair e by a float
    // reciprocal (e < 2^10, so the quotient is exact after rounding down)
    const int wdt = n + nrhs - j - 1, cnt = (n - j - 1) * wdt;
    const float iw = 1.0f / (float)wdt;
    for (int e = lane; e < cnt; e += 32) {
      const int r = (int)(((float)e + 0.5f) * iw);
      const int i = j + 1 + r, c = j + 1 + e - r * wdt;
      M[i * ld + c] = fma(-lm[i], M[j * ld + c], M[i * ld + c]);
    }
    __syncwarp();
  }
  // back substitution, column by column of U: x_i = y_i / u_ii, then
  // y_k -= u_ki x_i for the rows above
  const float ir = 1.0f / (float)nrhs;
  for (int i = n - 1; i >= 0; --i) {
    for (int c = lane; c < nrhs; c += 32) M[i * ld + n + c] *= dinv[i];
    __syncwarp();
    for (int e = lane; e < i * nrhs; e += 32) {
      const int k = (int)(((float)e + 0.5f) * ir), c = e - k * nrhs;
      M[k * ld + n + c] = fma(-M[k * ld + i], M[i * ld + n + c], M[k * ld + n + c]);
    }
    __syncwarp();
  }
  return true;
}

}  // namespace

namespace {

// Update tasks of a column with R rows below it, in order: row i = 1..R, the
// entries under column k = 1..R, the right-hand side; task t is lane t mod
// 32's slot t / 32 (the next pivot (1, 1): lane 0's first); spare slots repeat
// the lane's first.
__host__ __device__ constexpr int limb_slots(int R) { return (R * (R + 1) + 31) / 32; }

// Columns of a limb before the first one with ten rows below it: that is an x
// (rod row 0 mod 4) of a limb eliminated from its first row, a z (2 mod 4) of
// one eliminated from its last.  Limbs with a free end start there (rods have
// 4 N - 1 rows); one whose border was fixed away starts at the twist angle
// behind it, with seven rows.
__host__ __device__ constexpr int limb_lead(int first, int n, int dir) {
  return dir ? (first + n - 1 + 2) & 3 : (4 - (first & 3)) & 3;
}

struct LimbLane {
  int to[4][4], uo[4][4], lo[4][4];  // byte offsets by column type: target, U entry, multiplier
  int so, ro;                        // the lane's product with the reciprocal: source, destination
  bool walks;                        // ... in the record (moves with the column)
  __device__ __forceinline__ void load(int lane, int rec, int lw) {
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      const int R = 10 - t;
#pragma unroll
      for (int h = 0; h < 4; ++h) {
        if (h >= limb_slots(R)) continue;
        int e = lane + 32 * h;
        if (e >= R * (R + 1)) e = lane;
        const int i = e / (R + 1) + 1, k = e - (i - 1) * (R + 1) + 1;  // k = R + 1: right-hand side
        to[t][h] = 8 * (kRow * i + (k <= R ? 10 + k - i : 21));
        uo[t][h] = 8 * (k <= R ? 10 + k : 21);
        lo[t][h] = lw + 8 * (i - 1);
      }
    }
    // lanes 0-9: the multiplier of row i = lane + 1; 10-19: U; 20 on: y
    so = 8 * (lane < 10 ? kRow * (lane + 1) + 9 - lane : lane < 20 ? lane + 1 : 21);
    walks = lane >= 10;
    ro = lane < 10 ? lw + 8 * lane : rec + 8 * (lane < 20 ? lane - 9 : 0);
  }
};

extern __shared__ __align__(16) char g_lsm[];
__device__ __forceinline__ double &lsm(int off) { return *reinterpret_cast<double *>(g_lsm + off); }

// Column u of a block whose pivot row is `w` bytes in; rj its pivot's
// reciprocal (in), the next column's (out).  The reciprocal's chain starts at
// the first update; the other updates are tied to its steps (RcpChain), since
// in-order issue would hold the chain back behind them (64 cycles each).
__device__ __forceinline__ void limb_column(const LimbLane &ln, const int t, const int u, int w, double &rj, bool act,
                                            unsigned zero) {
  const int NK = limb_slots(10 - t), wu = w + 8 * kRow * u;
  lsm(ln.ro + (ln.walks ? 8 * kLRec * u : 0)) = lsm(ln.so + wu) * rj;
  double uq[4], dv[4], v[4];
#pragma unroll
  for (int h = 0; h < 4; ++h)
    if (h < NK) {
      uq[h] = lsm(ln.uo[t][h] + wu);
      dv[h] = lsm(ln.to[t][h] + wu);
    }
  __syncwarp();
  v[0] = fma(-lsm(ln.lo[t][0]), uq[0], dv[0]);
  v[1] = fma(-lsm(ln.lo[t][1]), uq[1], dv[1]);
  RcpChain ch;
  ch.seed(__shfl_sync(kFull, v[0], 0));
  if (NK > 2) v[2] = fma(-lsm(ln.lo[t][2]), after(uq[2], ch.S, zero), dv[2]);
  ch.residual();
  if (NK > 3) v[3] = fma(-lsm(ln.lo[t][3]), after(uq[3], (unsigned)ch.t, zero), dv[3]);
  rj = ch.result();
  if (act) {
#pragma unroll
    for (int h = 0; h < 4; ++h)
      if (h < NK) lsm(ln.to[t][h] + wu) = v[h];
  }
  __syncwarp();
}

// packed upper-triangle index of an 11 x 11 symmetric matrix (i <= j)
__host__ __device__ constexpr int up11(int i, int j) { return i * 11 - i * (i - 1) / 2 + (j - i); }

struct LimbRows {
  int N, st, e0, f, n, d0, dir;  // rod nodes, stencil of rod node 1, first edge, limb's rod row, rows, DOF, direction
  const unsigned *fmask;         // the limb's fixed rows, a bit each
  double *A;
};

// Rod row 4 node + C (a lane per node, C a constant: every index below is one)
// of the limb into its band (entry (r, r - d) and its mirror image; zeroed
// before): the lower band row of a single rod's Jacobian -- stencils m = node
// - 1, node, node + 1 (4m-4 <= r <= 4m+6; joints sit at rod ends, so a rod's
// stencils and edges run along it), the edges at its node, M/dt^2 and damping
// -- and the node's 3 x 3 ground terms, which friction makes nonsymmetric
// (`trans`: their transpose, hence the transposed matrix).  Entries to rows
// outside the limb are border coupling.
template <int C>
__device__ __forceinline__ void limb_row(const SolveGenArgs &a, const LimbRows &q, int node) {
  const int k = 4 * node + C - q.f;
  if (k < 0 || k >= q.n) return;
  const int g = q.d0 + k;  // DOF
  const double *sh = a.sh + q.st + node - 1;  // entry e of stencil m = node + h: sh[e ns + h]
  const bool s0 = node >= 2, s1 = node >= 1 && node <= q.N - 2, s2 = node <= q.N - 3;
  constexpr int L0 = 8 + C, L1 = 4 + C, L2 = C;  // the row's place in the three stencils
  double b[11], b1[11], b2[11];
#pragma unroll
  for (int d = 0; d < 11; ++d) {
    b[d] = C < 3 && d <= L0 && s0 ? sh[(size_t)up11(L0 - d, L0) * a.ns - 1] : 0.0;
    b1[d] = d <= L1 && s1 ? sh[(size_t)up11(L1 - d, L1) * a.ns] : 0.0;
    b2[d] = d <= L2 && s2 ? sh[(size_t)up11(L2 - d, L2) * a.ns + 1] : 0.0;
  }
  const double dc = a.dconst[g];
  // edges: the one that starts at the node (its block's entries under the
  // diagonal), the one that ends there (its whole row of the block), and the
  // ground terms: row C and column C of the node's block
  double es[3] = {0.0, 0.0, 0.0}, ee[3] = {0.0, 0.0, 0.0}, gx[3] = {0.0, 0.0, 0.0}, gy[3] = {0.0, 0.0, 0.0};
  if (C < 3) {
    const int v = a.nt ? a.dof_node[g] : 0;
#pragma unroll
    for (int cp = 0; cp < 3; ++cp) {
      const int lo = cp < C ? cp : C, hi = cp < C ? C : cp;
      const double *src = a.es + (size_t)(3 + (lo == 0 ? hi : lo == 1 ? 2 + hi : 5)) * a.ne + q.e0 + node;
      if (cp <= C && node <= q.N - 2) es[cp] = src[0];
      if (node >= 1) ee[cp] = src[-1];
      if (a.nt && cp <= C) {
        gx[cp] = a.nt[(size_t)(3 + 3 * C + cp) * a.nn + v];
        gy[cp] = a.nt[(size_t)(3 + 3 * cp + C) * a.nn + v];
      }
    }
  }
  // bit d: row k - d is fixed (rows before the limb count as fixed)
  const int w = k >> 5;
  const unsigned fx = __brev(__funnelshift_l(w > 0 ? q.fmask[w - 1] : ~0u, q.fmask[w], 31 - (k & 31)));
  const int p = q.dir ? q.n - 1 - k : k, s = q.dir ? 1 : -1;
  double *A = q.A + p * kRow + 10;
  if (fx & 1u) {
    A[0] = dc;
    return;
  }
#pragma unroll
  for (int d = 0; d < 11; ++d) {
    if (d <= L1) b[d] = C < 3 ? b[d] + b1[d] : b1[d];
    if (d <= L2) b[d] += b2[d];
  }
  b[0] += dc;
  double up[3] = {0.0, 0.0, 0.0};  // what the mirror image of b[1], b[2] has more (friction)
  if (C < 3) {
#pragma unroll
    for (int cp = 0; cp < 3; ++cp) {
      if (cp <= C) {
        b[C - cp] += es[cp] + ee[cp] + (a.trans ? gy[cp] : gx[cp]);
        up[C - cp] = a.trans ? gx[cp] - gy[cp] : gy[cp] - gx[cp];
      }
      b[4 + C - cp] -= ee[cp];
    }
  }
  A[0] = b[0];
#pragma unroll
  for (int d = 1; d < 11; ++d) {
    if (d > (C < 3 ? L0 : L1) || ((fx >> d) & 1u)) continue;
    A[s * d] = b[d];
    A[s * d * kRow - s * d] = d < 3 ? b[d] + up[d] : b[d];
  }
}

}  // namespace

__global__ void __launch_bounds__(128) k_gen_limb_factor(SolveGenArgs a) {
  const int wi = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int L = blockIdx.x * (blockDim.x >> 5) + wi;
  if (L >= a.nlimb) return;
  const int w = a.lb_gsys[L];
  if (!a.gs_fast[w]) return;
  const int s = a.gen_sys[w];
  if (!wants_solve(a, s)) return;
  // per warp: the band [n + 11][22] (eleven zero rows behind it), a block's
  // records, the multipliers of a column, the small block
  const int per = a.limb_nmax * kRow + kLimbExtra;
  double *A = reinterpret_cast<double *>(g_lsm) + (size_t)wi * per;
  const int n = a.lb_n[L], m = a.lb_m[L], nbc = a.lb_nbc[L], dir = a.lb_dir[L];
  double *rec = A + a.limb_nmax * kRow + 11 * kRow, *lw = rec + kLBlk * kLRec, *M = lw + 12;
  const int d0 = a.lb_dof0[L], f = a.lb_first[L];
  double *G = a.gen;
  double *U = G + a.lb_y[L];  // [n][12] records of the rows, out
  // (C_m and R_m arrive while the limb is eliminated: the block's first m
  // rows' last columns, the rows after them)
  const int ldm = m + nbc + 1;
  {
    const double *C = G + a.lb_C[L], *R = G + a.lb_R[L];
    for (int e = lane; e < m * nbc; e += 32) {
      const int r = e / nbc, c = e / m;
      cp_async8(M + r * ldm + m + e - r * nbc, C + e);
      cp_async8(M + (m + c) * ldm + e - c * m, R + e);
    }
    cp_async_commit();
  }
  const int rod = a.lb_rod[L];
  LimbRows q{a.npr[rod], 0, a.rod_edge0[rod], f, n, d0, dir, reinterpret_cast<unsigned *>(rec), A};
  q.st = q.N > 2 ? a.slot2st[a.rod_slot0[rod]] : 0;
  for (int e = lane; e < (n + 11) * kRow / 2; e += 32) reinterpret_cast<double2 *>(A)[e] = make_double2(0.0, 0.0);
#pragma unroll 4
  for (int k0 = 0; k0 < n; k0 += 32) {
    const bool fx = k0 + lane < n && a.fixed[d0 + k0 + lane];
    const unsigned bits = __ballot_sync(kFull, fx);
    if (lane == 0) reinterpret_cast<unsigned *>(rec)[k0 >> 5] = bits;
  }
  __syncwarp();
  for (int node = (f >> 2) + lane; 4 * node < f + n; node += 32) {
    limb_row<0>(a, q, node);
    limb_row<1>(a, q, node);
    limb_row<2>(a, q, node);
    limb_row<3>(a, q, node);
  }
#pragma unroll 4
  for (int p = lane; p < n; p += 32) A[p * kRow + 21] = -a.f[d0 + (dir ? n - 1 - p : p)];
  __syncwarp();
  for (int e = lane; e < kLBlk * kLRec; e += 32) rec[e] = 0.0;  // (their last words stay zero)
  LimbLane ln;
  const int w0 = (int)(reinterpret_cast<char *>(A) - g_lsm);
  ln.load(lane, (int)(reinterpret_cast<char *>(rec) - g_lsm), (int)(reinterpret_cast<char *>(lw) - g_lsm));
  __syncwarp();
  const int ne = n - m;  // rows eliminated inside the limb
  bool bad = false;
  double rj = rcp_any(A[10]);
  // after columns j0 .. j0 + cnt - 1: their pivots' range, their records
  const auto finish = [&](int j0, int cnt) {
    if (lane < cnt && !rcp64_in_range(A[(j0 + lane) * kRow + 10])) bad = true;
    for (int e = lane; e < cnt * (kLRec / 2); e += 32)
      *reinterpret_cast<double2 *>(U + (size_t)j0 * kLRec + 2 * e) = *reinterpret_cast<const double2 *>(rec + 2 * e);
    __syncwarp();
  };
  // the columns before the envelope's first one of ten rows, with all ten rows
  const int lead = min(limb_lead(f, n, dir), ne);
#pragma unroll 1
  for (int u = 0; u < lead; ++u) limb_column(ln, 0, u, w0, rj, true, a.zero);
  if (lead > 0) finish(0, lead);
  for (int j0 = lead; j0 < ne; j0 += kLBlk) {
#pragma unroll
    for (int u = 0; u < kLBlk; ++u) limb_column(ln, u & 3, u, w0 + 8 * kRow * j0, rj, j0 + u < ne, a.zero);
    finish(j0, min(kLBlk, ne - j0));
  }
  bad = __any_sync(kFull, bad);
  if (!bad && m > 0) {
    // [A_m C_m y_m; R_m 0 0], eliminated in order; a pivot below 2^-43 of its
    // starting diagonal entry, or not finite, sends the limb to partial pivoting
    const int rows = m + nbc;
    cp_async_wait_all();
    for (int e = lane; e < m * (m + 1); e += 32) {
      const int r = e / (m + 1), c = e - r * (m + 1);
      M[r * ldm + (c < m ? c : rows)] = A[(ne + r) * kRow + (c < m ? 10 + c - r : 21)];
    }
    for (int e = lane; e < nbc * (nbc + 1); e += 32) {
      const int r = e / (nbc + 1);
      M[(m + r) * ldm + m + e - r * (nbc + 1)] = 0.0;
    }
    const int thr = lane < m ? pivot_floor(A[(ne + lane) * kRow + 10]) : 0;
    __syncwarp();
    bool ok = true;
    for (int c = 0; c < m; ++c) {
      const double pv = M[c * ldm + c];
      if (!pivot_ok(pv, __shfl_sync(kFull, thr, c))) {
        ok = false;  // uniform
        break;
      }
      const int wd = rows - c;  // entries right of the pivot
      const double rp = rcp_any(pv);
      if (lane < wd) M[c * ldm + c + 1 + lane] *= rp;
      __syncwarp();
      // rows c+1.., a lane per column: two rows at a time once 16 lanes do
      const bool twin = wd <= 16;
      const int col = c + 1 + (twin ? lane & 15 : lane), stp = twin ? 2 : 1;
      if (col <= rows) {
        const double u = M[c * ldm + col];
#pragma unroll 4
        for (int i = c + 1 + (twin ? lane >> 4 : 0); i < rows; i += stp)
          M[i * ldm + col] = fma(-M[i * ldm + c], u, M[i * ldm + col]);
      }
      __syncwarp();
    }
    double *Z = G + a.lb_Y[L];
    const int32_t *bc = a.lb_bcols + a.lb_bc0[L];
    const int nB = a.gs_nB[w], ldb = nbc + 1;
    double *S = G + a.gs_JBB[w], *rB = G + a.gs_rB[w];
    if (ok) {
      // the condensed rows for the back substitution: U right of the pivot
      // within the block, the couplings to the border and y over the pivot
      for (int e = lane; e < m * kLRec; e += 32) {
        const int r = e / kLRec, k = e - r * kLRec;
        U[(size_t)ne * kLRec + e] = k >= 1 && r + k < m ? M[r * ldm + r + k] : 0.0;
      }
      for (int e = lane; e < m * ldb; e += 32) {
        const int r = e / ldb;
        Z[e] = M[r * ldm + m + e - r * ldb];
      }
      for (int e = lane; e < nbc * ldb; e += 32) {
        const int b1 = e / ldb, b2 = e - b1 * ldb;
        const double v = M[(m + b1) * ldm + m + b2];
        if (b2 < nbc) atomicAdd(S + (int64_t)bc[b1] * nB + bc[b2], v);
        else atomicAdd(rB + bc[b1], v);
      }
    } else {
      __syncwarp();
      const double *C = G + a.lb_C[L], *R = G + a.lb_R[L];
      const int ld = m + ldb;
      double *Rs = M + kFastMaxM * (kFastMaxM + kFastMaxBC + 1);
      double *lm = Rs + kFastMaxBC * kFastMaxM, *dinv = lm + kFastMaxM;
      for (int e = lane; e < m * ld; e += 32) {
        const int r = e / ld, c = e - r * ld;
        M[e] = c < m ? A[(ne + r) * kRow + 10 + c - r] : c < m + nbc ? C[r * nbc + c - m] : A[(ne + r) * kRow + 21];
      }
      for (int e = lane; e < nbc * m; e += 32) Rs[e] = R[e];
      __syncwarp();
      if (!warp_lu_solve(M, m, ld, ldb, lm, dinv, lane)) {
        bad = true;
      } else {
        // Z = A_m^{-1} [C_m | y_m]: the condensed rows without each other
        for (int e = lane; e < m * kLRec; e += 32) U[(size_t)ne * kLRec + e] = 0.0;
        for (int e = lane; e < m * ldb; e += 32) {
          const int r = e / ldb;
          Z[e] = M[r * ld + m + e - r * ldb];
        }
        // Schur complement and right-hand side of the border system
        for (int e = lane; e < nbc * ldb; e += 32) {
          const int b1 = e / ldb, b2 = e - b1 * ldb;
          double v = 0.0;
          for (int r = 0; r < m; ++r) v = fma(Rs[b1 * m + r], M[r * ld + m + b2], v);
          if (b2 < nbc) atomicAdd(S + (int64_t)bc[b1] * nB + bc[b2], -v);
          else atomicAdd(rB + bc[b1], -v);
        }
      }
    }
  }
  cp_async_wait_all();
  if (bad && lane == 0) atomicOr(a.gen_bad + w, 1);
}

// The border system [S | r] (row-major, leading dimension nB + 1, right-hand
// side in the last column) solved by a block of kGenBorderThreads: Gaussian
// elimination in order, the trailing update spread over all threads (one
// matrix entry per thread and step) and the next pivot's reciprocal taken by
// the thread that updates it, so one barrier per column; a pivot below
// 2^-43 of its original diagonal entry restarts the elimination with
// partial pivoting (the pivot search, row swap and multipliers by warp 0).
// Then a column-oriented back substitution by warp 0 with the right-hand
// sides in registers (rows lane, lane + 32, lane + 64).
__global__ void __launch_bounds__(kGenBorderThreads) k_gen_border(SolveGenArgs a) {
  extern __shared__ double sm[];
  __shared__ int flag[4];  // go, bad, -, pivot ok
  const int w = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nt = blockDim.x;
  if (w >= a.ngen || !a.gs_fast[w]) return;  // block-uniform
  const int s = a.gen_sys[w];
  if (tid == 0) {
    int go = 0, bad = 0;
    if (a.sys_active[s] && a.ls_action && a.ls_action[s] == 1) {
      atomicAdd(&a.ctrl[0], 1);  // backtracking: no solve this round
    } else if (a.sys_active[s]) {
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
    if (go) {
      bad = a.gen_bad[w];
      a.gen_bad[w] = 0;
    }
    flag[0] = go;
    flag[1] = bad;
  }
  __syncthreads();
  const int go = flag[0];
  bool bad = flag[1] != 0;
  const int nB = a.gs_nB[w];
  const int ld = nB + 1;
  double *S = sm, *rinv = sm + (size_t)nB * ld, *lm = rinv + nB;
  int *least = reinterpret_cast<int *>(lm + nB);  // per row: the smallest pivot taken
  const int32_t *bd = a.border_dof + a.gs_border0[w];
  double *J = a.gen + a.gs_JBB[w];
  double *acc = a.gen + a.gs_rB[w];
  // the border block [S | r] from the assembled block and the limbs' Schur sums
  // (asynchronous copies for the matrix, all in flight at once)
  auto load = [&]() {
    for (int e = tid; e < nB * nB; e += nt) {
      const int r = e / nB;
      cp_async8(S + r * ld + e - r * nB, J + e);
    }
    cp_async_commit();
    for (int b = tid; b < nB; b += nt) S[b * ld + nB] = acc[b] - a.f[bd[b]];
    cp_async_wait_all();
  };
  if (go && !bad && nB > 0) {
    load();
    __syncthreads();
    for (int b = tid; b < nB; b += nt) least[b] = pivot_floor(S[b * ld + b]);
    if (tid == 0) flag[3] = 1;
    __syncthreads();
    // first attempt: elimination in order, without pivoting; the thread that
    // updates the next pivot takes its reciprocal (one barrier per column).
    // A pivot below 2^-43 of its original diagonal entry, or not
    // finite, abandons it for partial pivoting.
    if (tid == 0) {
      const double v = S[0];
      if (!pivot_ok(v, least[0])) flag[3] = 0;
      else rinv[0] = limb_recip(v);
    }
    __syncthreads();
    for (int j = 0; j < nB && flag[3]; ++j) {
      const double rp = rinv[j];
      const int nc = nB - j;
      const float inv = 1.0f / (float)nc;
      for (int e = tid; e < (nB - j - 1) * nc; e += nt) {
        const int r = (int)(((float)e + 0.5f) * inv);
        const int i = j + 1 + r, c = j + 1 + e - r * nc;
        const double v = fma(-(S[i * ld + j] * rp), S[j * ld + c], S[i * ld + c]);
        S[i * ld + c] = v;
        if (r == 0 && c == j + 1) {
          if (!pivot_ok(v, least[j + 1])) flag[3] = 0;
          else rinv[j + 1] = limb_recip(v);
        }
      }
      __syncthreads();
    }
    if (!flag[3]) {
      // partial pivoting on a fresh copy
      __syncthreads();
      load();
      __syncthreads();
      for (int j = 0; j < nB; ++j) {
        // warp 0: pivot search, row swap, reciprocal and multipliers
        if (warp == 0) {
          double best = -1.0;
          int bi = j;
          for (int i = j + lane; i < nB; i += 32) {
            const double v = fabs(S[i * ld + j]);
            if (v > best) {
              best = v;
              bi = i;
            }
          }
#pragma unroll
          for (int o = 16; o; o >>= 1) {
            const double ob = __shfl_xor_sync(kFull, best, o);
            const int oi = __shfl_xor_sync(kFull, bi, o);
            if (ob > best || (ob == best && oi < bi)) {
              best = ob;
              bi = oi;
            }
          }
          const bool ok = (best > 0.0) && isfinite(best);
          if (ok) {
            if (bi != j)
              for (int c = j + lane; c <= nB; c += 32) {
                const double t = S[j * ld + c];
                S[j * ld + c] = S[bi * ld + c];
                S[bi * ld + c] = t;
              }
            __syncwarp();
            const double rp = limb_recip(S[j * ld + j]);
            if (lane == 0) rinv[j] = rp;
            for (int i = j + 1 + lane; i < nB; i += 32) lm[i] = S[i * ld + j] * rp;
          }
          if (lane == 0) flag[3] = ok;
        }
        __syncthreads();
        if (!flag[3]) {
          bad = true;
          break;  // uniform
        }
        // rows j+1.., columns j+1..nB (the right-hand side included); the row
        // of entry e by a float reciprocal: the quotient is below 96 and at
        // least 0.5/96 from an integer, its float error below 2e-5
        const int nc = nB - j;
        const float inv = 1.0f / (float)nc;
        for (int e = tid; e < (nB - j - 1) * nc; e += nt) {
          const int r = (int)(((float)e + 0.5f) * inv);
          const int i = j + 1 + r, c = j + 1 + e - r * nc;
          S[i * ld + c] = fma(-lm[i], S[j * ld + c], S[i * ld + c]);
        }
        __syncthreads();
      }
    }
    if (!bad && warp == 0) {
      double b0 = lane < nB ? S[lane * ld + nB] : 0.0;
      double b1 = lane + 32 < nB ? S[(lane + 32) * ld + nB] : 0.0;
      double b2 = lane + 64 < nB ? S[(lane + 64) * ld + nB] : 0.0;
      for (int i = nB - 1; i >= 0; --i) {
        const int hi = i >> 5;
        const double src = hi == 0 ? b0 : (hi == 1 ? b1 : b2);
        const double xi = __shfl_sync(kFull, src, i & 31) * rinv[i];
        if (lane == 0) lm[i] = xi;
        if (lane < i) b0 = fma(-S[lane * ld + i], xi, b0);
        if (lane + 32 < i) b1 = fma(-S[(lane + 32) * ld + i], xi, b1);
        if (lane + 64 < i) b2 = fma(-S[(lane + 64) * ld + i], xi, b2);
      }
    }
    __syncthreads();
    if (!bad) {
      double *xB = a.gen + a.gs_xB[w];
      for (int b = tid; b < nB; b += nt) {
        xB[b] = lm[b];
        a.q[bd[b]] += lm[b];
      }
    }
  }
  if (go && nB > 0) {
    // the border block and the limbs' Schur sums, left zero for the next
    // round's assembly and atomics (the limb factors ran: go)
    for (int e = tid; e < nB * nB; e += nt) J[e] = 0.0;
    for (int b = tid; b < nB; b += nt) acc[b] = 0.0;
  }
  if (tid == 0) {
    int g = go;
    if (g && bad) {
      a.sys_status[s] = DM_ERR_DEGENERATE;
      a.sys_active[s] = 0;
      atomicAdd(&a.ctrl[1], 1);
      atomicMin(&a.ctrl[2], s);
      g = 0;
    }
    a.gen_go[w] = g;
    if (g) {
      a.sys_iters[s] += 1;
      if (a.ls_trial) a.ls_trial[s] = 1;
      atomicAdd(&a.ctrl[0], 1);
      if (a.units) {
        int nd = nB;
        for (int l = 0; l < a.gs_nlimb[w]; ++l) nd += a.lb_n[a.gs_limb0[w] + l];
        atomicAdd(a.units, (unsigned long long)nd);
      }
    }
  }
}

// Rows from the border end up: the row of step t is n - 1 - t (elimination
// order), pending in lane t mod 32; a step takes its x by a shuffle and
// subtracts its part from the next ten rows (record word d of a row d steps
// later; word 11 is zero).  The m condensed rows start from the border values.
// Each lane stages its own rows' records, two groups of 32 steps ahead.
__global__ void __launch_bounds__(128) k_gen_limb_back(SolveGenArgs a) {
  constexpr int kRing = 3;
  extern __shared__ double dyn[];
  const int wi = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int L = blockIdx.x * (blockDim.x >> 5) + wi;
  if (L >= a.nlimb) return;
  const int w = a.lb_gsys[L];
  if (!a.gs_fast[w] || !a.gen_go[w]) return;
  static_assert(gen_back_smem() == 32 * kRing * kLRec, "ring");
  double *ring = dyn + (size_t)wi * gen_back_smem() + lane * (kRing * kLRec);
  const int n = a.lb_n[L], m = a.lb_m[L], nbc = a.lb_nbc[L], dir = a.lb_dir[L];
  const int d0 = a.lb_dof0[L];
  const double *G = a.gen;
  const double *U = G + a.lb_y[L];
  auto fetch = [&](int g) {
    const int p = n - 1 - (32 * g + lane);
    double *dst = ring + kLRec * (g % kRing);
    if (p >= 0) {
#pragma unroll
      for (int e = 0; e < kLRec; e += 2) {
        const unsigned d = (unsigned)__cvta_generic_to_shared(dst + e);
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(U + (size_t)p * kLRec + e) : "memory");
      }
    } else {
#pragma unroll
      for (int e = 0; e < kLRec; ++e) dst[e] = 0.0;
    }
  };
#pragma unroll
  for (int g = 0; g < kRing; ++g) fetch(g);
  cp_async_commit();
  // the condensed rows n-1 .. n-m (steps 0 .. m - 1) from the border values:
  // the nbc values this limb couples to fetched one per lane, then broadcast
  double v;
  {
    const double *xB = G + a.gs_xB[w];
    const int32_t *bc = a.lb_bcols + a.lb_bc0[L];
    const double xbv = lane < nbc ? xB[bc[lane]] : 0.0;
    const double *Z = G + a.lb_Y[L] + (lane < m ? m - 1 - lane : 0) * (nbc + 1);
    v = lane < m ? Z[nbc] : 0.0;
#pragma unroll
    for (int b = 0; b < kFastMaxBC; ++b) {
      if (b >= nbc) break;  // uniform
      const double xb = __shfl_sync(kFull, xbv, b);
      if (lane < m) v = fma(-Z[b], xb, v);
    }
  }
  cp_async_wait_all();
  if (lane >= m) v = ring[0];
  int idx[32];
#pragma unroll
  for (int u = 0; u < 32; ++u) {
    const int d = (lane - u) & 31;
    idx[u] = d == 0 || d > 11 ? 11 : d;
  }
  const int groups = (n + 31) / 32;
  for (int g = 0; g < groups; ++g) {
    const double *ra = ring + kLRec * (g % kRing), *rb = ring + kLRec * ((g + 1) % kRing);
    const double zn = rb[0];
    double x_own = 0.0;
#pragma unroll
    for (int u = 0; u < 32; ++u) {
      const double x = __shfl_sync(kFull, v, u);
      if (lane == u) {
        x_own = x;
        v = zn;
      }
      v = fma(-(lane <= u ? rb : ra)[idx[u]], x, v);
    }
    const int p = n - 1 - (32 * g + lane);
    if (p >= 0) atomicAdd(a.q + d0 + (dir ? n - 1 - p : p), x_own);
    fetch(g + kRing);
    cp_async_commit();
    asm volatile("cp.async.wait_group 1;\n" ::: "memory");
  }
  cp_async_wait_all();
}

}  // namespace dm
