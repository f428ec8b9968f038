// Line Gauss-Seidel along z (Sec. 4.4, LGS): the points of a z-column (i, j)
// are updated together.  The column's right-hand side is its share of b minus
// the couplings to the columns earlier in the sweep (already new), and the
// tridiagonal system of the offsets (0,0,-1), (0,0,0), (0,0,+1) is solved
// exactly.  The couplings to later columns, old in a full sweep, are taken off
// b beforehand by a parallel kernel (k_line_half), so one sweep kernel serves
// both kinds.  Columns run in lexicographic (i, j) order (reversed for the
// backward sweep): one x-plane per CTA at a time (atomic ticket), column j of
// plane i after column j + 1 (or j) of plane i - 1.
//
// What bounds a column is a chain of dependent FP64 instructions (about 67
// cycles each): the last three coupling terms, the tridiagonal solve, the
// hand-over; at nz = 64 it takes 2800 cycles (waits 360, late terms and
// elimination 790, reduction 1150, recovery 300, stores 250), at nz = 128
// with two solving warps 3450, where one kernel with every term and every
// row's work on it took 10000.  A sweep at 128 x 112 x 128 on 27 points takes
// 0.90 ms (before: 2.03 from zero, 2.48 full).  So the work is split by what
// is on that chain:
//  * helper warps form the right-hand side up to the terms of the previous
//    column of the same plane, a column ahead;
//  * the solving warps (1, 2 or 4, one per SM sub-partition) add those terms
//    and solve.  A column is cut into 32 chunks per solving warp, of m rows,
//    one chunk per thread (partition method): every thread eliminates its rows
//    2..m in terms of its own first unknown P_c and the next chunk's P_{c+1},
//    the chunk-first unknowns form a tridiagonal system solved by parallel
//    cyclic reduction, and each thread then recovers its rows.  Chunk c belongs
//    to warp c mod warps, so all but the first reduction steps stay inside a
//    warp (shuffles); values that cross warps go through shared memory, one
//    barrier each.  Everything that depends only on the matrix is computed at
//    set-up, so a sweep does no division.  In exact arithmetic the result is
//    the Thomas solution; the rounding differs;
//  * a loader warp polls the previous plane's mailbox (mailbox.cuh) and keeps
//    its last columns in shared memory; a record warp fetches the columns'
//    coefficients and factors by bulk copies.
// Every wait is bounded; on expiry the error word is set, the CTA waits for
// its copies in flight and leaves.
#include <algorithm>
#include <climits>

#include "mailbox.cuh"
#include "smg_internal.cuh"

namespace {

using tri::ld_acq_cta;
using tri::st_rel_cta;

constexpr int kHelpers = 8;      // helper warps
constexpr int kMaxM = 8;         // rows per chunk: nz <= 1024
constexpr int kMaxStages = 4;    // columns of records in flight

// Solving warps and rows per chunk of a column of nz points.
__host__ __device__ inline int line_warps(int nz) { return nz <= 64 ? 1 : nz <= 128 ? 2 : 4; }
__host__ __device__ inline int line_rows(int nz) { return nz <= 256 ? 2 : nz <= 512 ? 4 : 8; }

// Column block of the line factors, in doubles, every field C = 32 * warps
// wide, chunk c at (c % warps) * 32 + c / warps: for chunk rows r = 1..m-1 the
// fields F_W (-a_r / den_r), F_INV (1 / den_r), F_CP (-c_r / den_r), F_G, F_H
// (x_r = e_r + g_r P_{c+1} + h_r P_c); then per chunk C_A0, C_C0 (minus the
// couplings of its first row), C_INVB (1 / final pivot), C_AL + t, C_GA + t
// (the multipliers of reduction step t, stride 2^t).
enum { F_W, F_INV, F_CP, F_G, F_H, F_N };
enum { C_A0, C_C0, C_INVB, C_STEP };
__host__ __device__ constexpr int row_field(int r, int f) { return (r - 1) * F_N + f; }
__host__ __device__ constexpr int chunk_field(int m, int f) { return (m - 1) * F_N + f; }
__host__ __device__ constexpr int step_field(int m, int t, int which) {
  return (m - 1) * F_N + C_STEP + 2 * t + which;
}
__host__ __device__ constexpr int log2_chunks(int warps) { return warps == 1 ? 5 : warps == 2 ? 6 : 7; }
__host__ __device__ constexpr int block_fields(int m, int warps) {
  return (m - 1) * F_N + C_STEP + 2 * log2_chunks(warps);
}

// Stencil entries of one direction of the sweep, in sweep coordinates: early
// ones (previous plane: column offset ec in {-1, 0, 1}) and late ones (the
// previous column of the same plane), each with its z offset; and the later
// columns' entries (natural offsets) of the half product.
struct LineTerms {
  int ne, nh, dep;  // dep: largest ec (-2 without early entries)
  int ee[9], ec[9], ez[9];
  int le[3];  // by z offset + 1; -1 where the mask lacks it
  int he[12], hx[12], hy[12], hz[12];
};

LineTerms line_terms(const Stencil& s, int dir) {
  LineTerms t{};
  t.dep = -2;
  t.le[0] = t.le[1] = t.le[2] = -1;
  for (int q = 0; q < s.ns; ++q) {
    const int e = dir > 0 ? q : s.ns - 1 - q;
    const int dx = dir * s.off[e][0], dy = dir * s.off[e][1], dz = s.off[e][2];
    if (dx == 0 && dy == 0) continue;
    if (dx < 0) {
      t.ee[t.ne] = e;
      t.ec[t.ne] = dy;
      t.ez[t.ne++] = dz;
      t.dep = std::max(t.dep, dy);
    } else if (dx == 0 && dy < 0) {
      t.le[dz + 1] = e;
    } else {
      t.he[t.nh] = e;
      t.hx[t.nh] = s.off[e][0];
      t.hy[t.nh] = s.off[e][1];
      t.hz[t.nh++] = dz;
    }
  }
  return t;
}

struct LineIdx {
  int sub, diag, sup;  // stencil entries of (0,0,-1), (0,0,0), (0,0,+1); -1 if absent
};

// Tridiagonal coefficients of row k of column col (identity beyond nz).
__device__ __forceinline__ void line_coef(const Grid& g, int ns, const LineIdx& e, const double* A, long long col,
                                          int k, double& a, double& b, double& c) {
  if (k >= g.nz) {
    a = 0.0;
    b = 1.0;
    c = 0.0;
    return;
  }
  const long long p = col * g.nz + k;
  a = (k > 0 && e.sub >= 0) ? A[p * ns + e.sub] : 0.0;
  b = A[p * ns + e.diag];
  c = (k + 1 < g.nz && e.sup >= 0) ? A[p * ns + e.sup] : 0.0;
}

// The oracle's breakdown rule: every Thomas pivot of every column positive.
__global__ void k_lgs_pivots(Grid g, int ns, LineIdx e, const double* __restrict__ A, int* err) {
  const long long col = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (col >= (long long)g.nx * g.ny) return;
  double cprev = 0.0;
  for (int k = 0; k < g.nz; ++k) {
    double a, b, c;
    line_coef(g, ns, e, A, col, k, a, b, c);
    const double piv = b - a * cprev;
    if (!(piv > 0.0)) {
      atomicCAS(err, 0, SMG_EBREAKDOWN);
      return;
    }
    cprev = c / piv;
  }
}

// One block per column, thread c = chunk c: the partitioned elimination of
// rows c*m + 1 .. c*m + m-1 and the reduced system's multipliers (neighbour
// values through shared memory).
__global__ void __launch_bounds__(128) k_lgs_factor(Grid g, int ns, LineIdx e, const double* __restrict__ A,
                                                    double* __restrict__ Fo, int m, int warps, int* err) {
  __shared__ double xa[128], xb[128], xc[128];
  const int C = 32 * warps, steps = log2_chunks(warps);
  const long long col = blockIdx.x;
  const int c = threadIdx.x;
  double* F = Fo + col * (long long)block_fields(m, warps) * C + (c % warps) * 32 + c / warps;
  double cp[kMaxM], fp[kMaxM];
  bool bad = false;
  for (int r = 1; r < m; ++r) {
    double a, b, cc;
    line_coef(g, ns, e, A, col, c * m + r, a, b, cc);
    const double den = r == 1 ? b : b - a * cp[r - 1];
    bad |= !(den > 0.0);
    const double inv = 1.0 / den;
    cp[r] = cc * inv;
    fp[r] = (r == 1 ? a : -a * fp[r - 1]) * inv;
    F[row_field(r, F_W) * C] = -a * inv;
    F[row_field(r, F_INV) * C] = inv;
    F[row_field(r, F_CP) * C] = -cp[r];
  }
  double gg = cp[m - 1], hh = fp[m - 1];
  const double glast = gg, hlast = hh;
  F[row_field(m - 1, F_G) * C] = -gg;
  F[row_field(m - 1, F_H) * C] = -hh;
  for (int r = m - 2; r >= 1; --r) {
    hh = fp[r] - cp[r] * hh;
    gg = -cp[r] * gg;
    F[row_field(r, F_G) * C] = -gg;
    F[row_field(r, F_H) * C] = -hh;
  }
  // reduced row of chunk c in P_{c-1}, P_c, P_{c+1}
  double a0, b0, c0;
  line_coef(g, ns, e, A, col, c * m, a0, b0, c0);
  xa[c] = glast;
  xb[c] = hlast;
  __syncthreads();
  const double gl = c > 0 ? xa[c - 1] : 0.0, hl = c > 0 ? xb[c - 1] : 0.0;
  double Ar = -a0 * hl;
  double Br = b0 - a0 * gl - c0 * hh;  // hh, gg now hold h_1, g_1
  double Cr = -c0 * gg;
  F[chunk_field(m, C_A0) * C] = -a0;
  F[chunk_field(m, C_C0) * C] = -c0;
  for (int t = 0; t < steps; ++t) {
    const int s = 1 << t;
    __syncthreads();
    xa[c] = Ar;
    xb[c] = Br;
    xc[c] = Cr;
    __syncthreads();
    const bool lo = c >= s, hi = c + s < C;
    const double Am = lo ? xa[c - s] : 0.0, Bm = lo ? xb[c - s] : 1.0, Cm = lo ? xc[c - s] : 0.0;
    const double Ap = hi ? xa[c + s] : 0.0, Bp = hi ? xb[c + s] : 1.0, Cp = hi ? xc[c + s] : 0.0;
    const double al = lo ? -Ar / Bm : 0.0, ga = hi ? -Cr / Bp : 0.0;
    const double nB = Br + al * Cm + ga * Ap;
    Ar = al * Am;
    Cr = ga * Cp;
    Br = nB;
    F[step_field(m, t, 0) * C] = al;
    F[step_field(m, t, 1) * C] = ga;
  }
  bad |= !(Br > 0.0);
  F[chunk_field(m, C_INVB) * C] = 1.0 / Br;
  if (bad) atomicCAS(err, 0, SMG_EBREAKDOWN);
}

// Line records: per column (natural index) the coefficients of the early and
// then the three late entries (zero where the mask lacks one), negated, each
// nzp (nz rounded up to even) wide.
__global__ void __launch_bounds__(256) k_line_records(Grid g, int ns, LineTerms T, int nzp,
                                                      const double* __restrict__ A, double* __restrict__ rec) {
  const long long p = (long long)blockIdx.x * 256 + threadIdx.x;
  if (p >= g.n) return;
  const long long col = p / g.nz;
  const int k = (int)(p % g.nz), n = T.ne + 3;
  double* r = rec + col * (long long)n * nzp + k;
  for (int q = 0; q < n; ++q) {
    const int e = q < T.ne ? T.ee[q] : T.le[q - T.ne];
    r[(long long)q * nzp] = e >= 0 ? -A[p * ns + e] : 0.0;
  }
}

// y = (couplings to later columns) x, or, with c, y = that and c = b - y.
__global__ void __launch_bounds__(256) k_line_half(Grid g, int ns, LineTerms T, const double* __restrict__ A,
                                                   const double* __restrict__ x, const double* __restrict__ b,
                                                   double* __restrict__ y, double* __restrict__ c) {
  const long long p = (long long)blockIdx.x * 256 + threadIdx.x;
  if (p >= g.n) return;
  const int k = (int)(p % g.nz), j = (int)((p / g.nz) % g.ny), i = (int)(p / ((long long)g.ny * g.nz));
  const double* a = A + p * ns;
  double acc = 0.0;
#pragma unroll 4
  for (int q = 0; q < T.nh; ++q) {
    const int a0 = i + T.hx[q], a1 = j + T.hy[q], a2 = k + T.hz[q];
    const bool in = (unsigned)a0 < (unsigned)g.nx && (unsigned)a1 < (unsigned)g.ny && (unsigned)a2 < (unsigned)g.nz;
    const double xv = in ? x[p + ((long long)T.hx[q] * g.ny + T.hy[q]) * g.nz + T.hz[q]] : 0.0;
    acc = fma(a[T.he[q]], xv, acc);
  }
  if (y) y[p] = acc;
  if (c) c[p] = b[p] - acc;
}

struct LsParams {
  Grid g;
  LineTerms T;
  int dir, nzp, log_stages, slots;  // record stages and columns of the previous plane kept (powers of two)
  unsigned long long budget_ns;
  const double *rec, *F, *b, *h;
  double *u, *emit;
  ulonglong2* mail;
  SweepWs* ws;
  int* err;
};

struct LineShared {
  unsigned long long full[kMaxStages];  // records landed
  unsigned long long rhs[2];            // right-hand side of a column formed (one arrival per active helper warp)
  int hready;                           // columns < hready of the previous plane are in the ring
  int done;                             // columns < done are solved
  int abort;
  int quit;                             // the solving warps leave in this column
  int plane;
};

// Shared memory, in doubles: ring of the previous plane's columns (a zero on
// either side), two right-hand sides, exchange rows, record stages.
__host__ __device__ inline long long line_ring(int nz, int slots) { return (long long)slots * (nz + 2) + (slots & 1); }
__host__ __device__ inline long long line_fixed(int nz, int C, int m, int slots) {
  return (line_ring(nz, slots) + 1) / 2 * 2 + 2LL * C * m + 6LL * C;
}
__host__ __device__ inline long long line_stage(int nzp, int terms, int m, int warps) {
  return (long long)nzp * terms + (long long)block_fields(m, warps) * 32 * warps;
}

// Spin until ok() or the CTA aborts; false on abort.
template <typename Ok>
__device__ __forceinline__ bool wait_for(LineShared& sh, Ok&& ok) {
  bool good = true;
  while (!ok())
    if (ld_acq_cta(&sh.abort)) {
      good = false;
      break;
    }
  return __all_sync(0xffffffffu, good);
}

template <int NWS, int M>
__global__ void __launch_bounds__((NWS + kHelpers + 2 + (NWS < 4 ? 2 - NWS : 0)) * 32, 1) k_lsweep(LsParams P) {
  constexpr int C = 32 * NWS, STEPS = log2_chunks(NWS);
  constexpr int FIELDS = block_fields(M, NWS);
  __shared__ LineShared sh;
  extern __shared__ __align__(128) double sm[];
  const Grid g = P.g;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nz = g.nz, terms = P.T.ne + 3;
  double* ring = sm;
  double* rhs = sm + (line_ring(nz, P.slots) + 1) / 2 * 2;  // two of C * M, row r of chunk c at r * C + position of c
  double* xch = rhs + 2 * C * M;                            // six rows of C
  double* stage0 = xch + 6 * C;
  const long long stage_len = line_stage(P.nzp, terms, M, NWS);
  // Warp roles, so that helpers share the sub-partitions (warp % 4) without a
  // solving warp where there are fewer than four: solvers first, then
  //   4 solvers: 8 helpers, loader, records;
  //   1 or 2:    (idle,) 2 helpers, loader, records, 6 helpers.
  int helper = -1;
  bool is_loader = false, is_record = false;
  if (NWS == 4) {
    if (warp >= 4 && warp < 12) helper = warp - 4;
    is_loader = warp == 12;
    is_record = warp == 13;
  } else {
    if (warp == 2 || warp == 3) helper = warp - 2;
    if (warp >= 6) helper = warp - 4;
    is_loader = warp == 4;
    is_record = warp == 5;
  }
  const int active = min(kHelpers, (nz + 31) / 32);  // helper warps with points
  const unsigned tag = (unsigned)P.ws->epoch + 1u;
  if (threadIdx.x == 0) {
    for (int t = 0; t < kMaxStages; ++t) tri::mbar_init(&sh.full[t], 1);
    tri::mbar_init(&sh.rhs[0], active);
    tri::mbar_init(&sh.rhs[1], active);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  const unsigned stages = 1u << P.log_stages;
  unsigned base = 0;  // columns of the planes before this one (every plane has ny)
  for (;;) {
    __syncthreads();
    if (threadIdx.x == 0) {
      sh.plane = atomicAdd(&P.ws->ticket, 1);
      sh.hready = 0;
      sh.done = 0;
      sh.abort = 0;
      sh.quit = INT_MAX;
    }
    for (int t = threadIdx.x; t < P.slots * (nz + 2); t += blockDim.x) ring[t] = 0.0;
    for (int t = threadIdx.x; t < 2 * C * M; t += blockDim.x) rhs[t] = 0.0;  // rows beyond nz stay zero
    __syncthreads();
    const int I = sh.plane;
    if (I >= g.nx) break;
    const int i = P.dir > 0 ? I : g.nx - 1 - I;
    auto column = [&](int J) { return (long long)i * g.ny + (P.dir > 0 ? J : g.ny - 1 - J); };
    auto stage = [&](int J) { return stage0 + (long long)((base + J) & (stages - 1)) * stage_len; };
    auto landed = [&](int J) {
      const unsigned f = base + J;
      return tri::mbar_test(&sh.full[f & (stages - 1)], (f >> P.log_stages) & 1u);
    };

    if (warp < NWS) {
      // ---- solving warps: chunk c = lane * NWS + warp
      const int c = lane * NWS + warp, pos = warp * 32 + lane;
      const int k0 = c * M;
      auto bar = [&]() {
        if (NWS > 1) asm volatile("bar.sync 2, %0;" ::"n"(C) : "memory");
        else __syncwarp();
      };
      // value of chunk c + d (0 beyond the ends), exchange row q
      auto position = [&](int cc) { return (cc % NWS) * 32 + cc / NWS; };
      auto from_low = [&](double v, int q) {  // chunk c - 1
        if (NWS == 1) {
          const double o = __shfl_up_sync(0xffffffffu, v, 1);
          return c > 0 ? o : 0.0;
        }
        xch[q * C + pos] = v;
        bar();
        return c > 0 ? xch[q * C + position(c - 1)] : 0.0;
      };
      auto from_high = [&](double v, int q) {  // chunk c + 1
        if (NWS == 1) {
          const double o = __shfl_down_sync(0xffffffffu, v, 1);
          return c + 1 < C ? o : 0.0;
        }
        xch[q * C + pos] = v;
        bar();
        return c + 1 < C ? xch[q * C + position(c + 1)] : 0.0;
      };
      double x[M], xlo = 0.0, xhi = 0.0;  // the previous column's rows, and the rows below and above them
#pragma unroll
      for (int r = 0; r < M; ++r) x[r] = 0.0;
      for (int J = 0; J < g.ny; ++J) {
        const long long col = column(J);
        double hv[M];
#pragma unroll
        for (int r = 0; r < M; ++r) hv[r] = (P.h && k0 + r < nz) ? P.h[col * nz + k0 + r] : 0.0;
        // Warp 0 waits for the right-hand side (which the helpers form once the
        // records are there), the others for warp 0.  If it gives up it says so
        // before the barrier, and every solving warp leaves at the end of this
        // column (whose work is then harmless).
        const double* rec = stage(J);
        const double* F = rec + P.nzp * terms + pos;
        const double* rr = rhs + ((base + J) & 1) * (C * M) + pos;
        if (warp == 0) {
          const bool ok =
              wait_for(sh, [&] { return tri::mbar_test(&sh.rhs[(base + J) & 1], ((base + J) >> 1) & 1u); });
          if (!ok && lane == 0) sh.quit = J;
          __syncwarp();
        }
        bar();
        double d[M], lc[3][M];
#pragma unroll
        for (int r = 0; r < M; ++r) d[r] = rr[r * C];
#pragma unroll
        for (int q = 0; q < 3; ++q)
#pragma unroll
          for (int r = 0; r < M; ++r) lc[q][r] = k0 + r < nz ? rec[(P.T.ne + q) * P.nzp + k0 + r] : 0.0;
        double al[STEPS], ga[STEPS];
#pragma unroll
        for (int t = 0; t < STEPS; ++t) {
          al[t] = F[step_field(M, t, 0) * C];
          ga[t] = F[step_field(M, t, 1) * C];
        }
        const double a0 = F[chunk_field(M, C_A0) * C], c0 = F[chunk_field(M, C_C0) * C];
        const double invb = F[chunk_field(M, C_INVB) * C];
        // the previous column's terms, rows 1.. first (their elimination follows)
        if (J > 0) {
#pragma unroll
          for (int rr2 = 1; rr2 <= M; ++rr2) {
            const int r = rr2 % M;
            if (P.T.le[0] >= 0) d[r] = fma(lc[0][r], r > 0 ? x[r > 0 ? r - 1 : 0] : xlo, d[r]);
            if (P.T.le[1] >= 0) d[r] = fma(lc[1][r], x[r], d[r]);
            if (P.T.le[2] >= 0) d[r] = fma(lc[2][r], r + 1 < M ? x[r + 1 < M ? r + 1 : r] : xhi, d[r]);
          }
        }
        double em[M];
#pragma unroll
        for (int r = 0; r < M; ++r) em[r] = d[r];
        // rows 1..M-1 in terms of P_c and P_{c+1}: d_r becomes e_r
#pragma unroll
        for (int r = 1; r < M; ++r) {
          const double iv = F[row_field(r, F_INV) * C];
          d[r] = r == 1 ? d[r] * iv : fma(F[row_field(r, F_W) * C], d[r - 1], d[r] * iv);
        }
#pragma unroll
        for (int r = M - 2; r >= 1; --r) d[r] = fma(F[row_field(r, F_CP) * C], d[r + 1], d[r]);
        const double elow = from_low(d[M - 1], 0);
        double D = fma(c0, d[1], fma(a0, elow, d[0]));
#pragma unroll
        for (int t = 0; t < STEPS; ++t) {
          const int s = 1 << t;
          double Dm, Dp;
          if (s < NWS) {  // the neighbours are in other warps
            const int q = 1 + t;
            xch[q * C + pos] = D;
            bar();
            Dm = c >= s ? xch[q * C + position(c >= s ? c - s : 0)] : 0.0;
            Dp = c + s < C ? xch[q * C + position(c + s < C ? c + s : 0)] : 0.0;
          } else {
            Dm = __shfl_up_sync(0xffffffffu, D, s / NWS);
            Dp = __shfl_down_sync(0xffffffffu, D, s / NWS);
            Dm = c >= s ? Dm : 0.0;
            Dp = c + s < C ? Dp : 0.0;
          }
          D = fma(al[t], Dm, fma(ga[t], Dp, D));
        }
        const double Pv = D * invb;
        const double Pn = from_high(Pv, 3);
        x[0] = Pv;
#pragma unroll
        for (int r = 1; r < M; ++r)
          x[r] = fma(F[row_field(r, F_G) * C], Pn, fma(F[row_field(r, F_H) * C], Pv, d[r]));
        ulonglong2* mb = P.mail + ((long long)I * g.ny + J) * nz;
#pragma unroll
        for (int r = 0; r < M; ++r)
          if (k0 + r < nz) tri::Mail<double>::put(mb + k0 + r, x[r], tag);
        xhi = Pn;
        xlo = from_low(x[M - 1], 4);
#pragma unroll
        for (int r = 0; r < M; ++r)
          if (k0 + r < nz) {
            P.u[col * nz + k0 + r] = x[r];
            if (P.emit) P.emit[col * nz + k0 + r] = em[r] + hv[r];
          }
        bar();  // every solving warp is past its reads of this column's records
        // no release: what the readers of done reuse has been read, not written
        if (threadIdx.x == 0) tri::st_relaxed_cta(&sh.done, J + 1);
        if (sh.quit <= J) break;
      }
    } else if (helper >= 0 && helper < active) {
      // ---- helper warps: the right-hand side but for the previous column's
      // terms, one point per thread (and 256 points further)
      for (int J = 0; J < g.ny; ++J) {
        const long long col = column(J);
        double bv[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int k = helper * 32 + lane + 256 * q;
          bv[q] = k < nz ? P.b[col * nz + k] : 0.0;
        }
        const int need = I == 0 || P.T.ne == 0 ? 0 : min(J + 1 + P.T.dep, g.ny);
        // Nothing else bounds a copy in flight (plane 0 has no loader), so once
        // the rest is there a copy that is due counts against the budget.
        unsigned long long t_wait = 0;
        const bool ok = wait_for(sh, [&] {
          if (ld_acq_cta(&sh.hready) < need || ld_acq_cta(&sh.done) < J - 1) return false;
          if (landed(J)) return true;
          if (ld_acq_cta(&sh.done) + (int)stages > J) {
            const unsigned long long now = globaltimer_ns();
            if (t_wait == 0) t_wait = now;
            else if (now - t_wait > P.budget_ns) {
              atomicCAS(P.err, 0, DEV_ERR_TIMEOUT);
              st_rel_cta(&sh.abort, 1);
            }
          }
          return false;
        });
        if (!ok) break;
        const double* rec = stage(J);
        double* out = rhs + ((base + J) & 1) * (C * M);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int k = helper * 32 + lane + 256 * q;
          if (256 * q >= C * M) break;
          if (k < C * M) {
            double acc = bv[q];
            if (k < nz && I > 0) {
#pragma unroll
              for (int e = 0; e < 9; ++e) {
                if (e >= P.T.ne) break;
                const int Jn = J + P.T.ec[e];
                if ((unsigned)Jn >= (unsigned)g.ny) continue;
                acc = fma(rec[(long long)e * P.nzp + k], ring[(Jn & (P.slots - 1)) * (nz + 2) + 1 + k + P.T.ez[e]], acc);
              }
            }
            const int cc = k / M;
            out[(k - cc * M) * C + (cc % NWS) * 32 + cc / NWS] = acc;
          }
        }
        __syncwarp();
        if (lane == 0)
          asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tri::smem_u32(&sh.rhs[(base + J) & 1])) : "memory");
      }
    } else if (is_loader) {
      // ---- loader warp: the previous plane's columns, in order
      unsigned long long t_wait = 0;
      unsigned iter = 0;
      bool stop = I == 0 || P.T.ne == 0;
      for (int J = 0; J < g.ny && !stop; ++J) {
        const ulonglong2* mb = P.mail + ((long long)(I - 1) * g.ny + J) * nz;
        double* dst = ring + (J & (P.slots - 1)) * (nz + 2) + 1;
        for (int kb = 0; kb < nz && !stop;) {
          // the slot's previous column is no longer read; up to four points a lane at once
          bool room = true;
          if (kb == 0) room = __shfl_sync(0xffffffffu, ld_acq_cta(&sh.done), 0) + P.slots - 2 >= J;
          bool all = room;
          if (room) {
            ulonglong2 v[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              const int k = kb + 32 * q + lane;
              v[q] = tri::Mail<double>::value(0.0, tag);
              if (k < nz) v[q] = tri::Mail<double>::get(mb + k);
            }
            bool ok = true;
#pragma unroll
            for (int q = 0; q < 4; ++q) ok = ok && tri::Mail<double>::ok(v[q], tag);
            all = __all_sync(0xffffffffu, ok);
            if (all) {
#pragma unroll
              for (int q = 0; q < 4; ++q) {
                const int k = kb + 32 * q + lane;
                if (k < nz) dst[k] = tri::Mail<double>::val(v[q]);
              }
              kb += 128;
              t_wait = 0;
            }
          }
          if (!all) {
            bool s = false;
            if (lane == 0) {
              if (room) {
                // bounded: the previous plane must make progress within the budget
                const unsigned long long now = globaltimer_ns();
                if (t_wait == 0) t_wait = now;
                else if (now - t_wait > P.budget_ns) {
                  atomicCAS(P.err, 0, DEV_ERR_TIMEOUT);
                  s = true;
                }
              }
              if ((++iter & 63u) == 0) s = s || ld_relaxed(P.err) != 0;
              s = s || ld_acq_cta(&sh.abort) != 0;
              if (s) st_rel_cta(&sh.abort, 1);
            }
            stop = __shfl_sync(0xffffffffu, s, 0);
            if (!room) __nanosleep(100);
          }
        }
        if (!stop) {
          __syncwarp();
          if (lane == 0) st_rel_cta(&sh.hready, J + 1);
        }
      }
    } else if (is_record && lane == 0) {
      // ---- record warp, one lane
      int issued = 0;
      bool stop = false;
      for (int J = 0; J < g.ny && !stop; ++J) {
        while (ld_acq_cta(&sh.done) + (int)stages <= J) {
          if (ld_acq_cta(&sh.abort)) {
            stop = true;
            break;
          }
          __nanosleep(20);
        }
        if (stop) break;
        const long long col = column(J);
        unsigned long long* bar = &sh.full[(base + J) & (stages - 1)];
        double* st = stage(J);
        const unsigned rb = (unsigned)(P.nzp * terms * sizeof(double)), fb = (unsigned)(FIELDS * C * sizeof(double));
        tri::mbar_expect_tx(bar, rb + fb);
        if (rb) tri::bulk_copy_g2s(st, P.rec + col * (long long)(P.nzp * terms), rb, bar);
        tri::bulk_copy_g2s(st + (long long)P.nzp * terms, P.F + col * (long long)(FIELDS * C), fb, bar);
        issued = J + 1;
      }
      // every copy has landed before the plane is left
      for (int J = max(0, issued - (int)stages); J < issued; ++J) {
        const unsigned long long t0 = globaltimer_ns();
        while (!landed(J))
          if (globaltimer_ns() - t0 > tri::kCopyWaitNs) break;
      }
    }
    base += (unsigned)g.ny;
    __syncthreads();
    if (sh.abort) break;
  }
  if (threadIdx.x == 0) {
    __threadfence();
    sh.plane = (atomicAdd(&P.ws->finished, 1) == (int)gridDim.x - 1);
  }
  __syncthreads();
  if (sh.plane && threadIdx.x == 0) {
    P.ws->ticket = 0;
    P.ws->epoch = (int)tag;
    __threadfence();
    P.ws->finished = 0;
  }
}

LineIdx line_idx(const Stencil& s) {
  LineIdx e{-1, -1, -1};
  for (int t = 0; t < s.ns; ++t) {
    if (s.off[t][0] != 0 || s.off[t][1] != 0) continue;
    if (s.off[t][2] == -1) e.sub = t;
    if (s.off[t][2] == 0) e.diag = t;
    if (s.off[t][2] == 1) e.sup = t;
  }
  return e;
}

constexpr long long kLineSmem = 216 * 1024;

template <int NWS, int M>
cudaError_t launch_line(LsParams P, int grid, cudaStream_t st) {
  const int terms = P.T.ne + 3;
  const long long per = line_stage(P.nzp, terms, M, NWS) * 8;
  P.slots = P.g.nz <= 512 ? 8 : 4;
  const long long fixed = line_fixed(P.g.nz, 32 * NWS, M, P.slots) * 8;
  const long long fit = (kLineSmem - fixed) / per;
  P.log_stages = fit >= kMaxStages ? 2 : fit >= 2 ? 1 : 0;
  const size_t smem = (size_t)(fixed + (per << P.log_stages));
  auto kern = k_lsweep<NWS, M>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  kern<<<grid, (NWS + kHelpers + 2 + (NWS < 4 ? 2 - NWS : 0)) * 32, smem, st>>>(P);
  return cudaGetLastError();
}

int padded(int nz) { return nz + (nz & 1); }

}  // namespace

long long lgs_block_doubles(int nz) {
  const int w = line_warps(nz);
  return (long long)block_fields(line_rows(nz), w) * 32 * w;
}

bool lgs_supported(const Grid& g, const Stencil& s) { return line_idx(s).diag >= 0 && g.nz <= 1024; }

long long lgs_record_doubles(const Grid& g, const Stencil& s, int dir) {
  const LineTerms T = line_terms(s, dir);
  return (long long)g.nx * g.ny * (T.ne + 3) * padded(g.nz);
}

cudaError_t launch_lgs_setup(const Grid& g, const Stencil& s, const double* A, double* F, double* recf, double* recb,
                             int* err, cudaStream_t st) {
  if (!lgs_supported(g, s)) return cudaErrorNotSupported;
  const LineIdx e = line_idx(s);
  const long long ncol = (long long)g.nx * g.ny;
  const int warps = line_warps(g.nz);
  k_lgs_pivots<<<div_up(ncol, 128), 128, 0, st>>>(g, s.ns, e, A, err);
  k_lgs_factor<<<(unsigned)ncol, 32 * warps, 0, st>>>(g, s.ns, e, A, F, line_rows(g.nz), warps, err);
  k_line_records<<<div_up(g.n, 256), 256, 0, st>>>(g, s.ns, line_terms(s, +1), padded(g.nz), A, recf);
  k_line_records<<<div_up(g.n, 256), 256, 0, st>>>(g, s.ns, line_terms(s, -1), padded(g.nz), A, recb);
  smg_count_launch(4);
  return cudaGetLastError();
}

cudaError_t launch_line_half(const Grid& g, const Stencil& s, int dir, const double* A, const double* x,
                             const double* b, double* y, double* c, cudaStream_t st) {
  k_line_half<<<div_up(g.n, 256), 256, 0, st>>>(g, s.ns, line_terms(s, dir), A, x, b, y, c);
  smg_count_launch(1);
  return cudaGetLastError();
}

cudaError_t launch_lsweep(const Grid& g, const Stencil& s, int dir, const double* rec, const double* F,
                          const double* b, const double* h, double* u, double* emit, void* mail, SweepWs* ws, int* err,
                          unsigned long long budget_ns, cudaStream_t st) {
  if (!lgs_supported(g, s)) return cudaErrorNotSupported;
  int dev = 0, nsm = 0;
  cudaError_t r = cudaGetDevice(&dev);
  if (r == cudaSuccess) r = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  if (r != cudaSuccess) return r;
  LsParams P;
  P.g = g;
  P.T = line_terms(s, dir);
  P.dir = dir;
  P.nzp = padded(g.nz);
  P.budget_ns = budget_ns;
  P.rec = rec;
  P.F = F;
  P.b = b;
  P.h = h;
  P.u = u;
  P.emit = emit;
  P.mail = (ulonglong2*)mail;
  P.ws = ws;
  P.err = err;
  const int grid = std::min(g.nx, nsm), warps = line_warps(g.nz), m = line_rows(g.nz);
  if (warps == 1) r = launch_line<1, 2>(P, grid, st);
  else if (warps == 2) r = launch_line<2, 2>(P, grid, st);
  else if (m == 2) r = launch_line<4, 2>(P, grid, st);
  else if (m == 4) r = launch_line<4, 4>(P, grid, st);
  else r = launch_line<4, 8>(P, grid, st);
  smg_count_launch(1);
  return r;
}
