// ILU(0) factorisation (Sec. 4.4 ILU formula, on the matrix mask of
// Sec. 4.2) for the canonical 7/19/27-point masks with one unknown per point,
// on the warp-pipelined wavefront of k_sweep3.cu.
//
// Row p of the factors depends on the finished rows of its lower
// neighbours, exactly like a forward triangular solve, so it runs on the same
// schedule t = SA*i + SB*j + k: one CTA per x-plane (taken by ticket), one
// lane per y-column, warps of 32 columns with their own time loops, a warp
// waits only for its left neighbour and for warps w-1..w+1 of the previous
// plane, and one publisher and one poller warp carry the per-warp progress
// between CTAs.  A step factors one row per lane:
//   for every lower entry k (in column order): l = a_pk / u_qq with q the
//   neighbour, then a_pj -= l * u_qj' for every later entry j of row p whose
//   offset difference o_j - o_k is an entry j' of row q (fill outside the
//   mask is dropped);  finally 1 / u_pp.
// The update pairs (j, j') of every k are derived at compile time from the
// mask, so the row lives in registers and every loop is unrolled.  Rows of
// the previous plane belong to another CTA and are read through L2.
//
// What bounds it: the chain of steps, of 123 FP64 instructions (64 cycles
// each) and the trips to L2 for the rows of twelve neighbours.  Those rows are
// loaded a chunk ahead of their use, without branches, so one chunk's trips
// overlap the work on the one before; the thirteenth, the step before of the
// same lane, stays in registers.  Set-up of a 256^3 hierarchy 108 to 88 ms, of
// a 7-point 160 x 96 x 224 one (27-point coarse levels) 28.6 to 23.1.
#include <algorithm>
#include <climits>
#include <utility>

#include "shapes.cuh"
#include "smg_internal.cuh"
#include "wavefront.cuh"

namespace {

template <int NS>
struct IluPairs {
  int kstart[NS + 1];
  int ej[128];
  int eq[128];
};

// For lower entry k (k < EC) the pairs kstart[k] .. kstart[k+1]-1 list every
// later entry j of the row with o_j - o_k in the mask (entry eq).
template <int NS>
__host__ __device__ constexpr IluPairs<NS> make_pairs() {
  using S = Shape<NS>;
  IluPairs<NS> t{};
  int n = 0;
  for (int ek = 0; ek < S::EC; ++ek) {
    t.kstart[ek] = n;
    for (int ej = ek + 1; ej < NS; ++ej) {
      int eq = -1;
      for (int e = 0; e < NS; ++e)
        if (S::o(e, 0) == S::o(ej, 0) - S::o(ek, 0) && S::o(e, 1) == S::o(ej, 1) - S::o(ek, 1) &&
            S::o(e, 2) == S::o(ej, 2) - S::o(ek, 2))
          eq = e;
      if (eq >= 0) {
        t.ej[n] = ej;
        t.eq[n] = eq;
        ++n;
      }
    }
  }
  for (int e = S::EC; e <= NS; ++e) t.kstart[e] = n;
  return t;
}

template <int NS>
struct IluTab {
  static constexpr IluPairs<NS> v = make_pairs<NS>();
};

// In-grid test of entry e for a point whose neighbour columns are described
// by xymask (bit (dx+1)*3 + dy+1) and whose z neighbours by zmask (bit dz+1).
template <int NS, int E>
__device__ __forceinline__ bool in_grid(unsigned xymask, unsigned zmask) {
  constexpr int ox = Shape<NS>::o(E, 0), oy = Shape<NS>::o(E, 1), oz = Shape<NS>::o(E, 2);
  return ((xymask >> ((ox + 1) * 3 + (oy + 1))) & 1u) && ((zmask >> (oz + 1)) & 1u);
}

// The lower entries are taken in chunks of three; what a chunk reads of its
// rows (1 / u_qq and the u_qj' of its pairs) is loaded while the chunk before
// is worked on.
constexpr int kChunk = 3;
template <int NS>
__host__ __device__ constexpr int chunk_pos(int ek) {  // place of entry ek's values in its chunk's buffer
  int n = 0;
  for (int e = ek / kChunk * kChunk; e < ek; ++e) n += 1 + IluTab<NS>::v.kstart[e + 1] - IluTab<NS>::v.kstart[e];
  return n;
}
template <int NS>
__host__ __device__ constexpr int chunk_size() {
  int m = 0;
  for (int e = 0; e < Shape<NS>::EC; ++e) {
    const int n = chunk_pos<NS>(e) + 1 + IluTab<NS>::v.kstart[e + 1] - IluTab<NS>::v.kstart[e];
    if (n > m) m = n;
  }
  return m;
}
template <int NS, int T>
constexpr int kEq = IluTab<NS>::v.eq[T];  // entry of the neighbour's row that pair T reads

template <int NS>
struct ChunkVals {
  double v[chunk_size<NS>()];
};

// The row of the point before in the own column (K - 1), from its centre on,
// and 1 / u_qq: the step before of the same lane, so it never leaves registers.
template <int NS>
struct PrevRow {
  double u[NS - Shape<NS>::EC], inv;
};

template <int NS>
struct RowArgs {
  long long p;
  const double *LU, *udinv;
  const int* lin;
  unsigned xymask, zmask;
};

// No branches on the grid's edge (a row's own place stands in for a neighbour
// that is not there): every load of a chunk is in flight at once.
template <int NS, int EK, int... Ts>
__device__ __forceinline__ void load_entry(ChunkVals<NS>& c, const RowArgs<NS>& a, const PrevRow<NS>& prev,
                                           std::integer_sequence<int, Ts...>) {
  constexpr int at = chunk_pos<NS>(EK), k0 = IluTab<NS>::v.kstart[EK];
  if constexpr (EK == Shape<NS>::EC - 1) {
    c.v[at] = prev.inv;
    ((c.v[at + 1 + Ts] = prev.u[kEq<NS, k0 + Ts> - Shape<NS>::EC]), ...);
    return;
  }
  const long long q = in_grid<NS, EK>(a.xymask, a.zmask) ? a.p + a.lin[EK] : a.p;
  const double* rowq = a.LU + q * NS;
  if constexpr (Shape<NS>::o(EK, 0) < 0) {  // the previous plane is another CTA's
    c.v[at] = __ldcg(a.udinv + q);
    ((c.v[at + 1 + Ts] = __ldcg(rowq + kEq<NS, k0 + Ts>)), ...);
  } else {
    c.v[at] = a.udinv[q];
    ((c.v[at + 1 + Ts] = rowq[kEq<NS, k0 + Ts>]), ...);
  }
}
template <int NS, int EK>
__device__ __forceinline__ void load_chunk(ChunkVals<NS>& c, const RowArgs<NS>& a, const PrevRow<NS>& prev) {
  if constexpr (EK < Shape<NS>::EC) {
    constexpr int n = IluTab<NS>::v.kstart[EK + 1] - IluTab<NS>::v.kstart[EK];
    load_entry<NS, EK>(c, a, prev, std::make_integer_sequence<int, n>{});
    if constexpr ((EK + 1) % kChunk != 0) load_chunk<NS, EK + 1>(c, a, prev);
  }
}

// a_pj -= l * u_qj' for pair T of the table, if both are on the grid
template <int NS, int T>
__device__ __forceinline__ void pair_update(double (&row)[NS], double l, double uv, bool in, const RowArgs<NS>& a) {
  constexpr int ej = IluTab<NS>::v.ej[T];
  const double v = fma(-l, uv, row[ej]);
  row[ej] = in && in_grid<NS, ej>(a.xymask, a.zmask) ? v : row[ej];
}
template <int NS, int EK, int... Ts>
__device__ __forceinline__ void pair_updates(double (&row)[NS], double l, bool in, const ChunkVals<NS>& c,
                                             const RowArgs<NS>& a, std::integer_sequence<int, Ts...>) {
  (pair_update<NS, IluTab<NS>::v.kstart[EK] + Ts>(row, l, c.v[chunk_pos<NS>(EK) + 1 + Ts], in, a), ...);
}

// Elimination of the chunk of lower entries from EK on: l = a_pk / u_qq, then its updates.
template <int NS, int EK>
__device__ __forceinline__ void eliminate(double (&row)[NS], const ChunkVals<NS>& c, const RowArgs<NS>& a) {
  if constexpr (EK < Shape<NS>::EC) {
    const bool in = in_grid<NS, EK>(a.xymask, a.zmask);
    const double l = row[EK] * c.v[chunk_pos<NS>(EK)];
    row[EK] = in ? l : row[EK];
    constexpr int n = IluTab<NS>::v.kstart[EK + 1] - IluTab<NS>::v.kstart[EK];
    pair_updates<NS, EK>(row, l, in, c, a, std::make_integer_sequence<int, n>{});
    if constexpr ((EK + 1) % kChunk != 0) eliminate<NS, EK + 1>(row, c, a);
  }
}
template <int NS, int EK>
__device__ __forceinline__ void factor_row(double (&row)[NS], const ChunkVals<NS>& cur, const RowArgs<NS>& a,
                                           const PrevRow<NS>& prev) {
  if constexpr (EK + kChunk < Shape<NS>::EC) {
    ChunkVals<NS> next;
    load_chunk<NS, EK + kChunk>(next, a, prev);
    eliminate<NS, EK>(row, cur, a);
    factor_row<NS, EK + kChunk>(row, next, a, prev);
  } else {
    eliminate<NS, EK>(row, cur, a);
  }
}

struct Ilu3Params {
  Grid g;
  WfCtl C;
  double* LU;     // in: A, out: factors (same layout)
  double* udinv;  // out: 1 / u_pp
  int lin[27];
};

// MW: most compute warps per plane the registers are cut for.
template <int NS, int MW>
__global__ void __launch_bounds__((MW + 2) * 32, 1) k_ilu3(Ilu3Params P) {
  using S = Shape<NS>;
  constexpr int SA = S::SA, SB = S::SB, EC = S::EC;
  __shared__ WfShared sh;
  const Grid g = P.g;
  wf_run(sh, P.C, [&](int I) {
    // compute warp w: columns 32w .. 32w+31 of plane I
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int i = I, j = 32 * w + lane;
    const bool colok = j < g.ny;
    const int jlast = min(32 * w + 31, g.ny - 1);
    const int s_begin = SB * 32 * w, s_end = SB * jlast + g.nz - 1;
    const int gt0 = SA * I;
    // in-grid mask of the (dx, dy) neighbour columns of this column
    unsigned xymask = 0;
#pragma unroll
    for (int a = -1; a <= 1; ++a)
#pragma unroll
      for (int c = -1; c <= 1; ++c)
        if ((unsigned)(i + a) < (unsigned)g.nx && (unsigned)(j + c) < (unsigned)g.ny)
          xymask |= 1u << ((a + 1) * 3 + (c + 1));
    const long long colbase = ((long long)i * g.ny + j) * g.nz;
    PrevRow<NS> prev = {};
    int have_left = (w == 0) ? kWfDone : INT_MIN, have_up = INT_MIN;
    for (int s = s_begin; s <= s_end; ++s) {
      // the rows of the previous plane this row reads end at local step s + SA - 1
      if (wf_wait(sh, P.C, w, s, gt0 + s, have_left, have_up, lane)) break;
      const int k = s - SB * j;
      if (colok && k >= 0 && k < g.nz) {
        const long long p = colbase + k;
        const unsigned zmask = (k > 0 ? 1u : 0u) | 2u | (k + 1 < g.nz ? 4u : 0u);
        double row[NS];
        const double* src = P.LU + p * NS;
#pragma unroll
        for (int e = 0; e < NS; ++e) row[e] = src[e];
        const RowArgs<NS> args{p, P.LU, P.udinv, P.lin, xymask, zmask};
        ChunkVals<NS> first;
        load_chunk<NS, 0>(first, args, prev);
        factor_row<NS, 0>(row, first, args, prev);
        const double piv = row[EC];
        if (!(piv > 0.0)) atomicCAS(P.C.err, 0, SMG_EBREAKDOWN);
        double* dst = P.LU + p * NS;
#pragma unroll
        for (int e = 0; e < NS; ++e) dst[e] = row[e];
        prev.inv = 1.0 / piv;
        P.udinv[p] = prev.inv;
#pragma unroll
        for (int e = EC; e < NS; ++e) prev.u[e - EC] = row[e];
      }
      wf_done(sh, w, s + 1, lane);  // row stored
    }
    if (lane == 0) wf_st_rel_cta(&sh.wdone[w], kWfDone);
  });
}

template <int NS>
bool canonical_mask(const Stencil& s) {
  if (s.ns != NS) return false;
  for (int e = 0; e < NS; ++e)
    for (int d = 0; d < 3; ++d)
      if (s.off[e][d] != Shape<NS>::o(e, d)) return false;
  return true;
}

}  // namespace

cudaError_t launch_ilu_factor3(Grid g, const Stencil& s, double* LU, double* udinv, SweepWs* ws, int* err,
                               unsigned long long budget_ns, cudaStream_t st) {
  int grid = 0, nthr = 0;
  cudaError_t e = wf_launch_shape(g, &grid, &nthr);
  if (e != cudaSuccess) return e;
  Ilu3Params P;
  P.g = g;
  P.LU = LU;
  P.udinv = udinv;
  for (int t = 0; t < 27; ++t) P.lin[t] = s.lin[t];
  auto go = [&](auto kern, int SA, int SB) {
    P.C = WfCtl{g.nx, (g.ny + 31) / 32, SA, SB, budget_ns, ws, err};
    cudaError_t a = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kWfOneCtaPerSmSmem);
    if (a != cudaSuccess) return a;
    kern<<<grid, nthr, kWfOneCtaPerSmSmem, st>>>(P);
    return cudaGetLastError();
  };
  const int NW = (g.ny + 31) / 32;
#define GO_(NS) \
  e = NW <= 4   ? go(k_ilu3<NS, 4>, Shape<NS>::SA, Shape<NS>::SB) \
      : NW <= 8 ? go(k_ilu3<NS, 8>, Shape<NS>::SA, Shape<NS>::SB) \
                : go(k_ilu3<NS, kWfMaxWarps>, Shape<NS>::SA, Shape<NS>::SB)
  if (canonical_mask<27>(s)) GO_(27);
  else if (canonical_mask<19>(s)) GO_(19);
  else if (canonical_mask<7>(s)) GO_(7);
  else return cudaErrorNotSupported;
#undef GO_
  smg_count_launch(1);
  return e;
}
