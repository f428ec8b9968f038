// Warp-pipelined wavefront sweeps (exact lexicographic order) on matrices and
// vectors in natural order, FP64, for the 7/19/27-point masks with one unknown
// per point: Gauss-Seidel (zero-guess and full, both directions) and the two
// ILU(0) triangular solves (Sec. 4.4).  They run the entry point that has no
// hierarchy to keep records in (smg_sweep_noalloc) and the level operations
// of levels without them; hierarchies run the sheared wavefront (tri.cuh),
// which forms its sums in the same order.
//
// Schedule: point (i,j,k) runs at global time t = SA*i + SB*j + k (the
// smallest skews that put every lower neighbour strictly earlier).
//  * A CTA owns one x-plane at a time (handed out by an atomic ticket, so a
//    CTA only ever waits on planes that running CTAs own).  The plane is cut
//    into warps of 32 y-columns, one lane per column, and every warp runs its
//    own loop over local steps s = t - SA*plane; lane J treats point
//    K = s - SB*J of its column at step s.
//  * A neighbour of the lower triangle is older than its point by a fixed
//    number of steps, its slack (SA*dx' + SB*dy' + dz' in sweep coordinates).
//    Previous-plane values are loaded one by one, as late as their slack
//    allows: a term of slack sigma is loaded min(2, sigma - 1) steps before
//    its point is finished.
//  * Inside a step: wait for the three counters it depends on (left warp,
//    right warp for the shared value ring, previous plane), issue the loads
//    whose slack is one step, pre-sum point K+1 (every term that is already
//    final), finish point K (own column, left column, the late
//    previous-plane terms), store it, publish the step, then load the
//    operands of K+1 and K+2.
//  * Order of a point's sum: b, the old values (Gauss-Seidel), the early
//    terms, the late ones, each group in sweep order (the stencil entries
//    mirrored for a backward sweep).
//  * Counters are per warp in shared memory (CTA-scope acquire/release); one
//    publisher warp copies the plane's counters to global memory (GPU-scope
//    release) and one poller warp copies the previous CTA's into shared
//    memory (GPU-scope acquire), so compute warps never execute a GPU-scope
//    fence.  One CTA per SM (the launch reserves more than half of the shared
//    memory) and the grid is capped at the SM count.
// Every wait is bounded; on expiry the error word is set and all CTAs drain.
#include <algorithm>
#include <climits>

#include "shapes.cuh"
#include "smg_internal.cuh"

namespace {

// Term classes, relative to the sweep direction.
enum { T_SKIP = 0, T_OWN = 1, T_Y = 2, T_X = 3, T_OLD = 4 };

template <int NS, int KIND, int DIR>
__host__ __device__ constexpr int cls(int e) {
  using S = Shape<NS>;
  const int sx = DIR * S::o(e, 0), sy = DIR * S::o(e, 1), sz = DIR * S::o(e, 2);
  if (e == S::EC) return T_SKIP;
  const bool is_new = sx < 0 || (sx == 0 && (sy < 0 || (sy == 0 && sz < 0)));
  if (!is_new) return KIND == SW_GS_FULL ? T_OLD : T_SKIP;
  if (sx == 0 && sy == 0) return T_OWN;  // (0, 0, -1)
  if (sx == 0) return T_Y;               // (0, -1, *): the left column
  return T_X;                            // (-1, *, *): the previous plane
}

// Steps between a new neighbour and its point.
template <int NS, int DIR>
__host__ __device__ constexpr int slack(int e) {
  using S = Shape<NS>;
  return -(S::SA * DIR * S::o(e, 0) + S::SB * DIR * S::o(e, 1) + DIR * S::o(e, 2));
}

// When an operand is consumed: in the pre-sum of K+1 (loaded two steps
// ahead), or in the finish of K (loaded one step ahead, or in the step).
enum { U_NONE = 0, U_PRE = 1, U_FIN1 = 2, U_FIN0 = 3, U_FINR = 4 };

template <int NS, int KIND, int DIR>
__host__ __device__ constexpr int use(int e) {
  const int c = cls<NS, KIND, DIR>(e);
  if (c == T_SKIP) return U_NONE;
  if (c == T_OLD) return U_PRE;
  if (c == T_OWN) return U_FINR;
  const int sg = slack<NS, DIR>(e);
  if (c == T_Y) return sg >= 2 ? U_PRE : U_FINR;  // left column, from the shared ring
  const int m = sg - 1 < 2 ? sg - 1 : 2;          // previous plane
  return m == 2 ? U_PRE : (m == 1 ? U_FIN1 : U_FIN0);
}

// Stencil entry of position t in sweep order.
template <int NS, int DIR>
__host__ __device__ constexpr int entry(int t) {
  return DIR > 0 ? t : NS - 1 - t;
}

struct Sweep3Params {
  Grid g;
  unsigned long long budget_ns;
  const double* M;     // GS: matrix [n][NS]; ILU: the factors [n][NS]
  const double* dinv;  // GS: inverse diagonal; ILU_U: 1/u_pp
  double w;
  const double* b;  // may alias u
  double* u;
  SweepWs* ws;  // prog[] indexed by plane and warp
  int* err;
};

constexpr int kMaxWarpsPerPlane = 16;
constexpr int kPrefetch = 10;
constexpr int kDone = INT_MAX / 2;
constexpr size_t kOneCtaPerSmSmem = 120 * 1024;
constexpr unsigned kPublishGapNs = 100;
// Shared ring of the last kRing values of every column.  A column's value
// at point k is overwritten by point k + kRing.  A warp publishes step s
// once point k is stored, before it reads the ring for point k+1, so its
// left-hand neighbour may run at most kRing - SB - 2 steps ahead of the
// published step without overwriting a value still to be read.
constexpr int kRing = 16;

__device__ __forceinline__ int ld_acq_cta(const int* p) {
  int v;
  asm volatile("ld.acquire.cta.shared.s32 %0, [%1];" : "=r"(v) : "r"((unsigned)__cvta_generic_to_shared(p)) : "memory");
  return v;
}
__device__ __forceinline__ void st_rel_cta(int* p, int v) {
  asm volatile("st.release.cta.shared.s32 [%0], %1;" ::"r"((unsigned)__cvta_generic_to_shared(p)), "r"(v) : "memory");
}
__device__ __forceinline__ void prefetch_l2(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

struct Shared3 {
  int wdone[kMaxWarpsPerPlane];  // per compute warp: all local steps < value are finished
  int avail[kMaxWarpsPerPlane];  // previous CTA's plane, per warp: global time finished
  int abort;
  int group;
};

// Publisher warp: lane w publishes the progress of warp w of the CTA's last
// plane (wd: that plane's counters, local steps) as global time gt0 + T with
// a GPU-scope release store whenever it grows.
__device__ __forceinline__ void publisher_warp(Shared3& sh, const int* wd, const Sweep3Params& P, int I, int NW, int gt0,
                                               int lane) {
  const bool mine = lane < NW;
  int* out_slot = P.ws->prog + (size_t)I * NW + lane;
  int published = INT_MIN;
  for (;;) {
    const int T = mine ? ld_acq_cta(&wd[lane]) : kDone;
    if (__any_sync(0xffffffffu, mine && T != published)) {
      // one release (one GPU-scope fence) covers every lane's value; a
      // fence also stalls the SM's other memory traffic, so they are
      // spaced by a fraction of a step
      if (mine) st_release(out_slot, T >= kDone ? kDone : gt0 + T);
      published = T;
      if (__all_sync(0xffffffffu, T >= kDone)) break;
      __nanosleep(kPublishGapNs);
    } else {
      __nanosleep(32);
    }
    if (__any_sync(0xffffffffu, ld_acq_cta(&sh.abort) != 0)) {
      // release everything downstream; the error word is already set
      if (mine) st_release(out_slot, kDone);
      break;
    }
  }
}

// Poller warp: lane w forwards the progress of warp w of the previous CTA's
// last plane into sh.avail (GPU-scope acquire loads).  Bounded: the previous
// CTA must make progress within the budget, else the error word and the
// CTA's abort flag are set.
__device__ __forceinline__ void poller_warp(Shared3& sh, const Sweep3Params& P, int I, int NW, int lane) {
  const bool mine = lane < NW;
  const int* in_slot = P.ws->prog + (size_t)(I - 1) * NW + lane;
  int seen = (I == 0 || !mine) ? kDone : 0;
  unsigned long long t_wait = 0;
  unsigned iter = 0;
  while (__any_sync(0xffffffffu, seen < kDone)) {
    int v = seen;
    if (seen < kDone) asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(in_slot) : "memory");
    const bool fresh = v > seen;
    bool stop = false;
    if (__any_sync(0xffffffffu, fresh)) {
      if (fresh) {
        seen = v;
        st_rel_cta(&sh.avail[lane], v);
      }
      t_wait = 0;
    } else if (lane == 0) {
      const unsigned long long now = globaltimer_ns();
      if (t_wait == 0) t_wait = now;
      else if (now - t_wait > P.budget_ns) {
        atomicCAS(P.err, 0, DEV_ERR_TIMEOUT);
        stop = true;
      }
    }
    if ((++iter & 63u) == 0 && lane == 0) stop = stop || ld_relaxed(P.err) != 0 || ld_acq_cta(&sh.abort) != 0;
    if (__shfl_sync(0xffffffffu, stop, 0)) {
      if (lane == 0) st_rel_cta(&sh.abort, 1);
      break;
    }
  }
}

// The sweeps hold their operands in register pairs: they get at most 12
// compute warps (ny <= 384) and the registers that leaves, 8 (ny <= 256)
// when they use every stencil entry.
template <int KIND>
__host__ __device__ constexpr int max_threads() {
  return KIND == SW_GS_FULL ? 320 : 448;
}

template <int NS, int KIND, int DIR>
__global__ void __launch_bounds__(max_threads<KIND>(), 1) k_sweep3(Sweep3Params P) {
  using S = Shape<NS>;
  constexpr int SA = S::SA, SB = S::SB;
  constexpr bool NEED_D = KIND != SW_ILU_L;
  extern __shared__ __align__(16) double hist[];  // value ring [k % kRing][column]
  __shared__ Shared3 sh;

  const Grid g = P.g;
  const int NW = (g.ny + 31) >> 5;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  constexpr int LEAD = kRing - SB - 2;  // largest lead over the right-hand warp
  for (int t = threadIdx.x; t < kRing * NW * 32; t += blockDim.x) hist[t] = 0.0;

  for (;;) {
    __syncthreads();
    if (threadIdx.x == 0) {
      sh.group = atomicAdd(&P.ws->ticket, 1);
      sh.abort = 0;
    }
    __syncthreads();
    const int I = sh.group;
    if (I >= g.nx) break;
    if (threadIdx.x < kMaxWarpsPerPlane) {
      // a warp has trivially finished every step before its first one;
      // nothing precedes the first plane; 0 is below every time a later
      // plane asks for
      sh.wdone[threadIdx.x] = (int)threadIdx.x < NW ? SB * 32 * (int)threadIdx.x - 2 : kDone;
      sh.avail[threadIdx.x] = (I == 0) ? kDone : 0;
    }
    __syncthreads();

    if (warp == NW) {
      publisher_warp(sh, sh.wdone, P, I, NW, SA * I, lane);
    } else if (warp == NW + 1) {
      poller_warp(sh, P, I, NW, lane);
    } else if (warp < NW) {
      const int w = warp;
      const double* b = P.b;
      double* u = P.u;
      const double* __restrict__ dinv = P.dinv;
      const bool relax = P.w != 1.0;
      const double wv = P.w;
      const int i = DIR > 0 ? I : g.nx - 1 - I;
      const int J = 32 * w + lane;
      const bool colok = J < g.ny;
      const int j = DIR > 0 ? J : g.ny - 1 - J;
      const int jlast = min(32 * w + 31, g.ny - 1);
      const int s_begin = SB * 32 * w - 2;
      const int s_end = SB * jlast + g.nz - 1;
      const int gt0 = SA * I;
      int have_left = (w == 0) ? kDone : INT_MIN;        // cached progress of the left warp
      int have_right = (w + 1 == NW) ? kDone : INT_MIN;  // cached progress of the right warp
      int have_up = INT_MIN;                             // cached progress of the previous plane
      auto index = [&](int dx, int dy, int kk) -> long long {
        return ((long long)(i + dx) * g.ny + (j + dy)) * g.nz + kk;
      };

      // stage 2: operands of point K+2, loaded at step s, pre-summed at s+1
      double c2[NS], x2[NS];
      double b2 = 0.0, d2 = 0.0, uo2 = 0.0;
      // finish operands of point K (pre-summed at s-1) and of point K+1
      double cfK[NS], cfN[NS];
      double accK = 0.0, dK = 0.0, uoK = 0.0;
      double x1[NS];  // previous-plane terms of point K loaded one step ahead
      double carry = 0.0;
#pragma unroll
      for (int e = 0; e < NS; ++e) c2[e] = cfK[e] = cfN[e] = x2[e] = x1[e] = 0.0;

      // value of neighbour e of the point with grid index kk.  The load is
      // issued unconditionally: a neighbour off the grid has a coefficient of
      // exactly zero (zero padding), so it reads the point's own right-hand
      // side instead (finite, in bounds) and the term adds zero -- no select
      // has to wait for the load.
      auto nb = [&](int e, int kk) -> double {
        const int ox = S::o(e, 0), oy = S::o(e, 1), oz = S::o(e, 2);
        const bool in = (unsigned)(i + ox) < (unsigned)g.nx && (unsigned)(j + oy) < (unsigned)g.ny &&
                        (unsigned)(kk + oz) < (unsigned)g.nz;
        const double* q = in ? u + index(ox, oy, kk + oz) : b + index(0, 0, kk);
        // the previous schedule plane of another CTA: read through L2;
        // everything else through L1
        return DIR * ox < 0 ? __ldcg(q) : *q;
      };
      // value of the left column's point kk from the shared ring; the ring
      // starts zeroed, so a slot read off the grid (coefficient zero) is finite
      auto ring = [&](int kk) -> double { return hist[(kk & (kRing - 1)) * (NW * 32) + (J > 0 ? J - 1 : 0)]; };

      bool aborted = false;
      for (int s = s_begin; s <= s_end; ++s) {
        // -- dependencies, against counters cached in registers.  Every lane
        // checks them (the same values in all lanes, so the warp does not
        // diverge); only when the cache is stale do the lanes poll the shared
        // counters, each with its own acquire load (one broadcast).  The
        // previous plane's points this warp reads lie in columns
        // 32w-1 .. 32w+32: warps w-1..w+1, SA steps ahead.
        const int need = gt0 + s;
        if (__any_sync(0xffffffffu, have_left < s || have_right < s - LEAD || have_up < need)) {
          unsigned long long t_start = 0;
          for (;;) {
            if (have_left < s) have_left = ld_acq_cta(&sh.wdone[w - 1]);
            if (have_right < s - LEAD) have_right = ld_acq_cta(&sh.wdone[w + 1]);
            if (have_up < need) {
              int T = kDone;
              for (int ww = max(w - 1, 0); ww <= min(w + 1, NW - 1); ++ww) T = min(T, ld_acq_cta(&sh.avail[ww]));
              have_up = T;
            }
            if (have_left >= s && have_right >= s - LEAD && have_up >= need) break;
            if (ld_acq_cta(&sh.abort)) { aborted = true; break; }
            const unsigned long long now = globaltimer_ns();
            if (t_start == 0) t_start = now;
            else if (now - t_start > P.budget_ns) {
              if (lane == 0) {
                atomicCAS(P.err, 0, DEV_ERR_TIMEOUT);
                st_rel_cta(&sh.abort, 1);
              }
              aborted = true;
              break;
            }
          }
          // lanes leave the loop together unless one gave up: agree
          aborted = __any_sync(0xffffffffu, aborted);
          if (aborted) break;
        }
        const int K = s - SB * J;
        const bool okK = colok && K >= 0 && K < g.nz;
        const bool okK1 = colok && K + 1 >= 0 && K + 1 < g.nz;
        const int kK = DIR > 0 ? K : g.nz - 1 - K;

        // (a) previous-plane terms of K whose slack is one step: loaded now
        double x0[NS];
#pragma unroll
        for (int e = 0; e < NS; ++e) {
          x0[e] = 0.0;
          if (use<NS, KIND, DIR>(e) == U_FIN0 && okK) x0[e] = nb(e, kK);
        }

        // (b) pre-sum of point K+1: the old values, then every new term that
        // is final by now
        double accN = 0.0, dN = 0.0, uoN = 0.0;
        if (okK1) {
          double a = b2;
#pragma unroll
          for (int pass = 0; pass < 2; ++pass)
#pragma unroll
            for (int t = 0; t < NS; ++t) {
              const int e = entry<NS, DIR>(t);
              if (use<NS, KIND, DIR>(e) != U_PRE || (cls<NS, KIND, DIR>(e) == T_OLD) != (pass == 0)) continue;
              const double tv = cls<NS, KIND, DIR>(e) == T_Y ? ring(K + 1 + DIR * S::o(e, 2)) : x2[e];
              a = fma(-c2[e], tv, a);
            }
          accN = a;
          dN = d2;
          uoN = uo2;
        }
#pragma unroll
        for (int e = 0; e < NS; ++e) {
          const int us = use<NS, KIND, DIR>(e);
          if (us == U_FIN0 || us == U_FIN1 || us == U_FINR) cfN[e] = c2[e];
        }

        // (c) finish point K
        if (okK) {
          double a = accK;
#pragma unroll
          for (int t = 0; t < NS; ++t) {
            const int e = entry<NS, DIR>(t);
            const int us = use<NS, KIND, DIR>(e);
            if (us != U_FIN0 && us != U_FIN1 && us != U_FINR) continue;
            double tv;
            if (cls<NS, KIND, DIR>(e) == T_OWN) tv = carry;
            else if (cls<NS, KIND, DIR>(e) == T_Y) tv = ring(K + DIR * S::o(e, 2));
            else tv = us == U_FIN0 ? x0[e] : x1[e];
            a = fma(-cfK[e], tv, a);
          }
          double r = a;
          if (KIND != SW_ILU_L) {
            r = a * dK;
            if (KIND != SW_ILU_U && relax)
              r = (KIND == SW_GS_ZERO) ? wv * r : fma(wv, r, __dmul_rn(1.0 - wv, uoK));
          }
          u[index(0, 0, kK)] = r;
          hist[(K & (kRing - 1)) * (NW * 32) + J] = r;
          carry = r;
        }
        // -- point K is stored: publish step s before the loads below are
        // issued, so the release does not wait for them
        __syncwarp();
        if (lane == 0) st_rel_cta(&sh.wdone[w], s + 1);
        accK = accN;
        dK = dN;
        uoK = uoN;
#pragma unroll
        for (int e = 0; e < NS; ++e) cfK[e] = cfN[e];

        // (d) previous-plane terms of K+1 whose slack allows one step
        if (okK1) {
          const int k1 = DIR > 0 ? K + 1 : g.nz - 2 - K;
#pragma unroll
          for (int e = 0; e < NS; ++e)
            if (use<NS, KIND, DIR>(e) == U_FIN1) x1[e] = nb(e, k1);
        }

        // (e) operands of point K+2
        const int K2 = K + 2;
        if (colok && K2 >= 0 && K2 < g.nz) {
          const int k2 = DIR > 0 ? K2 : g.nz - 1 - K2;
          const long long p2 = index(0, 0, k2);
          const double* __restrict__ a = P.M + p2 * NS;
#pragma unroll
          for (int e = 0; e < NS; ++e)
            if (use<NS, KIND, DIR>(e) != U_NONE) c2[e] = a[e];
          if (NEED_D) d2 = dinv[p2];
          if (K2 + kPrefetch < g.nz) {
            const char* pf = (const char*)(P.M + (p2 + DIR * kPrefetch) * NS);
            prefetch_l2(pf);
            prefetch_l2(pf + NS * sizeof(double) - 1);
          }
#pragma unroll
          for (int e = 0; e < NS; ++e)
            if (use<NS, KIND, DIR>(e) == U_PRE && cls<NS, KIND, DIR>(e) != T_Y) x2[e] = nb(e, k2);
          b2 = b[p2];
          if (KIND == SW_GS_FULL && relax) uo2 = u[p2];
        }
      }
      if (lane == 0) st_rel_cta(&sh.wdone[w], kDone);
    }
  }
  if (threadIdx.x == 0) {
    __threadfence();
    sh.group = (atomicAdd(&P.ws->finished, 1) == (int)gridDim.x - 1);
  }
  __syncthreads();
  if (sh.group) {
    for (int q = threadIdx.x; q < g.nx * NW; q += blockDim.x) P.ws->prog[q] = 0;
    __syncthreads();
    if (threadIdx.x == 0) {
      P.ws->ticket = 0;
      __threadfence();
      P.ws->finished = 0;
    }
  }
}

template <int NS>
bool canonical(const Stencil& s) {
  if (s.ns != NS) return false;
  for (int e = 0; e < NS; ++e)
    for (int d = 0; d < 3; ++d)
      if (s.off[e][d] != Shape<NS>::o(e, d)) return false;
  return true;
}

template <int NS>
cudaError_t launch_kind(int kind, int dir, const Sweep3Params& P, cudaStream_t st) {
  const int NW = (P.g.ny + 31) / 32;
  const int nthr = (NW + 2) * 32;
  // the value ring needs at most 48 KB; reserving more than half of the SM's
  // 228 KB keeps a second CTA off the SM
  const size_t smem = std::max(sizeof(double) * (size_t)kRing * NW * 32, kOneCtaPerSmSmem);
  int dev = 0, nsm = 0;
  cudaError_t ae = cudaGetDevice(&dev);
  if (ae == cudaSuccess) ae = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  if (ae != cudaSuccess) return ae;
  const int grid = std::min(P.g.nx, nsm);
  auto go = [&](auto kern) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    kern<<<grid, nthr, smem, st>>>(P);
    return cudaGetLastError();
  };
  if (kind == SW_GS_ZERO) return go(k_sweep3<NS, SW_GS_ZERO, 1>);
  if (kind == SW_GS_FULL) return dir > 0 ? go(k_sweep3<NS, SW_GS_FULL, 1>) : go(k_sweep3<NS, SW_GS_FULL, -1>);
  if (kind == SW_ILU_L) return go(k_sweep3<NS, SW_ILU_L, 1>);
  return go(k_sweep3<NS, SW_ILU_U, -1>);
}

}  // namespace

// The FP64 natural-order kernel's levels: one unknown per point, a canonical
// mask, at most 12 warps of columns (8 for Gauss-Seidel with old values).
bool sweep3_supported(const LevelView& L, int kind) {
  const int ns = L.s.ns;
  if (L.B != 1 || L.pk != K64) return false;
  if (!((ns == 27 && canonical<27>(L.s)) || (ns == 7 && canonical<7>(L.s)) || (ns == 19 && canonical<19>(L.s))))
    return false;
  const int NW = (L.g.ny + 31) / 32;
  const int maxt = kind == SW_GS_FULL ? max_threads<SW_GS_FULL>() : max_threads<SW_ILU_L>();
  return (NW + 2) * 32 <= maxt && (size_t)L.g.nx * NW <= (size_t)kProgSlots;
}

cudaError_t launch_sweep3(const LevelView& L, int kind, int dir, const void* M, const void* dinv, double w,
                          const void* b, void* u, SweepWs* ws, int* err, const SweepCfg& cfg, cudaStream_t st) {
  if (!sweep3_supported(L, kind)) return cudaErrorNotSupported;
  Sweep3Params P;
  P.g = L.g;
  P.budget_ns = cfg.budget_ns;
  P.M = (const double*)M;
  P.dinv = (const double*)dinv;
  P.w = w;
  P.b = (const double*)b;
  P.u = (double*)u;
  P.ws = ws;
  P.err = err;
  cudaError_t e;
  if (L.s.ns == 27) e = launch_kind<27>(kind, dir, P, st);
  else if (L.s.ns == 7) e = launch_kind<7>(kind, dir, P, st);
  else e = launch_kind<19>(kind, dir, P, st);
  smg_count_launch(1);
  return e;
}
