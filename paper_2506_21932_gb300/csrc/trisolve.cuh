// Kernel of the sheared wavefront (tri.cuh), included by one translation unit
// per working precision.
//
// A CTA owns a tile: one strip of 32 I (one lane each) and G consecutive
// sheared planes P.  All its planes advance in lock step, one point per lane
// and time step, with one barrier per step; values of the last steps live in
// a shared ring [plane][time][lane], where every operand of a point is a
// constant (plane, time, lane) offset away.  Two planes below the tile and
// the lane left of the strip belong to other CTAs.
//
// Hand-over between CTAs: every point that another tile reads is also written
// to its tile's mailbox as 64-bit words that carry half of the value (FP64)
// or all of it (FP32) beside the launch's tag, so the word itself says whether
// it is there: the reader polls the words it needs, without flags or fences,
// and a hop costs about one trip to L2 and back.  Tags are the number of the
// launch on this workspace; nothing is reset between launches.
//
// Warps of a CTA:
//  * G main warps finish the points of their plane: the terms one step old
//    (own column, left lane, previous plane), the diagonal, the stores;
//  * H = 3 helper warps per plane (FP64, 19/27-point) form the partial sum of
//    the older terms ahead of time, four or more steps old, then three, then
//    two, handing it on through shared memory.  An SM sub-partition issues
//    one FP64 warp instruction per 64 cycles and a warp issues in order, so
//    one warp alone would take the 13 or 14 FP64 instructions of a 27-point
//    step in a row.  The sums keep one order with and without helpers.
//    Coefficients of the next step are loaded before the barrier that opens it;
//  * the sync warp joins the step barrier once the halo and the records of
//    the next step are there;
//  * three loader warps (one per plane below the tile, one for the lane left
//    of the strip) poll the mailboxes and fill the ring, the record warp issues
//    one bulk copy per step and array into a ring of stages, the tracker warp
//    waits for them in order: these run ahead of the steps.
// Tiles are claimed by a ticket in the order of their first time step, so a
// CTA only waits for tiles that running CTAs own.  Every wait is bounded; on
// expiry the error word is set and every CTA drains its copies and leaves.
#pragma once
#include <algorithm>
#include <climits>

#include "mailbox.cuh"
#include "tri.cuh"

namespace tri {

constexpr int kRing = 16;             // time slots of the value ring
constexpr int kAhead = 3;             // the oldest-terms stage works kAhead steps ahead
constexpr int kRecAhead = kAhead + 1;  // and loads its coefficients one step before that
constexpr int kOldest = 7;            // largest age of an operand
constexpr int kDone = INT_MAX / 2;
constexpr int kLanes = 33;            // ring row: lane -1 and the strip's 32

// The step barrier: barrier 1 of N threads.
template <int N>
__device__ __forceinline__ void step_barrier() {
  asm volatile("bar.sync 1, %0;" ::"n"(N) : "memory");
}
// Products that must not be contracted into a following add.
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }

// Age of the operand of lower entry e (steps since it was finished), and the
// stage that adds it: 0 four or more, 1 three, 2 two, 3 one step old.
template <int NS>
__host__ __device__ constexpr int age(int e) {
  using S = Shape<NS>;
  return -(S::SA * S::o(e, 0) + S::SB * S::o(e, 1) + S::o(e, 2));
}
template <int NS>
__host__ __device__ constexpr int stage_of(int e) {
  return age<NS>(e) >= 4 ? 0 : 4 - age<NS>(e);
}

struct TriParams {
  Grid g;
  int ntiles, ngrp, F;  // tiles; groups of planes per strip; steps per tile
  const int* tiles;     // strip << 16 | group, in the order they are claimed
  int flip;
  unsigned long long budget_ns;
  const void *rec, *b, *h, *old;
  void *u, *emit;
  int relax;
  double w;
  void* mail;
  SweepWs* ws;
  int* err;
};

struct TriShared {
  unsigned long long full[16];  // stage barriers
  int hready[3];                // per loader: its halo values of every time < hready are in the ring
  int rready;                   // records and vectors of every time < rready are in their stages
  int done;                     // every step < done is finished
  int abort;                    // a wait ran out (or another CTA's did)
  int quit;                     // the warps of the step barrier leave in this step
  int tile;
};

template <int G, int H>
__host__ __device__ constexpr int tri_threads() {
  return (G * (H + 1) + 6) * 32;
}
template <int PK, int NS, bool HD, int G, int H>
struct TriSmem {
  using V = typename Prec<PK>::vec;
  static constexpr int RB = TriRec<PK, NS, HD>::BYTES;
  static constexpr size_t ring = sizeof(V) * (G + 2) * kRing * kLanes;
  static constexpr size_t hand = H ? sizeof(V) * 3 * 2 * G * 32 : 0;
  __host__ __device__ static constexpr size_t stage(int nvec) { return (size_t)G * (RB + nvec * 32 * sizeof(V)); }
  static constexpr size_t head = (ring + hand + 127) / 128 * 128;
};

// Terms of a stage in the order they are added: sweep order, but where both
// kinds are two steps old the terms of the same x-plane (o0 == 0) first: the
// order of the natural-layout sweep (k_sweep3.cu).
template <int NS>
__host__ __device__ constexpr int nterms(int stg) {
  int n = 0;
  for (int e = 0; e < Shape<NS>::EC; ++e) n += stage_of<NS>(e) == stg;
  return n;
}
template <int NS>
__host__ __device__ constexpr int term(int stg, int t) {
  for (int pass = 0; pass < 2; ++pass)
    for (int e = 0; e < Shape<NS>::EC; ++e) {
      if (stage_of<NS>(e) != stg) continue;
      if ((stg == 2 ? (Shape<NS>::o(e, 0) == 0) != (pass == 0) : pass != 0)) continue;
      if (t-- == 0) return e;
    }
  return 0;
}

template <int PK, int NS, int STG>
struct Terms {
  using V = typename Prec<PK>::vec;
  static constexpr int N = nterms<NS>(STG);
  V c[N ? N : 1];
  // coefficients from a record (stored negated where the sum starts from b)
  __device__ __forceinline__ void load(const char* rec, int lane) {
#pragma unroll
    for (int t = 0; t < N; ++t) {
      const int e = term<NS>(STG, t);
      if constexpr (PK == KBF) {
        const unsigned wd = reinterpret_cast<const unsigned*>(rec)[(e >> 1) * 32 + lane];
        c[t] = __bfloat162float(__ushort_as_bfloat16((unsigned short)((e & 1) ? (wd >> 16) : (wd & 0xffffu))));
      } else {
        c[t] = reinterpret_cast<const V*>(rec)[e * 32 + lane];
      }
    }
  }
  // a plus the terms of the point of time T; rb: the lane's cell of plane p - 2, time 0
  __device__ __forceinline__ V add(V a, const V* rb, int T) const {
    using S = Shape<NS>;
    V x[N ? N : 1];
#pragma unroll
    for (int t = 0; t < N; ++t) {
      const int e = term<NS>(STG, t);
      const int dl = S::o(e, 0), dp = S::o(e, 0) + S::o(e, 1);
      x[t] = rb[(2 + dp) * (kRing * kLanes) + ((T - age<NS>(e)) & (kRing - 1)) * kLanes + dl];
    }
#pragma unroll
    for (int t = 0; t < N; ++t) a = fma(c[t], x[t], a);
    return a;
  }
};

// CTAs per SM the registers are cut for: two where the tile is small.
template <int G, int H>
__host__ __device__ constexpr int tri_ctas() {
  return tri_threads<G, H>() <= 480 ? 2 : 1;
}

template <int PK, int NS, bool HD, int G, int H, int NSTG>
__global__ void __launch_bounds__(tri_threads<G, H>(), tri_ctas<G, H>()) k_tri(TriParams P) {
  using V = typename Prec<PK>::vec;
  using S = Shape<NS>;
  using R = TriRec<PK, NS, HD>;
  using SM = TriSmem<PK, NS, HD, G, H>;
  constexpr int SP = Shear<NS>::SP, SL = Shear<NS>::SL;
  constexpr int NC = G * (H + 1);  // compute warps
  using ML = Mail<V>;
  constexpr int ME = 64 + (G > 2 ? G - 2 : 0);  // mailbox entries of a step: the last two planes, lane 31 of the others
  extern __shared__ __align__(128) unsigned char dyn[];
  __shared__ TriShared sh;
  V* ring = reinterpret_cast<V*>(dyn);
  V* hand = reinterpret_cast<V*>(dyn + SM::ring);
  // a stage: the records of G planes, then rows of G x 32 vector values: the
  // right-hand side, h, the old iterate
  const int nvec = 1 + (P.h != nullptr) + (P.relax == 2);
  const int hoff = G * 32, ooff = (1 + (P.h != nullptr)) * G * 32;
  const unsigned stage_bytes = (unsigned)SM::stage(nvec);
  char* stages = reinterpret_cast<char*>(dyn) + SM::head;

  const Grid g = P.g;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nstrip = (g.nx + 31) >> 5;
  V* u = (V*)P.u;
  V* ev = (V*)P.emit;
  // Slot of point (I, p, time T) in the result's stream: column(I, p) + dstep * T.
  const int dstep = P.flip ? -G * 32 : G * 32;
  auto column = [&](int I, int p) -> long long {
    int c = I, q = p, k0 = -(SP * p + SL * I);  // K = T + k0
    if (P.flip) {
      c = g.nx - 1 - I;
      q = g.nx + g.ny - 2 - p;
      k0 = g.nz - 1 - k0;  // the mirrored K at T = 0
    }
    const int cw = c >> 5, cl = c & 31, pr = q - 32 * cw, cd = pr / G, cg = pr % G;
    return (((long long)(cw * P.ngrp + cd) * P.F + SP * cg + SL * cl + k0) * G + cg) * 32 + cl;
  };
  if (threadIdx.x == 0) {
    for (int t = 0; t < NSTG; ++t) mbar_init(&sh.full[t], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  typename ML::word* mail = (typename ML::word*)P.mail;
  const unsigned tag = (unsigned)P.ws->epoch + 1u;
  unsigned base = 0;  // stage fills of the tiles before this one
  for (;;) {
    __syncthreads();
    if (threadIdx.x == 0) {
      const int t = atomicAdd(&P.ws->ticket, 1);
      sh.tile = t < P.ntiles ? P.tiles[t] : -1;
    }
    __syncthreads();
    const int tile = sh.tile;
    if (tile < 0) break;
    const int w = tile >> 16, dg = tile & 0xffff;
    const int p0 = 32 * w + G * dg;  // first plane
    const int T0 = SP * p0 + SL * 32 * w;
    const int Te = SP * (p0 + G - 1) + SL * min(32 * w + 31, g.nx - 1) + g.nz - 1;
    for (int t = threadIdx.x; t < (G + 2) * kRing * kLanes; t += blockDim.x) ring[t] = V(0);
    if (threadIdx.x == 0) {
      sh.hready[0] = sh.hready[1] = sh.hready[2] = T0 - kOldest;
      sh.rready = T0;
      sh.done = T0 - kRecAhead;
      sh.abort = 0;
      sh.quit = INT_MAX;
    }
    __syncthreads();
    const int I = 32 * w + lane;

    if (warp < NC) {
      // ---- compute warps
      int role, pl;
      if (H == 0) {
        role = 0;
        pl = warp;
      } else {
        role = warp / G;
        pl = warp % G;
        // two planes: spread the 4 + 5 + 3 + 2 FP64 instructions of a plane's
        // warps so that every sub-partition (warp % 4) gets 7
        if (G == 2 && role >= 2) pl = 1 - pl;
      }
      const int p = p0 + pl, J = p - I;
      const bool colok = I < g.nx && J >= 0 && J < g.ny;
      const int koff = SP * p + SL * I;
      const V* rb = ring + pl * (kRing * kLanes) + lane + 1;
      V* own = ring + (pl + 2) * (kRing * kLanes) + lane + 1;
      auto rec_of = [&](int T) { return stages + ((unsigned)(base + T - T0) % NSTG) * stage_bytes + pl * R::BYTES; };
      auto vec_of = [&](int T, int which) {
        return reinterpret_cast<const V*>(stages + ((unsigned)(base + T - T0) % NSTG) * stage_bytes + G * R::BYTES) +
               which + pl * 32 + lane;
      };
      // hand-over cells of stage pair sp: [sp][time & 1][plane][lane]
      auto cell = [&](int sp, int T) -> V& { return hand[((sp * 2 + (T & 1)) * G + pl) * 32 + lane]; };
      long long at = colok ? column(I, p) + (long long)dstep * (T0 - kRecAhead) : 0;
      const V wv = (V)P.w;
      // mailbox entry of this lane: every lane of the last two planes, lane 31 of the others
      const bool post = pl >= G - 2 || lane == 31;
      typename ML::word* mb = mail + ((long long)(w * P.ngrp + dg) * P.F - T0) * ME +
                              (pl >= G - 2 ? (pl - (G - 2)) * 32 + lane : 64 + pl);
      // opens step T; false after the last step.  The sync warp leaves at the
      // barrier of step quit; a warp reads that at the end of a step, off the
      // critical path (the step in between only does harmless work), and
      // leaves once it has passed that barrier too.
      auto open = [&](int T) {
        step_barrier<(NC + 1) * 32>();
        return T <= Te;
      };
      auto start = [&](int T) { return PK == KBF ? V(0) : *vec_of(T, 0); };
      // first step: its last loads are the first ones of a record that exists
      const int Tb = T0 - kRecAhead;
      if (role == 0) {
        // H == 0: c1, c2, c3 are the partial sums of T + 1, T + 2, T + 3 before this step's share
        Terms<PK, NS, 3> k3;
        Terms<PK, NS, 2> k2;
        Terms<PK, NS, 1> k1;
        Terms<PK, NS, 0> k0;
        V d = V(0), c1 = V(0), c2 = V(0), c3 = V(0), b3 = V(0);
        auto fetch = [&](int T) {  // operands of step T that do not depend on the step before
          k3.load(rec_of(T), lane);
          if (HD) d = reinterpret_cast<const V*>(rec_of(T) + R::D_OFF)[lane];
          if (H == 0) {
            k2.load(rec_of(T + 1), lane);
            k1.load(rec_of(T + 2), lane);
            k0.load(rec_of(T + 3), lane);
            b3 = start(T + 3);
          }
        };
        fetch(Tb);
        for (int T = Tb; open(T); ++T) {
          const int K = T - koff;
          const bool ok = colok && K >= 0 && K < g.nz;
          V a = k3.add(H ? cell(2, T) : c1, rb, T);
          if (PK == KBF) {
            a = mul_rn(V(reinterpret_cast<const float*>(rec_of(T) + R::S_OFF)[lane]), a);
            a = *vec_of(T, 0) - a;
          }
          V r = a;
          if (HD) r = a * d;
          if (P.relax) r = P.relax == 1 ? wv * r : fma(wv, r, mul_rn(V(1) - wv, *vec_of(T, ooff)));
          own[(T & (kRing - 1)) * kLanes] = ok ? r : V(0);
          if (ok) {
            if (post) ML::put(mb + (long long)T * ME, r, tag);
            u[at] = r;
            if (ev) ev[at] = P.h ? a + *vec_of(T, hoff) : a;
          }
          at += dstep;
          if (H == 0) {
            c1 = k2.add(c2, rb, T + 1);
            c2 = k1.add(c3, rb, T + 2);
            c3 = k0.add(b3, rb, T + 3);
          }
          fetch(T + 1);
          if (sh.quit <= T) break;
        }
      } else if (role == 1) {
        Terms<PK, NS, 0> k;
        k.load(rec_of(Tb + 3), lane);
        V b3 = start(Tb + 3);
        for (int T = Tb; open(T); ++T) {
          cell(0, T + 3) = k.add(b3, rb, T + 3);
          k.load(rec_of(T + 4), lane);
          b3 = start(T + 4);
          if (sh.quit <= T) break;
        }
      } else if (role == 2) {
        Terms<PK, NS, 1> k;
        k.load(rec_of(Tb + 2), lane);
        for (int T = Tb; open(T); ++T) {
          cell(1, T + 2) = k.add(cell(0, T + 2), rb, T + 2);
          k.load(rec_of(T + 3), lane);
          if (sh.quit <= T) break;
        }
      } else {
        Terms<PK, NS, 2> k;
        k.load(rec_of(Tb + 1), lane);
        for (int T = Tb; open(T); ++T) {
          cell(2, T + 1) = k.add(cell(1, T + 1), rb, T + 1);
          k.load(rec_of(T + 2), lane);
          if (sh.quit <= T) break;
        }
      }
    } else if (warp == NC) {
      // ---- sync warp
      int hh = T0 - kOldest, rr = T0;
      for (int T = T0 - kRecAhead; T <= Te + 1; ++T) {
        bool ok = true;
        if (T <= Te) {
          // halo values up to time T - 1, records up to the one loaded in this step
          const int need = min(T + kRecAhead, Te);
          while (hh < T || rr <= need) {
            hh = min(min(ld_acq_cta(&sh.hready[0]), ld_acq_cta(&sh.hready[1])), ld_acq_cta(&sh.hready[2]));
            rr = ld_acq_cta(&sh.rready);
            if (hh >= T && rr > need) break;
            if (ld_acq_cta(&sh.abort)) {
              ok = false;
              break;
            }
          }
        }
        ok = __all_sync(0xffffffffu, ok);
        if (!ok && lane == 0) sh.quit = T;
        __syncwarp();
        step_barrier<(NC + 1) * 32>();
        if (!ok) break;
        if (lane == 0) st_rel_cta(&sh.done, T);
      }
    } else if (warp < NC + 4) {
      // ---- loader warps: plane p0-2, plane p0-1 (a column per lane), and the
      // column left of the strip (lane q < G + 2: plane p0-2+q)
      const int c = warp - (NC + 1);
      constexpr int SG = 32 / G;
      constexpr int kBatch = sizeof(V) == 8 ? 4 : 8;  // time steps asked for at once
      const int pc = p0 - 2 + (c < 2 ? c : lane), Ic = c < 2 ? I : 32 * w - 1, Jc = pc - Ic;
      const bool mine = c < 2 || lane < G + 2;
      const bool okc = mine && Ic >= 0 && Ic < g.nx && Jc >= 0 && Jc < g.ny;
      // owner: the tile below, or the left strip's tiles of planes p0-2, p0-1 and of the own planes
      const int cw = c < 2 ? w : w - 1;
      const int cd = c < 2 ? dg - 1 : lane < 2 ? dg + SG - 1 : dg + SG;
      const int cg = c < 2 ? G - 2 + c : lane < 2 ? G - 2 + lane : lane - 2;
      const int ct0 = SP * (32 * cw + G * cd) + SL * 32 * cw;
      const int e = cg >= G - 2 ? (cg - (G - 2)) * 32 + (c < 2 ? lane : 31) : 64 + cg;
      const typename ML::word* src =  // entry of time 0
          okc ? mail + ((long long)(cw * P.ngrp + cd) * P.F - ct0) * ME + e : mail;
      V* dst = ring + (c < 2 ? c : min(lane, G + 1)) * (kRing * kLanes) + (c < 2 ? lane + 1 : 0);
      // times at which this lane has a point to fetch
      const int t_lo = okc ? SP * pc + SL * Ic : INT_MAX, t_hi = okc ? t_lo + g.nz : INT_MIN;
      int tau = T0 - kOldest;
      unsigned long long t_wait = 0;
      unsigned iter = 0;
      int ask = 1;  // one step while waiting for the first, a batch once they come
      if (!__any_sync(0xffffffffu, okc)) tau = Te;
      while (tau < Te) {
        // lane 0's view for all: the votes below need every lane
        const int n = __shfl_sync(0xffffffffu, min(min(ld_acq_cta(&sh.done) + kRing - 4, Te) - tau, ask), 0);
        int got = 0;
        if (n > 0) {
          typename ML::word val[kBatch];
#pragma unroll
          for (int q = 0; q < kBatch; ++q) {
            val[q] = ML::value(V(0), tag);
            if (q < n && tau + q >= t_lo && tau + q < t_hi) val[q] = ML::get(src + (long long)(tau + q) * ME);
          }
#pragma unroll
          for (int q = 0; q < kBatch; ++q)
            if (q < n && got == q && __all_sync(0xffffffffu, ML::ok(val[q], tag))) {
              if (mine) dst[((tau + q) & (kRing - 1)) * kLanes] = ML::val(val[q]);
              got = q + 1;
            }
        }
        if (got > 0) {
          tau += got;
          __syncwarp();
          if (lane == 0) st_rel_cta(&sh.hready[c], tau);
          t_wait = 0;
          ask = kBatch;
          continue;
        }
        bool stop = false;
        if (lane == 0) {
          if (n > 0) {
            // bounded: the owners must make progress within the budget
            const unsigned long long now = globaltimer_ns();
            if (t_wait == 0) t_wait = now;
            else if (now - t_wait > P.budget_ns) {
              atomicCAS(P.err, 0, DEV_ERR_TIMEOUT);
              stop = true;
            }
          }
          if ((++iter & 63u) == 0) stop = stop || ld_relaxed(P.err) != 0;
          stop = stop || ld_acq_cta(&sh.abort) != 0;
        }
        if (__shfl_sync(0xffffffffu, stop, 0)) {
          if (lane == 0) st_rel_cta(&sh.abort, 1);
          break;
        }
        if (ask == 1) __nanosleep(100);
        else if (n <= 0) __nanosleep(40);
      }
      // the last steps need no more halo
      if (tau >= Te && lane == 0) st_rel_cta(&sh.hready[c], kDone);
    } else if (warp == NC + 4) {
      // ---- record warp
      // one lane; step f of the tile is one run in every stream
      if (lane == 0) {
        const int nfill = Te - T0 + 1;
        const long long step0 = (long long)(w * P.ngrp + dg) * P.F;
        const char* rec = (const char*)P.rec + step0 * (G * R::BYTES);
        const V* bv = (const V*)P.b + step0 * (G * 32);
        const V* hv = (const V*)P.h + step0 * (G * 32);
        const V* ov = (const V*)P.old + step0 * (G * 32);
        constexpr unsigned vbytes = G * 32 * sizeof(V);
        int done = T0 - kRecAhead, issued = 0;
        for (int f = 0; f < nfill; ++f) {
          const int T = T0 + f;
          // the stage's previous occupant (time T - NSTG) is finished
          bool stop = false;
          while (f >= NSTG && done <= T - NSTG) {
            done = ld_acq_cta(&sh.done);
            if (done > T - NSTG) break;
            if (ld_acq_cta(&sh.abort)) {
              stop = true;
              break;
            }
            __nanosleep(20);
          }
          if (stop) break;
          const unsigned slot = (base + f) % NSTG;
          unsigned long long* bar = &sh.full[slot];
          char* st = stages + slot * stage_bytes;
          V* sv = reinterpret_cast<V*>(st + G * R::BYTES);
          mbar_expect_tx(bar, stage_bytes);
          bulk_copy_g2s(st, rec + (long long)f * (G * R::BYTES), G * R::BYTES, bar);
          bulk_copy_g2s(sv, bv + (long long)f * (G * 32), vbytes, bar);
          if (P.h) bulk_copy_g2s(sv + hoff, hv + (long long)f * (G * 32), vbytes, bar);
          if (P.relax == 2) bulk_copy_g2s(sv + ooff, ov + (long long)f * (G * 32), vbytes, bar);
          issued = f + 1;
        }
        // every copy has landed before the tile is left (at once, unless a wait
        // ran out and the tracker left early)
        for (int f = max(0, issued - NSTG); f < issued; ++f) {
          const unsigned a = base + f;
          const unsigned long long t0 = globaltimer_ns();
          while (!mbar_try_wait(&sh.full[a % NSTG], (a / NSTG) & 1u))
            if (globaltimer_ns() - t0 > kCopyWaitNs) break;
        }
      }
    } else if (lane == 0) {
      // ---- tracker warp, one lane
      bool stop = false;
      for (int T = T0; T <= Te && !stop; ++T) {
        const unsigned f = base + (T - T0);
        unsigned long long t0 = 0;
        while (!mbar_try_wait(&sh.full[f % NSTG], (f / NSTG) & 1u)) {
          if (ld_acq_cta(&sh.abort)) {
            stop = true;
            break;
          }
          // the record warp waits for the steps, the steps for the halo: only
          // a copy that is due counts against the bound
          if (T > ld_acq_cta(&sh.done) + NSTG - 2) {
            t0 = 0;
            continue;
          }
          const unsigned long long now = globaltimer_ns();
          if (t0 == 0) t0 = now;
          else if (now - t0 > kCopyWaitNs) {
            atomicCAS(P.err, 0, DEV_ERR_TIMEOUT);
            st_rel_cta(&sh.abort, 1);
            stop = true;
            break;
          }
        }
        if (!stop) st_rel_cta(&sh.rready, T + 1);
      }
    }
    base += (unsigned)(Te - T0 + 1);
    __syncthreads();
    if (sh.abort) break;
  }
  if (threadIdx.x == 0) {
    __threadfence();
    sh.tile = (atomicAdd(&P.ws->finished, 1) == (int)gridDim.x - 1);
  }
  __syncthreads();
  if (sh.tile && threadIdx.x == 0) {
    P.ws->ticket = 0;
    P.ws->epoch = (int)tag;
    __threadfence();
    P.ws->finished = 0;
  }
}

template <int PK, int NS, bool HD, int G, int H, int NSTG>
cudaError_t launch_tri_kernel(const TriParams& P, cudaStream_t st) {
  using SM = TriSmem<PK, NS, HD, G, H>;
  const int nvec = 1 + (P.h != nullptr) + (P.relax == 2);
  const size_t smem = SM::head + NSTG * SM::stage(nvec);
  auto kern = k_tri<PK, NS, HD, G, H, NSTG>;
  int dev = 0, nsm = 0, per = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kern, tri_threads<G, H>(), smem);
  if (e != cudaSuccess) return e;
  const int grid = std::min(P.ntiles, nsm * std::max(1, per));
  kern<<<grid, tri_threads<G, H>(), smem, st>>>(P);
  return cudaGetLastError();
}

}  // namespace tri

// One entry per working precision, each compiled in its own translation unit.
cudaError_t tri_launch_k64(int ns, bool hd, int G, bool helpers, const tri::TriParams& P, cudaStream_t st);
cudaError_t tri_launch_k32(int ns, bool hd, const tri::TriParams& P, cudaStream_t st);
cudaError_t tri_launch_kbf(int ns, bool hd, const tri::TriParams& P, cudaStream_t st);
