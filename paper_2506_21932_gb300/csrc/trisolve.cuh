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
// What bounds a solve on all but the largest grids is the chain of time steps
// plus one hop per tile; a step is the barrier, three dependent multiply-adds
// and a warp's instructions one after another (27-point: 0.36 us FP64 with 2
// planes, 0.25 FP32, 0.20 BF16; 7-point 0.27 / 0.20), so whatever else a step
// needs is moved to other warps.  On the largest FP64 grids the FP64 pipe is
// full (384^3: 2.45 ms a solve, 1.56 ms of multiply-adds).
//
// Hand-over between CTAs: every point that another tile reads is written as
// 64-bit words that carry half of the value (FP64) or all of it (FP32) beside a
// tag, so the word itself says whether it is there: the reader polls the words
// it needs, without flags or fences.  CL consecutive tiles of a strip form a
// cluster: there the words go to a mailbox of kMail time steps in the reader's
// shared memory (tag: time + 1; the reader tells how far it has taken them) and
// a hop takes 0.45 us.  The tiles between clusters and the strip on the right
// read words in global memory (tag: number of the launch on this workspace, so
// nothing is reset between launches), 1.1 us a hop.
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
//    the next step are there and the next tile has room;
//  * three loader warps (one per plane below the tile, one for the lane left
//    of the strip) poll the mailboxes and fill the ring, the record warp issues
//    one bulk copy per array and chunk of steps into a ring of stages, the
//    tracker warp waits for them in order: these run ahead of the steps.
// Units of CL tiles are claimed by a ticket in the order of their first time
// step, so a cluster only waits for tiles that running clusters own.  Every
// wait is bounded; on expiry the error word is set, the steps of the tile run
// through without waiting, and every CTA drains its copies and leaves.
#pragma once
#include <algorithm>
#include <climits>
#include <type_traits>

#include "mailbox.cuh"
#include "tri.cuh"

namespace tri {

constexpr int kRing = 16;             // time slots of the value ring
constexpr int kAhead = 3;             // the oldest-terms stage works kAhead steps ahead
constexpr int kRecAhead = kAhead + 1;  // and loads its coefficients one step before that
constexpr int kOldest = 7;            // largest age of an operand
constexpr int kDone = INT_MAX / 2;
constexpr int kMail = 16;             // time slots of the mailbox in shared memory
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
  int nstg;             // record stages (steps)
  int nunits, ngrp;     // units of CL tiles; groups of planes stored per strip
  int rows, last_row;   // steps stored per group; stored step of the solve's last time
  int mrows;            // steps of a group in the mailbox
  const int* tiles;     // strip << 16 | first group of a unit, in the order they are claimed
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
  unsigned long long full[8];   // barriers of the chunks of stages
  PeerCounter taken[2];         // per plane that the next tile reads: it has taken every time < taken
  int hready[3];                // per loader: its halo values of every time < hready are in the ring
  int rready;                   // records and vectors of every time < rready are in their stages
  int done;                     // every step < done is finished
  int abort;                    // a wait ran out (or another CTA's did)
  int tile;
  int row, mrow;                // stored step of the tile's first time, in streams and mailbox
};

template <int G, int H>
__host__ __device__ constexpr int tri_threads() {
  return (G * (H + 1) + 6) * 32;
}
// Steps per bulk copy: a copy takes the record warp about 200 cycles to issue,
// more than half a step of the fast kernels for the two or three of a step.
template <int NSTG>
constexpr int kChunk = NSTG >= 16 ? 4 : 2;

template <int PK, int NS, bool HD, int G, int H>
struct TriSmem {
  using V = typename Prec<PK>::vec;
  static constexpr int RB = TriRec<PK, NS, HD>::BYTES;
  static constexpr size_t ring = sizeof(V) * (G + 2) * kRing * kLanes;
  static constexpr size_t hand = H ? sizeof(V) * 3 * 2 * G * 32 : 0;
  __host__ __device__ static constexpr size_t stage(int nvec) { return (size_t)G * (RB + nvec * 32 * sizeof(V)); }
  // the last two planes of the tile below, where the same cluster has it
  static constexpr size_t mail = sizeof(typename Mail<V>::word) * 2 * kMail * 32;
  static constexpr size_t head = (mail + ring + hand + 127) / 128 * 128;
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
  // coefficients from the lane's column of a record (stored negated where the sum starts from b)
  __device__ __forceinline__ void load(const char* rec) {
#pragma unroll
    for (int t = 0; t < N; ++t) {
      const int e = term<NS>(STG, t);
      if constexpr (PK == KBF) {
        const unsigned wd = reinterpret_cast<const unsigned*>(rec)[(e >> 1) * 32];
        c[t] = __bfloat162float(__ushort_as_bfloat16((unsigned short)((e & 1) ? (wd >> 16) : (wd & 0xffffu))));
      } else {
        c[t] = reinterpret_cast<const V*>(rec)[e * 32];
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
  typename ML::word* own_mail = reinterpret_cast<typename ML::word*>(dyn);  // [plane][time][lane]
  V* ring = reinterpret_cast<V*>(dyn + SM::mail);
  V* hand = reinterpret_cast<V*>(dyn + SM::mail + SM::ring);
  // stages: the records of G planes per step, then G x 32 vector values per
  // step: the right-hand side, h, the old iterate
  constexpr int C = kChunk<NSTG>;
  const int nstg = P.nstg, nch = nstg / C, nvec = 1 + (P.h != nullptr) + (P.relax == 2);
  const int hoff = nstg * G * 32, ooff = (1 + (P.h != nullptr)) * nstg * G * 32;
  char* stages = reinterpret_cast<char*>(dyn) + SM::head;
  V* const vecs = reinterpret_cast<V*>(stages + nstg * (G * R::BYTES));

  const Grid g = P.g;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  V* u = (V*)P.u;
  V* ev = (V*)P.emit;
  // Store of group d of strip w (d < ngrp + 32, few subtractions), and a stored step
  // of rows counted back below the first.
  auto group = [&](int w, int d) -> long long {
    while (d >= P.ngrp) d -= P.ngrp;
    return w * P.ngrp + d;
  };
  auto back = [&](int row, int rows) {
    while (row < 0) row += rows;
    return row;
  };
  if (threadIdx.x == 0) {
    for (int t = 0; t < nch; ++t) mbar_init(&sh.full[t], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  typename ML::word* mail = (typename ML::word*)P.mail;
  const unsigned tag = (unsigned)P.ws->epoch + 1u;
  unsigned base = 0;  // chunk fills of the tiles before this one
  const int rank = cluster_rank(), csize = cluster_size();
  if (threadIdx.x == 0) sh.abort = 0;
  for (;;) {
    cluster_sync();
    // the first CTA claims a unit for all, or ends the launch for all
    if (rank == 0 && threadIdx.x == 0) {
      bool stop = false;
      for (int r = 0; r < csize; ++r) stop = stop || ld_peer(peer_addr(&sh.abort, r)) != 0;
      const int t = stop ? P.nunits : atomicAdd(&P.ws->ticket, 1);
      const int unit = t < P.nunits ? P.tiles[t] : -1;
      for (int r = 0; r < csize; ++r) st_peer(peer_addr(&sh.tile, r), unit);
    }
    cluster_sync();
    const int tile = sh.tile;
    if (tile < 0) break;
    const int w = tile >> 16, dg = (tile & 0xffff) + rank;
    const int ntile = (g.ny + min(32, g.nx - 32 * w) - 1 + G - 1) / G;  // tiles of the strip
    const bool live = dg < ntile;                                      // a unit may end early
    const bool below = rank > 0, above = rank + 1 < csize && dg + 1 < ntile;  // neighbours in the cluster
    const int p0 = 32 * w + G * dg;  // first plane
    const int T0 = SP * p0 + SL * 32 * w;
    const int Te = SP * (p0 + G - 1) + SL * min(32 * w + 31, g.nx - 1) + g.nz - 1;
    for (int t = threadIdx.x; t < (G + 2) * kRing * kLanes; t += blockDim.x) ring[t] = V(0);
    // tags in it are times + 1
    for (int t = threadIdx.x; t < 2 * kMail * 32; t += blockDim.x) own_mail[t] = ML::value(V(0), 0);
    if (threadIdx.x == 0) {
      sh.taken[0].v = sh.taken[1].v = T0;
      sh.hready[0] = sh.hready[1] = sh.hready[2] = T0 - kOldest;
      sh.rready = T0;
      sh.done = T0 - kRecAhead;
      sh.abort = 0;
      sh.row = T0 % P.rows;
      sh.mrow = T0 % P.mrows;
    }
    cluster_sync();
    if (!live) continue;
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
        // two planes: the sub-partition (warp % 4) of a main warp gets the
        // shortest helper too (4 + 2 FP64 instructions), the others share one (5 + 3)
        if (G == 2 && role >= 2) role = 5 - role;
        // (four planes: every sub-partition has all four kinds)
      }
      const int p = p0 + pl, J = p - I;
      const bool colok = I < g.nx && J >= 0 && J < g.ny;
      const V* rb = ring + pl * (kRing * kLanes) + lane + 1;
      V* own = ring + (pl + 2) * (kRing * kLanes) + lane + 1;
      // stage of time T >= T0 - nstg and the one after it; the lane's column of
      // the record and its vector values there
      const int slot0 = (int)(base % (unsigned)nch) * C;
      auto stage_of_time = [&](int T) {
        const int t = slot0 + T - T0;
        return t < 0 ? t + nstg : t < nstg ? t : t - nstg;
      };
      auto next = [&](int q) { return q + 1 == nstg ? 0 : q + 1; };
      const char* const recl = stages + pl * R::BYTES + lane * (int)sizeof(V);
      const V* const vecl = vecs + pl * 32 + lane;
      auto rec = [&](int q) { return recl + q * (G * R::BYTES); };
      auto vec = [&](int q, int which) { return vecl[q * (G * 32) + which]; };
      // hand-over cells of stage pair sp: [sp][time & 1][plane][lane]
      auto cell = [&](int sp, int T) -> V& { return hand[((sp * 2 + (T & 1)) * G + pl) * 32 + lane]; };
      const V wv = (V)P.w;
      // The main warp's chain has to get into the FP64 pipe before the helpers of
      // its sub-partition: with two planes the one there waits for it (128^3: 0.45
      // to 0.41 ms a solve), with four, where a turn would come too late for
      // three, they hold back by about the chain's first product (256^3: 1.21 to 1.14;
      // the time is the clock's, 100 ns or 200 of the 2070 MHz cycles of these figures).
      constexpr bool kTurn = H && G == 2;
      auto hold = [&] {
        if (G == 4) __nanosleep(100);
      };
      auto start = [&](int q) { return PK == KBF ? V(0) : vec(q, 0); };
      // first step: its last loads are the first ones of a record that exists
      const int Tb = T0 - kRecAhead;
      if (role == 0) {
        const int koff = SP * p + SL * I;
        const unsigned nk = colok ? (unsigned)g.nz : 0u;
        // The lane's results: column (c, q) of the result's stream, whose time is T or
        // (mirrored) Tm - T; the stored steps run out at time tw.
        int c = I, q = p, row = back(sh.row - kRecAhead, P.rows), tw = Tb + P.rows - row;
        const int dstep = P.flip ? -G * 32 : G * 32;
        if (P.flip) {
          c = g.nx - 1 - I;
          q = g.nx + g.ny - 2 - p;
          row = back(P.last_row - row, P.rows);
          tw = Tb + row + 1;
        }
        const int cw = c >> 5, cp = q - 32 * cw;
        const long long at = colok ? ((group(cw, cp / G) * P.rows + row) * G + cp % G) * 32 + (c & 31) : 0;
        V* up = u + at;
        V* ep = ev + at;
        // mailbox entry (every lane of the last two planes, lane 31 of the others;
        // inside the cluster the next tile's own mailbox); its steps run out at mw
        const bool near = above && pl >= G - 2, post = (pl >= G - 2 && !above) || lane == 31;
        const unsigned peer = near ? peer_addr(own_mail + (pl - (G - 2)) * (kMail * 32) + lane, rank + 1) : 0u;
        const int mrow = back(sh.mrow - kRecAhead, P.mrows);
        int mw = Tb + P.mrows - mrow;
        typename ML::word* mb =
            mail + (group(w, dg) * P.mrows + mrow) * ME + (pl >= G - 2 ? (pl - (G - 2)) * 32 + lane : 64 + pl);
        // H == 0: c1, c2, c3 are the partial sums of T + 1, T + 2, T + 3 before this step's share
        constexpr bool kOlder = H == 0 && nterms<NS>(0) + nterms<NS>(1) + nterms<NS>(2) > 0;
        Terms<PK, NS, 3> k3;
        Terms<PK, NS, 2> k2;
        Terms<PK, NS, 1> k1;
        Terms<PK, NS, 0> k0;
        V d = V(0), c1 = V(0), c2 = V(0), c3 = V(0), b3 = V(0);
        // stages of T, T + 1, .. T + 4
        int q0 = stage_of_time(Tb - 1), q1 = next(q0), q2 = next(q1), q3 = next(q2), q4 = next(q3);
        auto fetch = [&]() {  // operands of step T + 1 that do not depend on step T
          k3.load(rec(q1));
          if (HD) d = reinterpret_cast<const V*>(rec(q1) + R::D_OFF)[0];
          if (kOlder) {
            k2.load(rec(q2));
            k1.load(rec(q3));
            k0.load(rec(q4));
            b3 = start(q4);
          } else if (H == 0) {
            c1 = start(q1);
          }
          q0 = q1;
          q1 = q2;
          q2 = q3;
          q3 = q4;
          q4 = next(q4);
        };
        fetch();
        // Steps between two turns of the stored steps.  Two forms, with and without
        // weight and emit: with one form for both the ILU(0) solves with helpers, two
        // planes, took 0.40 / 0.47 ms at 128^3 instead of 0.375 / 0.41.
        auto run = [&](auto full) {
          constexpr bool kFull = decltype(full)::value;
          auto step = [&](int T) {
            step_barrier<(NC + 1) * 32>();
            const bool ok = (unsigned)(T - koff) < nk;
            V a = k3.add(H ? cell(2, T) : c1, rb, T);
            if (PK == KBF) {
              a = mul_rn(V(reinterpret_cast<const float*>(rec(q0) + R::S_OFF)[0]), a);
              a = vec(q0, 0) - a;
            }
            V r = a;
            if (HD) r = a * d;
            if (kFull && P.relax) r = P.relax == 1 ? wv * r : fma(wv, r, mul_rn(V(1) - wv, vec(q0, ooff)));
            own[(T & (kRing - 1)) * kLanes] = ok ? r : V(0);
            if (kTurn) asm volatile("bar.arrive 2, %0;" ::"n"(G * 64) : "memory");
            if (ok) {
              if (near)
                ML::put_peer(peer + (T & (kMail - 1)) * (32 * (unsigned)sizeof(typename ML::word)), r, (unsigned)T + 1u);
              if (post) ML::put(mb, r, tag);
              *up = r;
              if (kFull && ev) *ep = P.h ? a + vec(q0, hoff) : a;
            }
            up += dstep;
            if (kFull) ep += dstep;
            mb += ME;
            if (kOlder) {
              c1 = k2.add(c2, rb, T + 1);
              c2 = k1.add(c3, rb, T + 2);
              c3 = k0.add(b3, rb, T + 3);
            }
            fetch();
          };
          for (int T = Tb; T <= Te;) {
            for (const int end = min(min(tw, mw), Te + 1); T < end; ++T) step(T);
            if (T == tw) {
              up -= (long long)P.rows * dstep;
              if (kFull) ep -= (long long)P.rows * dstep;
              tw += P.rows;
            }
            if (T == mw) {
              mb -= (long long)P.mrows * ME;
              mw += P.mrows;
            }
          }
        };
        if (P.relax || ev) run(std::true_type{});
        else run(std::false_type{});
      } else if (role == 1) {
        Terms<PK, NS, 0> k;
        int q = stage_of_time(Tb + 3);
        k.load(rec(q));
        V b3 = start(q);
        for (int T = Tb; T <= Te; ++T) {
          step_barrier<(NC + 1) * 32>();
          hold();
          cell(0, T + 3) = k.add(b3, rb, T + 3);
          q = next(q);
          k.load(rec(q));
          b3 = start(q);
        }
      } else if (role == 2) {
        Terms<PK, NS, 1> k;
        int q = stage_of_time(Tb + 2);
        k.load(rec(q));
        for (int T = Tb; T <= Te; ++T) {
          step_barrier<(NC + 1) * 32>();
          hold();
          cell(1, T + 2) = k.add(cell(0, T + 2), rb, T + 2);
          q = next(q);
          k.load(rec(q));
        }
      } else {
        Terms<PK, NS, 2> k;
        int q = stage_of_time(Tb + 1);
        k.load(rec(q));
        for (int T = Tb; T <= Te; ++T) {
          step_barrier<(NC + 1) * 32>();
          hold();
          if (kTurn) asm volatile("bar.sync 2, %0;" ::"n"(G * 64) : "memory");
          cell(2, T + 1) = k.add(cell(1, T + 1), rb, T + 1);
          q = next(q);
          k.load(rec(q));
        }
      }
    } else if (warp == NC) {
      // ---- sync warp: every lane watches one word, one load and one vote a look.
      // Step T takes halo values up to time T - 1, records up to T + kRecAhead,
      // and the places of values that the next tile has taken.
      // At cluster scope for all (the next CTA writes taken): two loads, one for
      // each scope, took 1 to 5 % of a solve.
      const int* word = lane < 3 ? &sh.hready[lane] : lane == 3 ? &sh.rready : &sh.taken[lane & 1].v;
      const int ahead = lane < 3 ? 0 : lane == 3 ? kRecAhead + 1 : above && lane < 6 ? 1 - kMail : -kDone;
      const int most = lane == 3 ? Te + 1 : INT_MAX;
      // Once a wait has run out the remaining steps run through on what is there
      // (nothing leaves its buffers, and the error word says what came of it).
      bool drain = false;
      for (int T = T0 - kRecAhead; T <= Te; ++T) {
        const int need = min(T + ahead, most);
        unsigned iter = 0;
        while (!drain && !__all_sync(0xffffffffu, ld_acq_cluster(word) >= need)) {
          if ((++iter & 31u) != 0) continue;
          // the waits of the next tile are bounded; it leaves the error word behind
          if ((iter & 1023u) == 0 && lane == 0 && ld_relaxed(P.err) != 0) st_relaxed_cta(&sh.abort, 1);
          drain = __any_sync(0xffffffffu, ld_acq_cta(&sh.abort) != 0);
        }
        step_barrier<(NC + 1) * 32>();
        if (lane == 0) st_relaxed_cta(&sh.done, T);  // behind the barrier: the steps before have read what they need
      }
    } else if (warp < NC + 4) {
      // ---- loader warps: plane p0-2, plane p0-1 (a column per lane), and the
      // column left of the strip (lane q < G + 2: plane p0-2+q)
      const int c = warp - (NC + 1);
      constexpr int SG = 32 / G;
      constexpr int kBatch = tri_mail_batch(PK);  // time steps asked for at once
      const int pc = p0 - 2 + (c < 2 ? c : lane), Ic = c < 2 ? I : 32 * w - 1, Jc = pc - Ic;
      const bool mine = c < 2 || lane < G + 2;
      const bool okc = mine && Ic >= 0 && Ic < g.nx && Jc >= 0 && Jc < g.ny;
      // owner: the tile below, or the left strip's tiles of planes p0-2, p0-1 and of the own planes
      const int cw = c < 2 ? w : w - 1;
      const int cd = c < 2 ? dg - 1 : lane < 2 ? dg + SG - 1 : dg + SG;
      const int cg = c < 2 ? G - 2 + c : lane < 2 ? G - 2 + lane : lane - 2;
      const int e = cg >= G - 2 ? (cg - (G - 2)) * 32 + (c < 2 ? lane : 31) : 64 + cg;
      const typename ML::word* src = okc ? mail + group(cw, cd) * P.mrows * ME + e : mail;
      const bool near = c < 2 && below;
      const typename ML::word* box = own_mail + (c & 1) * (kMail * 32) + lane;
      const unsigned taken = near ? peer_addr(&sh.taken[c], rank - 1) : 0u;
      V* dst = ring + (c < 2 ? c : min(lane, G + 1)) * (kRing * kLanes) + (c < 2 ? lane + 1 : 0);
      // times at which this lane has a point to fetch
      const int t_lo = okc ? SP * pc + SL * Ic : INT_MAX, t_hi = okc ? t_lo + g.nz : INT_MIN;
      int tau = T0 - kOldest, row = back(sh.mrow - kOldest, P.mrows);  // row: its step in the mailbox
      unsigned long long t_wait = 0;
      unsigned iter = 0;
      int ask = 1;  // one step while waiting for the first, a batch once they come
      if (!__any_sync(0xffffffffu, okc)) tau = Te;
      // the tile below in this cluster: it writes to the own mailbox, a word of
      // every step at a time
      unsigned long long t_near = 0;
      while (near && tau < Te) {
        const unsigned t1 = (unsigned)tau + 1u;
        typename ML::word v = ML::value(V(0), t1);
        if (tau >= t_lo && tau < t_hi) v = ML::get_own(box + (tau & (kMail - 1)) * 32);
        // one vote on both: a lane may see a later step than its neighbour
        if (__all_sync(0xffffffffu, ML::ok(v, t1) && tau < ld_acq_cta(&sh.done) + kRing - 4)) {
          dst[(tau & (kRing - 1)) * kLanes] = ML::val(v);
          ++tau;
          __syncwarp();
          if (lane == 0) {
            st_rel_cta(&sh.hready[c], tau);
            if ((tau & 3) == 0) st_peer(taken, tau);
          }
          iter = 0;
          continue;
        }
        if ((++iter & 255u) != 0) continue;
        bool stop = false;
        if (lane == 0) {
          const unsigned long long now = globaltimer_ns();
          if (iter == 256u) t_near = now;
          else if (now - t_near > P.budget_ns) {
            atomicCAS(P.err, 0, DEV_ERR_TIMEOUT);
            stop = true;
          }
          stop = stop || ld_relaxed(P.err) != 0 || ld_acq_cta(&sh.abort) != 0;
        }
        if (__shfl_sync(0xffffffffu, stop, 0)) {
          if (lane == 0) st_rel_cta(&sh.abort, 1);
          break;
        }
      }
      while (!near && tau < Te) {
        // lane 0's view for all: the votes below need every lane
        const int n = min(P.mrows - row,
                          __shfl_sync(0xffffffffu, min(min(ld_acq_cta(&sh.done) + kRing - 4, Te) - tau, ask), 0));
        int got = 0;
        if (n > 0) {
          typename ML::word val[kBatch];
#pragma unroll
          for (int q = 0; q < kBatch; ++q) {
            val[q] = ML::value(V(0), tag);
            if (q < n && tau + q >= t_lo && tau + q < t_hi) val[q] = ML::get(src + (long long)(row + q) * ME);
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
          row = row + got == P.mrows ? 0 : row + got;
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
      if (tau >= Te && lane == 0) {
        st_rel_cta(&sh.hready[c], kDone);
        if (near) st_peer(taken, kDone);
      }
    } else if (warp == NC + 4) {
      // ---- record warp
      // one lane; consecutive stored steps of the tile are one run in every stream
      if (lane == 0) {
        const int nfill = Te - T0 + 1;
        const long long step0 = group(w, dg) * P.rows;
        const char* rec = (const char*)P.rec + step0 * (G * R::BYTES);
        const V* bv = (const V*)P.b + step0 * (G * 32);
        const V* hv = (const V*)P.h + step0 * (G * 32);
        const V* ov = (const V*)P.old + step0 * (G * 32);
        constexpr unsigned vbytes = G * 32 * sizeof(V);
        int done = T0 - kRecAhead, ch = (int)(base % (unsigned)nch), issued = 0, row = sh.row;
        for (int f = 0; f < nfill; f += C) {
          // the previous occupants of the chunk, up to time T0 + f + C - 1 - nstg, are finished
          const int free_at = T0 + f + C - 1 - nstg;
          bool stop = false;
          while (f >= nstg && done <= free_at) {
            done = ld_acq_cta(&sh.done);
            if (done > free_at) break;
            if (ld_acq_cta(&sh.abort)) {
              stop = true;
              break;
            }
            __nanosleep(20);
          }
          if (stop) break;
          const int n = min(C, nfill - f);
          unsigned long long* bar = &sh.full[ch];
          char* sr = stages + ch * (C * G * R::BYTES);
          V* sv = vecs + ch * (C * G * 32);
          mbar_expect_tx(bar, n * (unsigned)(G * R::BYTES + nvec * vbytes));
          for (int left = n; left > 0;) {  // one run, or up to the last stored step and on from the first
            const int m = min(left, P.rows - row);
            const long long at = (long long)row * (G * 32);
            bulk_copy_g2s(sr, rec + (long long)row * (G * R::BYTES), m * G * R::BYTES, bar);
            bulk_copy_g2s(sv, bv + at, m * vbytes, bar);
            if (P.h) bulk_copy_g2s(sv + hoff, hv + at, m * vbytes, bar);
            if (P.relax == 2) bulk_copy_g2s(sv + ooff, ov + at, m * vbytes, bar);
            sr += m * (G * R::BYTES);
            sv += m * (G * 32);
            left -= m;
            row = row + m == P.rows ? 0 : row + m;
          }
          ++issued;
          ch = ch + 1 == nch ? 0 : ch + 1;
        }
        // every copy has landed before the tile is left (at once, unless a wait
        // ran out and the tracker left early)
        for (int f = max(0, issued - nch); f < issued; ++f) {
          const unsigned a = base + f;
          const unsigned long long t0 = globaltimer_ns();
          while (!mbar_try_wait(&sh.full[a % nch], (a / nch) & 1u))
            if (globaltimer_ns() - t0 > kCopyWaitNs) break;
        }
      }
    } else if (lane == 0) {
      // ---- tracker warp, one lane
      bool stop = false;
      int ch = (int)(base % (unsigned)nch);
      unsigned parity = (base / (unsigned)nch) & 1u;
      for (int T = T0; T <= Te && !stop; T += C) {
        unsigned long long t0 = 0;
        while (!mbar_try_wait(&sh.full[ch], parity)) {
          if (ld_acq_cta(&sh.abort)) {
            stop = true;
            break;
          }
          // the record warp waits for the steps, the steps for the halo: only
          // a copy that is due counts against the bound
          if (T + C > ld_acq_cta(&sh.done) + nstg - 1) {
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
        if (!stop) st_rel_cta(&sh.rready, T + C);
        ch = ch + 1 == nch ? 0 : ch + 1;
        parity ^= ch == 0;
      }
    }
    base += (unsigned)((Te - T0 + C) / C);
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
cudaError_t launch_tri_kernel(int CL, const TriParams& P, cudaStream_t st) {
  using SM = TriSmem<PK, NS, HD, G, H>;
  const int nvec = 1 + (P.h != nullptr) + (P.relax == 2);
  // as many stages as fit, whole chunks of them
  constexpr int C = kChunk<NSTG>, kMaxSmem = 227 * 1024;
  TriParams Q = P;
  Q.nstg = (int)std::min<size_t>(NSTG, (kMaxSmem - SM::head - 1024) / SM::stage(nvec)) / C * C;
  const size_t smem = SM::head + Q.nstg * SM::stage(nvec);
  return launch_clusters(k_tri<PK, NS, HD, G, H, NSTG>, CL, P.nunits, tri_threads<G, H>(),
                         tri_ctas<G, H>(), smem, Q, st);
}

}  // namespace tri

// One entry per working precision, each compiled in its own translation unit.
cudaError_t tri_launch_k64(int ns, bool hd, const TriShape& t, bool helpers, const tri::TriParams& P, cudaStream_t st);
cudaError_t tri_launch_k32(int ns, bool hd, const TriShape& t, const tri::TriParams& P, cudaStream_t st);
cudaError_t tri_launch_kbf(int ns, bool hd, const TriShape& t, const tri::TriParams& P, cudaStream_t st);
