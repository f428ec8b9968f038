// Point-block Gauss-Seidel (three coupled unknowns per point, Sec. 4.4 with
// 3x3 blocks) on the 7-point mask as sheared wavefront solves: the tiles,
// streams, mailboxes and service warps of trisolve.cuh, for
//   u_p = c_p - sum_{e lower} (D_p^-1 A_pe) u_{p+o_e}.
// The records hold D^-1 A (formed in FP64), so a point's nine terms per unknown
// are all that a step waits for; applying D^-1 in the step would put three more
// dependent instructions and a second barrier on it.  Every neighbour is one
// step old (T = P + K): a plane has one warp per unknown, nine FMAs each.
//
// What bounds it: the chain of planes, a step and 1/G of a hop between tiles
// each (0.45 us inside a cluster, 1.1 between clusters).  A step is the nine
// dependent FMAs of a warp and the barrier; FP64 issues one warp instruction
// per 64 cycles on a sub-partition, so two warps of one sub-partition take
// 1,150 cycles.  Lower / upper solve at 128 x 128 x 64 in ms, without clusters:
//   FP64  G = 2: 0.414 / 0.412   G = 4: 0.462 / 0.463
//   FP32  G = 2: 0.265 / 0.262   G = 4: 0.203 / 0.201   G = 8: 0.224 / 0.226
// and in clusters of 8: FP64 0.291 / 0.291, FP32 0.147 / 0.146.  (One x-plane
// per CTA, operands read in the step that uses them: a V-cycle with 16 solves
// took 15.4 ms, now 2.8.)
#include <algorithm>
#include <climits>

#include "mailbox.cuh"
#include "tri.cuh"

using namespace tri;

namespace {

constexpr int kRing = 8;    // time slots of the value ring
constexpr int kMail = 8;    // time slots of the mailbox in shared memory
constexpr int kLanes = 33;  // ring row: lane -1 and the strip's 32
constexpr int kStages = 8;  // record stages
constexpr int kDone = INT_MAX / 2;
constexpr int kTerms = 27;  // coefficients of a point
__host__ __device__ constexpr int threads_of(int G) { return (3 * G + 5) * 32; }
template <typename V>
constexpr int kPlanes = sizeof(V) == 8 ? 2 : 4;  // G
// mailbox entries of a step (three words each): the last plane, lane 31 of the others
__host__ __device__ constexpr int entries_of(int G) { return 32 + G - 1; }

struct BtriParams {
  Grid g;
  int nunits, ngrp, rows;
  const int* tiles;
  int flip, relax;
  unsigned long long budget_ns;
  const void *rec, *b, *h, *old;
  void *u, *emit;
  double w;
  void* mail;
  SweepWs* ws;
  int* err;
};

struct BtriShared {
  unsigned long long full[kStages];
  int hready[2];      // plane p0 - 1, the lane left of the strip
  PeerCounter taken;  // the next tile has taken every time < taken of the last plane
  int rready, done, abort, tile;
};

template <typename V>
__host__ __device__ constexpr size_t ring_bytes(int G) {
  return (sizeof(V) * 3 * (G + 1) * kRing * kLanes + 127) / 128 * 128;
}
template <typename V>
__host__ __device__ constexpr size_t mail_bytes() {
  return sizeof(typename Mail<V>::word) * 3 * kMail * 32;
}
template <typename V>
__host__ __device__ constexpr unsigned stage_size(int G, int nvec) {
  return (unsigned)(G * 32 * sizeof(V) * (kTerms + 3 * nvec));
}

template <typename V>
__global__ void __launch_bounds__(threads_of(kPlanes<V>), 1) k_btri(BtriParams P) {
  using ML = Mail<V>;
  constexpr int G = kPlanes<V>, NC = 3 * G, kEntries = entries_of(G);
  extern __shared__ __align__(128) unsigned char dyn[];
  __shared__ BtriShared sh;
  V* ring = reinterpret_cast<V*>(dyn);  // [unknown][plane + 1][time][lane + 1]
  // the last plane of the tile below, where the same cluster has it: [time][unknown][lane]
  typename ML::word* own_mail = reinterpret_cast<typename ML::word*>(dyn + ring_bytes<V>(G));
  char* stages = reinterpret_cast<char*>(dyn) + ring_bytes<V>(G) + mail_bytes<V>();
  const int nvec = 1 + (P.h != nullptr) + (P.relax == 2);
  const int hoff = G * 96, ooff = (1 + (P.h != nullptr)) * G * 96;
  const unsigned stage_bytes = stage_size<V>(G, nvec);
  const Grid g = P.g;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  V* u = (V*)P.u;
  V* ev = (V*)P.emit;
  typename ML::word* mail = (typename ML::word*)P.mail;
  const unsigned tag = (unsigned)P.ws->epoch + 1u;
  // first stored step of group d of strip w, and the stored step of time T
  auto group = [&](int w, int d) { return (long long)(w * P.ngrp + d % P.ngrp) * P.rows; };
  auto fold = [&](int T) { return T < 0 ? P.rows - 1 : T % P.rows; };  // T >= -1
  if (threadIdx.x == 0) {
    for (int t = 0; t < kStages; ++t) mbar_init(&sh.full[t], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  unsigned base = 0;  // stage fills of the tiles before this one
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
    const bool below = rank > 0, above = rank + 1 < csize && dg + 1 < ntile;  // neighbours in the cluster
    const int p0 = 32 * w + G * dg, T0 = p0, Te = p0 + G - 1 + g.nz - 1;
    for (int t = threadIdx.x; t < 3 * (G + 1) * kRing * kLanes; t += blockDim.x) ring[t] = V(0);
    for (int t = threadIdx.x; t < 3 * kMail * 32; t += blockDim.x) own_mail[t] = ML::value(V(0), 0);  // tags: time + 1
    if (threadIdx.x == 0) {
      sh.hready[0] = sh.hready[1] = T0 - 1;
      sh.rready = T0;
      sh.done = T0 - 1;
      sh.abort = 0;
      sh.taken.v = T0;
    }
    cluster_sync();
    if (dg >= ntile) continue;  // a unit may end early
    const int I = 32 * w + lane;
    if (warp < NC) {
      // ---- compute warps: unknown q of plane pl
      const int q = warp / G, pl = warp % G;
      const int p = p0 + pl, J = p - I;
      const bool colok = I < g.nx && J >= 0 && J < g.ny;
      auto stage = [&](int T) { return stages + ((unsigned)(base + T - T0) % kStages) * stage_bytes; };
      auto vec_of = [&](int T, int which) {
        return reinterpret_cast<const V*>(stage(T)) + G * 32 * kTerms + which + pl * 96 + q * 32 + lane;
      };
      // The lane's results: column (rc, rp) of the result's stream, whose time is T
      // or (mirrored) Tm - T; the stored steps run out at time tw (mailbox: mw).
      int rc = I, rp = p, row = fold(T0 - 1), tw = T0 - 1 + P.rows - row;
      const int dstep = P.flip ? -G * 96 : G * 96, mrow = row;
      int mw = tw;
      if (P.flip) {
        rc = g.nx - 1 - I;
        rp = g.nx + g.ny - 2 - p;
        row = fold(g.nx + g.ny - 2 + g.nz - T0);
        tw = T0 + row;
      }
      const int cw = rc >> 5, cp = rp - 32 * cw;
      const long long at = colok ? ((group(cw, cp / G) + row) * G + cp % G) * 96 + (rc & 31) + 32 * q : 0;
      V* up = u + at;
      V* ep = ev + at;
      // every lane of the last plane, lane 31 of the others; inside the cluster
      // the next tile's own mailbox
      const bool near = above && pl == G - 1, post = (pl == G - 1 && !above) || lane == 31;
      const unsigned peer = near ? peer_addr(own_mail + q * 32 + lane, rank + 1) : 0u;
      typename ML::word* mb = mail + ((group(w, dg) + mrow) * kEntries + (pl == G - 1 ? lane : 32 + pl)) * 3 + q;
      const V wv = (V)P.w;
      // operands in the ring at time T - 1: (I-1, P-1), (I, P-1), (I, P), three unknowns each
      constexpr int CS = (G + 1) * kRing * kLanes;
      const V* below = ring + pl * (kRing * kLanes) + lane + 1;
      V* own = ring + (pl + 1) * (kRing * kLanes) + lane + 1;
      V c[9], b1 = V(0);
      auto fetch = [&](int T) {
        const V* r = reinterpret_cast<const V*>(stage(T)) + pl * 32 * kTerms + 9 * q * 32 + lane;
#pragma unroll
        for (int t = 0; t < 9; ++t) c[t] = r[t * 32];
        b1 = *vec_of(T, 0);
      };
      const int Tb = T0 - 1;
      fetch(Tb);
      auto step = [&](int T) {
        asm volatile("bar.sync 1, %0;" ::"n"((NC + 1) * 32) : "memory");
        const int K = T - p;
        const bool ok = colok && K >= 0 && K < g.nz;
        const int s = ((T - 1) & (kRing - 1)) * kLanes;
        V x[9];
#pragma unroll
        for (int m = 0; m < 3; ++m) {
          x[m] = below[m * CS + s - 1];
          x[3 + m] = below[m * CS + s];
          x[6 + m] = own[m * CS + s];
        }
        V a = b1;
#pragma unroll
        for (int t = 0; t < 9; ++t) a = fma(c[t], x[t], a);
        V r = a;
        if (P.relax) r = P.relax == 1 ? wv * r : fma(wv, r, (V(1) - wv) * *vec_of(T, ooff));
        own[q * CS + (T & (kRing - 1)) * kLanes] = ok ? r : V(0);
        if (ok) {
          if (near)
            ML::put_peer(peer + (T & (kMail - 1)) * (96 * (unsigned)sizeof(typename ML::word)), r, (unsigned)T + 1u);
          if (post) ML::put(mb, r, tag);
          *up = r;
          if (ev) *ep = P.h ? a + *vec_of(T, hoff) : a;
        }
        up += dstep;
        ep += dstep;
        mb += 3 * kEntries;
        fetch(T + 1);
      };
      for (int T = Tb; T <= Te;) {
        for (const int end = min(min(tw, mw), Te + 1); T < end; ++T) step(T);
        if (T == tw) {
          up -= (long long)P.rows * dstep;
          ep -= (long long)P.rows * dstep;
          tw += P.rows;
        }
        if (T == mw) {
          mb -= (long long)P.rows * (3 * kEntries);
          mw += P.rows;
        }
      }
    } else if (warp == NC) {
      // ---- sync warp (as in trisolve.cuh)
      const int* word = lane < 2 ? &sh.hready[lane] : lane == 2 ? &sh.rready : &sh.taken.v;
      const int ahead = lane < 2 ? 0 : lane == 2 ? 2 : above && lane == 3 ? 1 - kMail : -kDone;
      const int most = lane == 2 ? Te + 1 : INT_MAX;
      bool drain = false;
      for (int T = T0 - 1; T <= Te; ++T) {
        const int need = min(T + ahead, most);
        unsigned iter = 0;
        while (!drain && !__all_sync(0xffffffffu, ld_acq_cluster(word) >= need)) {
          if ((++iter & 31u) != 0) continue;
          if ((iter & 1023u) == 0 && lane == 0 && ld_relaxed(P.err) != 0) st_relaxed_cta(&sh.abort, 1);
          drain = __any_sync(0xffffffffu, ld_acq_cta(&sh.abort) != 0);
        }
        asm volatile("bar.sync 1, %0;" ::"n"((NC + 1) * 32) : "memory");
        if (lane == 0) st_relaxed_cta(&sh.done, T);
      }
    } else if (warp < NC + 3) {
      // ---- loader warps: plane p0 - 1 (a column per lane); the column left of
      // the strip (lane m < G + 1: plane p0 - 1 + m)
      const int c = warp - (NC + 1);
      constexpr int SG = 32 / G, kBatch = 2;
      const int pc = p0 - 1 + (c ? lane : 0), Ic = c ? 32 * w - 1 : I, Jc = pc - Ic;
      const bool mine = !c || lane < G + 1;
      const bool okc = mine && Ic >= 0 && Ic < g.nx && Jc >= 0 && Jc < g.ny;
      const int cw = c ? w - 1 : w;
      const int cd = !c ? dg - 1 : lane < 1 ? dg + SG - 1 : dg + SG;
      const int cg = !c || lane < 1 ? G - 1 : lane - 1;
      const int e = cg == G - 1 ? (c ? 31 : lane) : 32 + cg;
      const typename ML::word* src = okc ? mail + (group(cw, cd) * kEntries + e) * 3 : mail;
      V* dst = ring + (c ? min(lane, G) : 0) * (kRing * kLanes) + (c ? 0 : lane + 1);
      constexpr int CS = (G + 1) * kRing * kLanes;
      const int t_lo = okc ? pc : INT_MAX, t_hi = okc ? pc + g.nz : INT_MIN;
      int tau = T0 - 1, row = fold(tau);  // row: its stored step
      unsigned long long t_wait = 0;
      unsigned iter = 0;
      int ask = 1;
      if (!__any_sync(0xffffffffu, okc)) tau = Te;
      const bool near = c == 0 && below;
      const unsigned taken = near ? peer_addr(&sh.taken, rank - 1) : 0u;
      unsigned long long t_near = 0;
      while (near && tau < Te) {
        const unsigned t1 = (unsigned)tau + 1u;
        typename ML::word v[3];
#pragma unroll
        for (int r = 0; r < 3; ++r) {
          v[r] = ML::value(V(0), t1);
          if (tau >= t_lo && tau < t_hi) v[r] = ML::get_own(own_mail + ((tau & (kMail - 1)) * 3 + r) * 32 + lane);
        }
        // one vote on all: a lane may see a later step than its neighbour
        if (__all_sync(0xffffffffu, ML::ok(v[0], t1) && ML::ok(v[1], t1) && ML::ok(v[2], t1) &&
                                        tau < ld_acq_cta(&sh.done) + kRing - 1)) {
#pragma unroll
          for (int r = 0; r < 3; ++r) dst[r * CS + (tau & (kRing - 1)) * kLanes] = ML::val(v[r]);
          ++tau;
          __syncwarp();
          if (lane == 0) {
            st_rel_cta(&sh.hready[c], tau);
            if ((tau & 1) == 0) st_peer(taken, tau);
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
        const int n = min(P.rows - row,
                          __shfl_sync(0xffffffffu, min(min(ld_acq_cta(&sh.done) + kRing - 1, Te) - tau, ask), 0));
        int got = 0;
        if (n > 0) {
          typename ML::word val[kBatch][3];
#pragma unroll
          for (int m = 0; m < kBatch; ++m)
#pragma unroll
            for (int r = 0; r < 3; ++r) {
              val[m][r] = ML::value(V(0), tag);
              if (m < n && tau + m >= t_lo && tau + m < t_hi)
                val[m][r] = ML::get(src + (long long)(row + m) * (3 * kEntries) + r);
            }
#pragma unroll
          for (int m = 0; m < kBatch; ++m)
            if (m < n && got == m &&
                __all_sync(0xffffffffu, ML::ok(val[m][0], tag) && ML::ok(val[m][1], tag) && ML::ok(val[m][2], tag))) {
              if (mine)
#pragma unroll
                for (int r = 0; r < 3; ++r) dst[r * CS + ((tau + m) & (kRing - 1)) * kLanes] = ML::val(val[m][r]);
              got = m + 1;
            }
        }
        if (got > 0) {
          tau += got;
          row = row + got == P.rows ? 0 : row + got;
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
      if (tau >= Te && lane == 0) {
        st_rel_cta(&sh.hready[c], kDone);
        if (near) st_peer(taken, kDone);
      }
    } else if (warp == NC + 3) {
      // ---- record warp, one lane
      if (lane == 0) {
        const int nfill = Te - T0 + 1;
        const long long step0 = group(w, dg);
        constexpr int RL = G * 32 * kTerms, VL = G * 96;
        const V* rec = (const V*)P.rec + step0 * RL;
        const V* bv = (const V*)P.b + step0 * VL;
        const V* hv = (const V*)P.h + step0 * VL;
        const V* ov = (const V*)P.old + step0 * VL;
        int done = T0 - 1, issued = 0, row = fold(T0);
        for (int f = 0; f < nfill; ++f) {
          const int T = T0 + f;
          bool stop = false;
          while (f >= kStages && done <= T - kStages) {
            done = ld_acq_cta(&sh.done);
            if (done > T - kStages) break;
            if (ld_acq_cta(&sh.abort)) {
              stop = true;
              break;
            }
            __nanosleep(20);
          }
          if (stop) break;
          unsigned long long* bar = &sh.full[(base + f) % kStages];
          V* st = reinterpret_cast<V*>(stages + ((base + f) % kStages) * stage_bytes);
          mbar_expect_tx(bar, stage_bytes);
          bulk_copy_g2s(st, rec + (long long)row * RL, RL * sizeof(V), bar);
          bulk_copy_g2s(st + RL, bv + (long long)row * VL, VL * sizeof(V), bar);
          if (P.h) bulk_copy_g2s(st + RL + hoff, hv + (long long)row * VL, VL * sizeof(V), bar);
          if (P.relax == 2) bulk_copy_g2s(st + RL + ooff, ov + (long long)row * VL, VL * sizeof(V), bar);
          row = row + 1 == P.rows ? 0 : row + 1;
          issued = f + 1;
        }
        // every copy has landed before the tile is left
        for (int f = max(0, issued - kStages); f < issued; ++f) {
          const unsigned a = base + f;
          const unsigned long long t0 = globaltimer_ns();
          while (!mbar_try_wait(&sh.full[a % kStages], (a / kStages) & 1u))
            if (globaltimer_ns() - t0 > kCopyWaitNs) break;
        }
      }
    } else if (lane == 0) {
      // ---- tracker warp, one lane
      bool stop = false;
      for (int T = T0; T <= Te && !stop; ++T) {
        const unsigned f = base + (T - T0);
        unsigned long long t0 = 0;
        while (!mbar_try_wait(&sh.full[f % kStages], (f / kStages) & 1u)) {
          if (ld_acq_cta(&sh.abort)) {
            stop = true;
            break;
          }
          // only a copy that is due counts against the bound
          if (T > ld_acq_cta(&sh.done) + kStages - 2) {
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

// ---- packing -----------------------------------------------------------------

// Point of lane il and row r (r = K) of plane pr of strip w, direction dir.
struct BLine {
  Grid g;
  int G, groups, rows, dir, w, pr;
  int t0;          // time of K = 0, folded
  long long base;  // first stream row of the plane
  __device__ __forceinline__ void enter(int strip, int plane) {
    w = strip;
    pr = plane;
    t0 = (32 * w + pr) % rows;
    base = (long long)(w * groups + pr / G % groups) * rows * G + pr % G;
  }
  __device__ __forceinline__ bool point(int il, int K, long long& p) const {
    const int I = 32 * w + il, J = pr - il;
    if (I >= g.nx || J < 0 || J >= g.ny || K >= g.nz) return false;
    const int i = dir > 0 ? I : g.nx - 1 - I, j = dir > 0 ? J : g.ny - 1 - J, k = dir > 0 ? K : g.nz - 1 - K;
    p = ((long long)i * g.ny + j) * g.nz + k;
    return true;
  }
  __device__ __forceinline__ long long row(int K) const {
    const int f = t0 + K;
    return base + (long long)(f < rows ? f : f - rows) * G;
  }
};

// Records -D^-1 A_e of the lower blocks in sweep order: [unknown][e][column].
template <typename V>
__global__ void __launch_bounds__(256) k_brecords(BLine ln, const double* __restrict__ A,
                                                  const double* __restrict__ dinv, V* __restrict__ rec) {
  ln.enter(blockIdx.x, blockIdx.z);
  const int lane = threadIdx.x & 31, K = blockIdx.y * 8 + (threadIdx.x >> 5);
  long long p;
  if (!ln.point(lane, K, p)) return;
  V* r = rec + ln.row(K) * (32 * kTerms) + lane;
  const double* D = dinv + p * 9;
  // the sweep's (I-1, J), (I, J-1), (.., K-1); in the stream's order of operands:
  // lane - 1 of plane P - 1, the same lane of P - 1, the own column
  for (int e = 0; e < 3; ++e) {
    const double* a = A + (p * 7 + (ln.dir > 0 ? e : 6 - e)) * 9;
    for (int q = 0; q < 3; ++q)
      for (int c = 0; c < 3; ++c)
        r[((q * 3 + e) * 3 + c) * 32] = (V)(-(D[q * 3] * a[c] + D[q * 3 + 1] * a[3 + c] + D[q * 3 + 2] * a[6 + c]));
  }
}

// Natural vector [n][3] to a stream (times D^-1 if given) and back.
template <typename V>
__global__ void __launch_bounds__(256) k_bcopy(BLine ln, int to_stream, const V* __restrict__ src,
                                               const V* __restrict__ dinv, V* __restrict__ dst) {
  __shared__ V t[3][32][33];
  ln.enter(blockIdx.x, blockIdx.z);
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5, k0 = blockIdx.y * 32;
  long long p;
  if (to_stream) {
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const int il = wp + 8 * c;
      if (!ln.point(il, k0 + lane, p)) continue;
      const V s0 = src[p * 3], s1 = src[p * 3 + 1], s2 = src[p * 3 + 2];
      if (dinv) {
        const V* D = dinv + p * 9;
#pragma unroll
        for (int q = 0; q < 3; ++q) t[q][lane][il] = fma(D[q * 3], s0, fma(D[q * 3 + 1], s1, D[q * 3 + 2] * s2));
      } else {
        t[0][lane][il] = s0;
        t[1][lane][il] = s1;
        t[2][lane][il] = s2;
      }
    }
    __syncthreads();
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const int kk = wp + 8 * c;
      if (!ln.point(lane, k0 + kk, p)) continue;
      V* o = dst + ln.row(k0 + kk) * 96 + lane;
#pragma unroll
      for (int q = 0; q < 3; ++q) o[q * 32] = t[q][kk][lane];
    }
  } else {
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const int kk = wp + 8 * c;
      if (!ln.point(lane, k0 + kk, p)) continue;
      const V* o = src + ln.row(k0 + kk) * 96 + lane;
#pragma unroll
      for (int q = 0; q < 3; ++q) t[q][kk][lane] = o[q * 32];
    }
    __syncthreads();
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const int il = wp + 8 * c;
      if (!ln.point(il, k0 + lane, p)) continue;
#pragma unroll
      for (int q = 0; q < 3; ++q) dst[p * 3 + q] = t[q][lane][il];
    }
  }
}

// The half of a sweep's matrix that stays old: h = D^-1 (blocks after the
// centre in sweep order) x, streams cs = D^-1 b - h and hs = h (unless null).
template <typename V>
__global__ void __launch_bounds__(256) k_bhalf(BLine ln, const V* __restrict__ A, const V* __restrict__ dinv,
                                               const V* __restrict__ x, const V* __restrict__ b, V* __restrict__ cs,
                                               V* __restrict__ hs) {
  __shared__ V t[3][32][33];
  ln.enter(blockIdx.x, blockIdx.z);
  const Grid g = ln.g;
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5, k0 = blockIdx.y * 32;
  const long long step[3] = {(long long)g.ny * g.nz, g.nz, 1};
  V h[4][3] = {};
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    const int il = wp + 8 * c, I = 32 * ln.w + il, J = ln.pr - il, K = k0 + lane;
    long long p;
    if (!ln.point(il, K, p)) continue;
    const bool in[3] = {I + 1 < g.nx, J + 1 < g.ny, K + 1 < g.nz};
    V s0 = V(0), s1 = V(0), s2 = V(0);
#pragma unroll
    for (int m = 2; m >= 0; --m) {  // outwards from the centre: z, y, x
      if (!in[m]) continue;
      const V* a = A + (p * 7 + (ln.dir > 0 ? 6 - m : m)) * 9;
      const V* xq = x + (p + ln.dir * step[m]) * 3;
      const V x0 = xq[0], x1 = xq[1], x2 = xq[2];
      s0 = fma(a[0], x0, fma(a[1], x1, fma(a[2], x2, s0)));
      s1 = fma(a[3], x0, fma(a[4], x1, fma(a[5], x2, s1)));
      s2 = fma(a[6], x0, fma(a[7], x1, fma(a[8], x2, s2)));
    }
    const V* D = dinv + p * 9;
    const V b0 = b[p * 3], b1 = b[p * 3 + 1], b2 = b[p * 3 + 2];
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      h[c][q] = fma(D[q * 3], s0, fma(D[q * 3 + 1], s1, D[q * 3 + 2] * s2));
      t[q][lane][il] = fma(D[q * 3], b0 - s0, fma(D[q * 3 + 1], b1 - s1, D[q * 3 + 2] * (b2 - s2)));
    }
  }
  for (int pass = 0; pass < (hs ? 2 : 1); ++pass) {
    if (pass) {
      __syncthreads();
#pragma unroll
      for (int c = 0; c < 4; ++c)
#pragma unroll
        for (int q = 0; q < 3; ++q) t[q][lane][wp + 8 * c] = h[c][q];
    }
    __syncthreads();
    V* out = pass ? hs : cs;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const int kk = wp + 8 * c;
      long long p;
      if (!ln.point(lane, k0 + kk, p)) continue;
      V* o = out + ln.row(k0 + kk) * 96 + lane;
#pragma unroll
      for (int q = 0; q < 3; ++q) o[q * 32] = t[q][kk][lane];
    }
  }
}

BLine line_of(const Grid& g, const TriShape& t, int dir) { return BLine{g, t.G, t.groups, t.rows, dir, 0, 0, 0, 0}; }

template <typename V>
cudaError_t go(int CL, const BtriParams& P, cudaStream_t st) {
  constexpr int G = kPlanes<V>;
  const int nvec = 1 + (P.h != nullptr) + (P.relax == 2);
  const size_t smem = ring_bytes<V>(G) + mail_bytes<V>() + (size_t)kStages * stage_size<V>(G, nvec);
  return launch_clusters(k_btri<V>, CL, P.nunits, threads_of(G), 1, smem, P, st);
}

}  // namespace

bool btri_supported(const LevelView& L) {
  if (L.B != 3 || L.pk == KBF || L.s.ns != 7) return false;
  for (int e = 0; e < 7; ++e)
    for (int d = 0; d < 3; ++d)
      if (L.s.off[e][d] != Shape<7>::o(e, d)) return false;
  return true;
}

TriShape btri_shape(const Grid& g, int pk) {
  TriShape t;
  t.ns = 7;
  t.G = pk == K64 ? kPlanes<double> : kPlanes<float>;
  t.strips = (g.nx + 31) / 32;
  t.groups = (g.ny + t.G - 1) / t.G;
  t.rows = g.nz;
  t.CL = tri_cluster(t, g, pk);
  return t;
}

size_t btri_rec_bytes(const TriShape& t, int pk) { return tri_slots(t) * kTerms * (pk == K64 ? 8 : 4); }
size_t btri_mail_bytes(const TriShape& t, int pk) {
  return (size_t)t.strips * t.groups * t.rows * entries_of(t.G) * 3 * (pk == K64 ? 16 : 8);
}

cudaError_t launch_btri_records(const Grid& g, const TriShape& t, int pk, const double* A, const double* dinv,
                                void* Lrec, void* Urec, cudaStream_t st) {
  const dim3 nb((unsigned)t.strips, (unsigned)((g.nz + 7) / 8), (unsigned)(g.ny + 31));
  for (int dir = 1; dir >= -1; dir -= 2) {
    void* out = dir > 0 ? Lrec : Urec;
    if (pk == K64) k_brecords<double><<<nb, 256, 0, st>>>(line_of(g, t, dir), A, dinv, (double*)out);
    else k_brecords<float><<<nb, 256, 0, st>>>(line_of(g, t, dir), A, dinv, (float*)out);
  }
  smg_count_launch(2);
  return cudaGetLastError();
}

cudaError_t launch_btri_copy(const Grid& g, const TriShape& t, int dir, int pk, bool to_stream, const void* src,
                             const void* dinv, void* dst, cudaStream_t st) {
  const dim3 nb((unsigned)t.strips, (unsigned)((g.nz + 31) / 32), (unsigned)(g.ny + 31));
  if (pk == K64)
    k_bcopy<double><<<nb, 256, 0, st>>>(line_of(g, t, dir), to_stream, (const double*)src, (const double*)dinv,
                                        (double*)dst);
  else
    k_bcopy<float><<<nb, 256, 0, st>>>(line_of(g, t, dir), to_stream, (const float*)src, (const float*)dinv,
                                       (float*)dst);
  smg_count_launch(1);
  return cudaGetLastError();
}

cudaError_t launch_btri_half(const LevelView& L, const TriShape& t, int dir, const void* dinv, const void* x,
                             const void* b, void* c, void* h, cudaStream_t st) {
  const dim3 nb((unsigned)t.strips, (unsigned)((L.g.nz + 31) / 32), (unsigned)(L.g.ny + 31));
  if (L.pk == K64)
    k_bhalf<double><<<nb, 256, 0, st>>>(line_of(L.g, t, dir), (const double*)L.A, (const double*)dinv,
                                        (const double*)x, (const double*)b, (double*)c, (double*)h);
  else
    k_bhalf<float><<<nb, 256, 0, st>>>(line_of(L.g, t, dir), (const float*)L.A, (const float*)dinv, (const float*)x,
                                       (const float*)b, (float*)c, (float*)h);
  smg_count_launch(1);
  return cudaGetLastError();
}

cudaError_t launch_btri(const LevelView& L, const TriShape& t, const TriCall& c, const int* tiles, void* mail,
                        SweepWs* ws, int* err, unsigned long long budget_ns, cudaStream_t st) {
  BtriParams P;
  P.g = L.g;
  P.nunits = tri_unit_count(L.g, t);
  P.ngrp = t.groups;
  P.rows = t.rows;
  P.tiles = tiles;
  P.flip = c.flip;
  P.relax = c.relax;
  P.budget_ns = budget_ns;
  P.rec = c.rec;
  P.b = c.b;
  P.h = c.h;
  P.old = c.old;
  P.u = c.u;
  P.emit = c.emit;
  P.w = c.w;
  P.mail = mail;
  P.ws = ws;
  P.err = err;
  const cudaError_t e = L.pk == K64 ? go<double>(t.CL, P, st) : go<float>(t.CL, P, st);
  if (e == cudaSuccess) smg_count_launch(1);
  return e;
}
