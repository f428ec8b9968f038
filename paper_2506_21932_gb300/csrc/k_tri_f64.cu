// Dispatch of the sheared wavefront solves (kernel in trisolve.cuh) and the
// FP64 instantiations.
#include <algorithm>
#include <vector>

#include "trisolve.cuh"

using namespace tri;

namespace {

template <int NS>
bool canonical(const Stencil& s) {
  if (s.ns != NS) return false;
  for (int e = 0; e < NS; ++e)
    for (int d = 0; d < 3; ++d)
      if (s.off[e][d] != Shape<NS>::o(e, d)) return false;
  return true;
}

template <int NS, bool HD>
cudaError_t go(const TriShape& t, bool helpers, const TriParams& P, cudaStream_t st) {
  if constexpr (NS == 7) {
    return launch_tri_kernel<K64, NS, HD, 4, 0, 16>(t.CL, P, st);
  } else {
    if (t.G == 4)
      return helpers ? launch_tri_kernel<K64, NS, HD, 4, 3, 10>(t.CL, P, st)
                     : launch_tri_kernel<K64, NS, HD, 4, 0, 10>(t.CL, P, st);
    return helpers ? launch_tri_kernel<K64, NS, HD, 2, 3, 16>(t.CL, P, st)
                   : launch_tri_kernel<K64, NS, HD, 2, 0, 16>(t.CL, P, st);
  }
}

}  // namespace

cudaError_t tri_launch_k64(int ns, bool hd, const TriShape& t, bool helpers, const TriParams& P, cudaStream_t st) {
  if (ns == 27) return hd ? go<27, true>(t, helpers, P, st) : go<27, false>(t, helpers, P, st);
  if (ns == 19) return hd ? go<19, true>(t, helpers, P, st) : go<19, false>(t, helpers, P, st);
  return hd ? go<7, true>(t, helpers, P, st) : go<7, false>(t, helpers, P, st);
}

// Planes per tile.  More planes mean fewer hops between tiles and more work per
// SM, but a longer step.  Lower / upper solve in ms, FP64 27-point:
//   G = 2: 0.44 / 0.47 at 128^3, 1.34 / 1.52 at 256^3
//   G = 4: 0.62 / 0.69           1.13 / 1.22
// (four planes fill the SM's FP64 pipe; they pay once the tiles outnumber the
// SMs), FP32 27-point with 4 and 8 planes: 0.23 and 0.26 at 128^3, 0.53 and 0.58
// at 256^3, 1.09 and 1.03 at 384^3.  BF16: 4 against 8 0.245 and 0.266 at
// 104 x 72 x 88.  The 7-point mask has a short step whatever the precision.
static int planes_per_tile(const Grid& g, int ns, int pk) {
  const long long plane = (long long)g.nx * g.ny;
  if (ns == 7) return 4;
  if (pk == K64) return plane > 192 * 192 ? 4 : 2;
  return pk == K32 && plane > 320 * 320 ? 8 : 4;
}

static int strip_tiles(const Grid& g, const TriShape& t, int w) {
  return (g.ny + std::min(32, g.nx - 32 * w) - 1 + t.G - 1) / t.G;
}

// Tiles per cluster (a divisor of 32 / G).  A hop inside a cluster takes 0.45
// us, between clusters 1.1, but clusters of eight leave some SMs idle, which
// costs more once there are several tiles per SM.  Lower solve in ms with 2, 4,
// 8 tiles per cluster:
//   BF16 27-point 192^3 (336 tiles) 0.489 0.428 0.405    384^3 (1248) 1.09 0.96
//   FP64  7-point 128^3 (160)       0.204 0.179 0.167    256^3 (576)  0.68 0.68 0.80
//   FP64 27-point 128^3 (320)       0.497 0.452 0.438    192^3 (672)  0.84 0.82 0.90
//                 320^3 (880)       1.75  1.82           384^3 (1248) 2.56 2.70 3.53
int tri_cluster(const TriShape& t, const Grid& g, int pk) {
  int n = 0;
  for (int w = 0; w < t.strips; ++w) n += strip_tiles(g, t, w);
  const int c = n <= 340 ? 8 : pk == K64 && t.ns != 7 && t.G == 4 && n > 600 ? 2 : 4;
  return std::min(c, 32 / t.G);
}

TriShape tri_shape(const Grid& g, int ns, int pk) {
  TriShape t;
  t.ns = ns;
  t.G = planes_per_tile(g, ns, pk);
  t.strips = (g.nx + 31) / 32;
  t.groups = (g.ny + t.G - 1) / t.G;
  t.rows = g.nz;
  t.CL = tri_cluster(t, g, pk);
  return t;
}

bool tri_supported(const LevelView& L) {
  return L.B == 1 && (canonical<27>(L.s) || canonical<19>(L.s) || canonical<7>(L.s));
}

size_t tri_mail_bytes(const TriShape& t, int pk) {
  const size_t word = pk == K64 ? 16 : 8;
  return word * (size_t)t.strips * t.groups * tri_mail_rows(t, pk) * (64 + std::max(0, t.G - 2));
}

size_t tri_rec_bytes(const TriShape& t, int pk, bool hd) {
  const int ns = t.ns;
#define RB_(PK, NS) (hd ? TriRec<PK, NS, true>::BYTES : TriRec<PK, NS, false>::BYTES)
#define RN_(PK) (ns == 27 ? RB_(PK, 27) : ns == 19 ? RB_(PK, 19) : RB_(PK, 7))
  const size_t b = pk == K64 ? RN_(K64) : pk == K32 ? RN_(K32) : RN_(KBF);
#undef RN_
#undef RB_
  return b * (tri_slots(t) / 32);
}

int tri_unit_count(const Grid& g, const TriShape& t) {
  int n = 0;
  for (int w = 0; w < t.strips; ++w) n += (strip_tiles(g, t, w) + t.CL - 1) / t.CL;
  return n;
}

// Units by the time of their first step, 32 (SP + SL) w + SP G d, the lower
// strip first: every unit comes after the ones its tiles wait for (CL divides
// 32 / G, so what a unit reads of the strip on its left is in two units).
void tri_unit_table(const Grid& g, const TriShape& t, int* out) {
  const int SA = t.ns == 27 ? Shape<27>::SA : t.ns == 19 ? Shape<19>::SA : Shape<7>::SA;
  const int SB = t.ns == 27 ? Shape<27>::SB : t.ns == 19 ? Shape<19>::SB : Shape<7>::SB;
  struct T {
    int t0, w, d;
  };
  std::vector<T> v;
  for (int w = 0; w < t.strips; ++w)
    for (int d = 0; d < strip_tiles(g, t, w); d += t.CL) v.push_back({32 * SA * w + SB * t.G * d, w, d});
  std::sort(v.begin(), v.end(), [](const T& a, const T& b) { return a.t0 != b.t0 ? a.t0 < b.t0 : a.w < b.w; });
  for (size_t q = 0; q < v.size(); ++q) out[q] = v[q].w << 16 | v[q].d;
}

cudaError_t launch_tri(const LevelView& L, const TriShape& t, const TriCall& c, const int* tiles, void* mail,
                       SweepWs* ws, int* err, unsigned long long budget_ns, cudaStream_t st) {
  TriParams P;
  P.g = L.g;
  P.nunits = tri_unit_count(L.g, t);
  P.ngrp = t.groups;
  P.rows = t.rows;
  P.mrows = tri_mail_rows(t, L.pk);
  const int SA = t.ns == 27 ? Shape<27>::SA : t.ns == 19 ? Shape<19>::SA : Shape<7>::SA;
  const int SB = t.ns == 27 ? Shape<27>::SB : t.ns == 19 ? Shape<19>::SB : Shape<7>::SB;
  P.last_row = (SA * (L.g.nx - 1) + SB * (L.g.ny - 1) + L.g.nz - 1) % t.rows;
  P.tiles = tiles;
  P.flip = c.flip;
  P.budget_ns = budget_ns;
  P.rec = c.rec;
  P.b = c.b;
  P.h = c.h;
  P.old = c.old;
  P.u = c.u;
  P.emit = c.emit;
  P.relax = c.relax;
  P.w = c.w;
  P.mail = mail;
  P.ws = ws;
  P.err = err;
  cudaError_t e;
  if (L.pk == K64) e = tri_launch_k64(t.ns, c.hd, t, tri_helpers(t.ns, L.pk, c.warps), P, st);
  else if (L.pk == K32) e = tri_launch_k32(t.ns, c.hd, t, P, st);
  else e = tri_launch_kbf(t.ns, c.hd, t, P, st);
  if (e == cudaSuccess) smg_count_launch(1);
  return e;
}
