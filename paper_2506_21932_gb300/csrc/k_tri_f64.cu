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

// Planes per tile.  More planes mean fewer tiles to hop between and, in FP64, more
// multiply-adds in flight, but a longer step.  Lower / upper solve in ms with both,
// FP64 27-point, 2 and 4 planes:
//   128^3 0.376 / 0.414  0.519 / 0.553      192^3 0.645 / 0.706  0.806 / 0.861
//   224^3 0.835 / 0.922  0.937 / 0.998      256^3 1.084 / 1.202  1.144 / 1.220
//   288^3 1.373 / 1.520  1.392 / 1.474      320^3 1.726 / 1.919  1.686 / 1.787
//   384^3 2.652 / 2.964  2.476 / 2.633      512 x 512 x 16 1.517 / 1.653  1.896 / 2.025
// Four planes fill an SM's FP64 pipe, which pays on the largest grids.  The line was
// drawn when two planes took 0.45 ms at 128^3 and 1.34 at 256^3; it now lies below
// the crossing (288^3 to 320^3, higher on flat boxes), at a cost of up to 25 % of a
// solve in between.  FP32 27-point, lower solve with 4 and 8 planes: 256^3 0.520
// 0.574, 320^3 0.751 0.773, 352^3 0.904 0.874, 384^3 1.083 1.022, 512 x 512 x 16
// 0.836 0.852, 1024 x 512 x 8 1.366 1.401: the line lies at the crossing of cubes.
// BF16: 4 against 8 0.245 and 0.266 at 104 x 72 x 88.  The 7-point mask has a short
// step whatever the precision.
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
// 8 tiles per cluster (number of tiles):
//   FP64 27-point  128^3 (320) 0.434 0.388 0.376   144^3 (432) 0.493 0.439 0.441
//                  192^3 (672) 0.698 0.642 0.705
//     four planes  208^3 (416) 0.902 0.861 0.949   256^3 (576) 1.153 1.144 1.315
//                  288^3 (720) 1.392 1.414 1.662   384^3 (1248) 2.478 2.614 3.199
//   FP32 27-point  192^3 (336) 0.410 0.366 0.348   208^3 (416) 0.453 0.403 0.402
//                  224^3 (448) 0.492 0.438 0.440   320^3 (880) 0.816 0.752 0.848
//   BF16 27-point  192^3 (336) 0.476 0.422 0.385   384^3 (1248) 1.061 0.942 0.889
//   FP64 7-point   128^3 (160) 0.224 0.200 0.186   144^3 (216) 0.260 0.228 0.232
//                  176^3 (308) 0.324 0.294 0.323   256^3 (576) 0.568 0.556 0.640
// The lines, 340 and 600 tiles, are those of the 27-point masks in FP64 and FP32,
// where both sides come to the same at 416 to 448 and 576 tiles.  BF16, whose step
// is the shortest part of a hop, stays ahead with eight throughout, and the 7-point
// mask in FP64 falls behind with eight from 240 tiles on (up to 10 %).
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
