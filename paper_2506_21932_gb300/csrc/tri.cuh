// Layout and interface of the sheared wavefront: exact lexicographic
// triangular solves on the 7/19/27-point masks with one unknown per point
// (the ILU(0) solves and, with the inverse diagonal, both halves of a
// Gauss-Seidel sweep).  Kernel in trisolve.cuh, packing kernels in
// k_shear.cu.
//
// Shear.  In sweep coordinates (I, J, K) (mirrored for the upper solve) a
// point depends on (I-1, J+1, .), (I-1, J, .), (I-1, J-1, .), (I, J-1, .) and
// on its own column.  With P = I + J the first of these stays in the same
// P and the others lie in P-1 and P-2, so in the (I, P) plane every
// dependency points to a lower or equal I and a lower or equal P: any
// rectangle of the (I, P) plane waits for its left and its lower neighbour
// only, whereas x-planes cut into y-strips also wait for the strip on their
// right.  Point (I, P, K) runs at time T = SP*P + SL*I + K, the schedule
// SA*I + SB*J + K of shapes.cuh (SP = SB, SL = SA - SB).
//
// Streams.  A CTA works on a tile: a strip of 32 I (lane = I mod 32) and G
// consecutive P, all planes one time step at a time.  Vectors and records are
// stored in that order, tile by tile and step by step, so a step of a tile is
// one contiguous run and one bulk copy per array:
//   tile (w, d): I = 32 w + lane, P = 32 w + G d + g, SP (G - 1) + 31 SL + nz steps.
// A lane has a point in only nz of these steps, one after another, and in only
// ny of its strip's planes, so times and tiles are stored modulo nz and modulo
// groups = ceil(ny / G), and no two points meet:
//   slot = (((w * groups + d mod groups) * nz + T mod nz)*G + g)*32 + lane.
// What is left of padding is a last strip of less than 32 I, and ny rounded up to
// G.  (With a slot for every step and tile the FP64 ILU(0) hierarchy of 1024 x
// 1024 x 8 took 3,850 bytes a point and that of 2048 x 1024 x 1 23,800; now 980 in
// both.)  A row thus holds values of several steps and tiles, each lane's of one:
// a tile copies whole rows, and a lane without a point at that step does not use
// its value.  The forward stream of a level uses I = i, J = j, K = k, the
// backward stream the mirrored coordinates; a solve reads its right-hand side in
// its own stream and writes its result to either (time T of one is Tmax - T of
// the other, so all lanes and tiles reach the end of the stored steps at once).
// A record is the strictly lower coefficients in sweep order, each 32 lanes
// wide, negated (an FP64 negation in the kernel would be an FP64 instruction),
// for BF16 plain and in pairs, then the FP32 row scale (BF16), then the
// inverse diagonal (HD).  One kernel serves lower and upper solves.
#pragma once

#include "shapes.cuh"
#include "smg_internal.cuh"

template <int NS>
struct Shear {
  static constexpr int SP = Shape<NS>::SB, SL = Shape<NS>::SA - Shape<NS>::SB;
};

template <int PK, int NS, bool HD>
struct TriRec {
  using Val = typename Prec<PK>::val;
  using Vec = typename Prec<PK>::vec;
  static constexpr int EC = Shape<NS>::EC;
  static constexpr int VAL_BYTES = PK == KBF ? (EC + 1) / 2 * 128 : EC * 32 * (int)sizeof(Val);
  static constexpr int S_OFF = VAL_BYTES;  // BF16 row scale
  static constexpr int D_OFF = S_OFF + (PK == KBF ? 128 : 0);
  static constexpr int BYTES = D_OFF + (HD ? 32 * (int)sizeof(Vec) : 0);
};

// Shape of a level's streams.
struct TriShape {
  int ns, G;              // mask, planes per tile
  int CL;                 // consecutive tiles of a strip taken by one cluster
  int strips;             // strips of I
  int groups, rows;       // groups of planes stored per strip, steps stored per group
};
TriShape tri_shape(const Grid& g, int ns, int pk);
int tri_cluster(const TriShape& t, const Grid& g, int pk);  // CL of a shape

// Steps that a loader asks the mailbox for at once, and steps per group stored in it,
// no fewer (2048 x 1024 x 1 FP32: a cycle of 41 ms with one, 26 with eight).
__host__ __device__ constexpr int tri_mail_batch(int pk) { return pk == K64 ? 4 : 8; }
inline int tri_mail_rows(const TriShape& t, int pk) {
  return t.rows < tri_mail_batch(pk) ? tri_mail_batch(pk) : t.rows;
}
// Slots of a stream (values of one vector).
inline size_t tri_slots(const TriShape& t) { return (size_t)t.strips * t.groups * t.rows * t.G * 32; }
// Mailbox bytes of a level (zeroed once; shared by its solves).
size_t tri_mail_bytes(const TriShape& t, int pk);
// Bytes of all records of one solve on a level.
size_t tri_rec_bytes(const TriShape& t, int pk, bool hd);

// Whether the sheared wavefront runs a level's sweeps: one unknown per point,
// a canonical 7/19/27-point mask.
bool tri_supported(const LevelView& L);
// Whether helper warps form the older terms: FP64 (a warp issues its FP64
// instructions one per 64 cycles), not on the 7-point mask, which has no terms older
// than one step to hand over, and not with option sweep_warps = 1.
inline bool tri_helpers(int ns, int pk, int warps) { return pk == K64 && ns != 7 && warps != 1; }

// Order in which the units of CL tiles are claimed: tri_unit_count() entries
// strip << 16 | first group.
int tri_unit_count(const Grid& g, const TriShape& t);
void tri_unit_table(const Grid& g, const TriShape& t, int* out);

struct TriCall {
  const void* rec;       // records of this solve
  bool hd;               // records carry the inverse diagonal; u = (..) * d
  int dir;               // +1 lower solve (forward), -1 upper solve
  const void* b;         // right-hand side, in the solve's own stream
  const void* h;         // addend of emit, own stream, or null
  const void* old;       // old iterate, own stream (relax 2), may alias u
  void* u;               // result
  void* emit;            // null, or receives b - (lower part) u (+ h), before the diagonal
  bool flip;             // u and emit in the other direction's stream (u may alias b only without it)
  int relax;             // 0: u = r; 1: u = w r; 2: u = (1 - w) old + w r
  double w;
  int warps;             // option sweep_warps: 1 no helper warps
};
cudaError_t launch_tri(const LevelView& L, const TriShape& t, const TriCall& c, const int* tiles, void* mail,
                       SweepWs* ws, int* err, unsigned long long budget_ns, cudaStream_t st);

// Records from the FP64 ILU factors LU [n][ns] and 1/u_pp (lower: unit
// diagonal, upper with 1/u_pp), or from A and 1/a_pp (both with 1/a_pp; one
// BF16 row scale for both halves, that of the whole row).
cudaError_t launch_tri_records_ilu(const Grid& g, const TriShape& t, int pk, const double* LU, const double* udinv,
                                   void* Lrec, void* Urec, cudaStream_t st);
cudaError_t launch_tri_records_gs(const Grid& g, const TriShape& t, int pk, const double* A, const double* dinv,
                                  void* Lrec, void* Urec, cudaStream_t st);

// Vector between natural order and a stream (dir: forward or backward; vb = 8
// or 4 bytes per value); add: dst += src (into natural order only).
cudaError_t launch_shear_copy(const Grid& g, const TriShape& t, int dir, int vb, bool to_stream, const void* src,
                              void* dst, bool add, cudaStream_t st);

// Forward stream out = b - A x, x and b in natural order.
cudaError_t launch_shear_residual(const LevelView& L, const TriShape& t, const void* x, const void* b, void* out,
                                  cudaStream_t st);

// Natural order: the product of the entries after (part +1) or before (-1)
// the centre with x, or b minus it where b is given.
cudaError_t launch_half(const LevelView& L, int part, const void* x, const void* b, void* y, cudaStream_t st);

// Forward streams d0 = f - h, d1 = h from natural f, h.
cudaError_t launch_shear_split(const Grid& g, const TriShape& t, int vb, const void* f, const void* h, void* d0,
                               void* d1, cudaStream_t st);

// ---- three unknowns per point (k_btri.cu): 7-point mask, FP64 and FP32 ----------
// The same streams with three values per slot, [slot / 32][unknown][lane], and
// records of -D^-1 A for the lower blocks; the solves are for D^-1 b.
bool btri_supported(const LevelView& L);
TriShape btri_shape(const Grid& g, int pk);
size_t btri_rec_bytes(const TriShape& t, int pk);
size_t btri_mail_bytes(const TriShape& t, int pk);
cudaError_t launch_btri(const LevelView& L, const TriShape& t, const TriCall& c, const int* tiles, void* mail,
                        SweepWs* ws, int* err, unsigned long long budget_ns, cudaStream_t st);
// Records of both solves from A [n][7][3][3] and D^-1 [n][3][3] in FP64.
cudaError_t launch_btri_records(const Grid& g, const TriShape& t, int pk, const double* A, const double* dinv,
                                void* Lrec, void* Urec, cudaStream_t st);
// Vector [n][3] between natural order and a stream, times D^-1 where dinv is
// given (into the stream only).
cudaError_t launch_btri_copy(const Grid& g, const TriShape& t, int dir, int pk, bool to_stream, const void* src,
                             const void* dinv, void* dst, cudaStream_t st);
// What a sweep of direction dir leaves old: h = D^-1 (blocks after the centre
// in sweep order) x; streams c = D^-1 b - h and h (may be null), x and b in
// natural order.
cudaError_t launch_btri_half(const LevelView& L, const TriShape& t, int dir, const void* dinv, const void* x,
                             const void* b, void* c, void* h, cudaStream_t st);
