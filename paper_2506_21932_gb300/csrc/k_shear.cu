// Packing kernels of the sheared wavefront (streams in tri.cuh): records,
// vectors between natural order and a stream, and residuals written to one.
// The vector kernels work on tiles of 32 lanes by 32 K of one plane of a strip:
// on the natural side a warp takes 32 consecutive K of a lane's column, on the
// stream side one row r = K + SL*lane of up to 32 lanes, through shared memory.
// Tiles cut along K rather than along r keep the natural side's warps full
// (cut along r, the residual ran 39% more warps for the same points and took
// 1.70 ms at 256^3 in FP64 where the natural-order one takes 0.82).
#include "tri.cuh"

namespace {

// One plane of a strip in a stream: w the strip, pr = P - 32 w the plane.
struct Line {
  Grid g;
  int SP, SL, G, groups, rows, dir, w, pr;
  int t0;          // time of row 0, folded
  long long base;  // first stream row of the plane
  __device__ __forceinline__ void enter(int strip, int plane) {
    w = strip;
    pr = plane;
    t0 = (SP * (32 * w + pr) + SL * 32 * w) % rows;
    base = (long long)(w * groups + pr / G % groups) * rows * G + pr % G;
  }
  // Whether lane il has a point at row r (K = r - SL il), and its natural
  // index and coordinates.
  __device__ __forceinline__ bool point(int il, int r, long long& p, int& i, int& j, int& k) const {
    const int I = 32 * w + il, J = pr - il, K = r - SL * il;
    if (I >= g.nx || J < 0 || J >= g.ny || K < 0 || K >= g.nz) return false;
    i = dir > 0 ? I : g.nx - 1 - I;
    j = dir > 0 ? J : g.ny - 1 - J;
    k = dir > 0 ? K : g.nz - 1 - K;
    p = ((long long)i * g.ny + j) * g.nz + k;
    return true;
  }
  __device__ __forceinline__ bool at(int il, int K, long long& p, int& i, int& j, int& k) const {
    return point(il, K + SL * il, p, i, j, k);
  }
  // Row q (0 <= q < KC + 31 SL) of the tile of K = k0 .. k0 + KC - 1: whether
  // lane has a point there, and its K offset kk and slot.
  template <int KC = 32>
  __device__ __forceinline__ bool slot(int lane, int k0, int q, int& kk, long long& s) const {
    kk = q - SL * lane;
    const int J = pr - lane;
    if (kk < 0 || kk >= KC || k0 + kk >= g.nz || 32 * w + lane >= g.nx || J < 0 || J >= g.ny) return false;
    s = row(k0 + q) * 32 + lane;
    return true;
  }
  // Stream row (32 slots) of row r.
  __device__ __forceinline__ long long row(int r) const {
    int f = t0 + r;
    if (f >= rows) f -= rows;
    if (f >= rows) f %= rows;  // short columns
    return base + (long long)f * G;
  }
};

// Largest magnitude of a[e0..e1) as the FP32 row scale (1 for a zero row).
__device__ __forceinline__ float row_scale(const double* a, int e0, int e1) {
  double mx = 0.0;
  for (int e = e0; e < e1; ++e) mx = fmax(mx, fabs(a[e]));
  return mx > 0.0 ? (float)mx : 1.0f;
}

// One record per warp: lane = I mod 32.  M is [n][NS] in natural order and
// entry order; dinv (HD) [n].  whole_scale: the BF16 scale covers the whole
// row of M (Gauss-Seidel), else the solve's own half (ILU).
template <int PK, int NS, bool HD>
__global__ void __launch_bounds__(256) k_records(Line ln, int whole_scale, const double* __restrict__ M,
                                                 const double* __restrict__ dinv, char* __restrict__ out) {
  using R = TriRec<PK, NS, HD>;
  using Val = typename Prec<PK>::val;
  using Vec = typename Prec<PK>::vec;
  constexpr int EC = Shape<NS>::EC;
  const int lane = threadIdx.x & 31, r = blockIdx.y * 8 + (threadIdx.x >> 5), dir = ln.dir;
  ln.enter(blockIdx.x, blockIdx.z);
  long long p;
  int i, j, k;
  if (!ln.point(lane, r, p, i, j, k)) return;
  const double* a = M + p * NS;
  char* rec = out + ln.row(r) * R::BYTES;
  if constexpr (PK == KBF) {
    const float sc = whole_scale ? row_scale(a, 0, NS) : dir > 0 ? row_scale(a, 0, EC) : row_scale(a, EC + 1, NS);
#pragma unroll
    for (int t = 0; t < (EC + 1) / 2; ++t) {
      unsigned wd = 0;
#pragma unroll
      for (int hf = 0; hf < 2; ++hf) {
        const int e = 2 * t + hf;
        if (e < EC)
          wd |= (unsigned)__bfloat16_as_ushort(__double2bfloat16(a[dir > 0 ? e : NS - 1 - e] / (double)sc)) << (16 * hf);
      }
      reinterpret_cast<unsigned*>(rec)[t * 32 + lane] = wd;
    }
    reinterpret_cast<float*>(rec + R::S_OFF)[lane] = sc;
  } else {
#pragma unroll
    for (int e = 0; e < EC; ++e) reinterpret_cast<Val*>(rec)[e * 32 + lane] = -(Val)a[dir > 0 ? e : NS - 1 - e];
  }
  if constexpr (HD) reinterpret_cast<Vec*>(rec + R::D_OFF)[lane] = (Vec)dinv[p];
}

// Tiles of KC points of 32 columns.  A row of a tile holds 32 lanes' points only
// where all their columns have one there, KC - 31 SL of KC + 31 SL rows, so a
// long tile wastes less: 27-point FP64 pack / unpack / add in ms with KC = 32, 64
// and 128 0.39 / 0.44 / 0.51, 0.31 / 0.33 / 0.40 and 0.28 / 0.31 / 0.43 at 384^3,
// 0.021 / 0.025 / 0.027, 0.019 / 0.020 / 0.025 and 0.021 / 0.023 / 0.031 at 128^3.
template <typename T, int KC>
__global__ void __launch_bounds__(256) k_shear_copy(Line ln, int to_stream, const T* __restrict__ src,
                                                    T* __restrict__ dst, int add) {
  __shared__ T t[KC][33];
  ln.enter(blockIdx.x, blockIdx.z);
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5, k0 = blockIdx.y * KC, rows = KC + 31 * ln.SL;
  long long p;
  int i, j, k, kk;
  if (to_stream) {
#pragma unroll
    for (int c = 0; c < KC / 8; ++c) {
      const int il = wp + 8 * (c & 3), kl = (c >> 2) * 32 + lane;
      if (ln.at(il, k0 + kl, p, i, j, k)) t[kl][il] = src[p];
    }
    __syncthreads();
    for (int q = wp; q < rows; q += 8)
      if (ln.template slot<KC>(lane, k0, q, kk, p)) dst[p] = t[kk][lane];
  } else {
#pragma unroll 4
    for (int q = wp; q < rows; q += 8)
      if (ln.template slot<KC>(lane, k0, q, kk, p)) t[kk][lane] = src[p];
    __syncthreads();
#pragma unroll
    for (int c = 0; c < KC / 8; ++c) {
      const int il = wp + 8 * (c & 3), kl = (c >> 2) * 32 + lane;
      if (ln.at(il, k0 + kl, p, i, j, k)) {
        const T v = t[kl][il];
        dst[p] = add ? dst[p] + v : v;
      }
    }
  }
}

// Stream out = b - A x, x and b in natural order.  A warp takes 32 points of a
// column.  Its rows of A, read lane by lane, are evicted from L1 before their
// last entry is used when too many warps do so, and too few registers keep too
// few loads in flight: residual at 384^3 in ms with 6, 8, 5, 4, 3 blocks per SM
//   FP64 3.98 5.69 3.02 2.94 3.00 (2.48 of multiply-adds).
// FP32 rows go through shared memory in whole lines (FP64 rows that way: 6.2 ms at
// 384^3), 32 KB a block on 27 points, so at most seven fit; seven or eight leave
// too few registers (256^3: 0.44 ms with 6 blocks, 0.81 with 7 or 8; without
// shared memory 0.72).  BF16 208 x 144 x 176: 0.139 with 8 blocks, 0.125 with 5.
template <int PK, int NS>
struct ResidualCfg {
  using Val = typename Prec<PK>::val;
  static constexpr bool STAGE = PK == K32;
  static constexpr int blocks = PK == K64 ? 4 : PK == K32 ? 6 : 5;  // per SM
  static constexpr size_t rows = STAGE ? sizeof(Val) * 8 * 32 * NS : 0;
};
template <int PK, int NS>
__global__ void __launch_bounds__(256, ResidualCfg<PK, NS>::blocks)
    k_shear_residual(Line ln, Stencil s, const typename Prec<PK>::val* __restrict__ A, const float* __restrict__ scale,
                     const typename Prec<PK>::vec* __restrict__ x, const typename Prec<PK>::vec* __restrict__ b,
                     typename Prec<PK>::vec* __restrict__ out) {
  using V = typename Prec<PK>::vec;
  using Val = typename Prec<PK>::val;
  __shared__ V t[32][33];
  extern __shared__ __align__(16) unsigned char rows_raw[];
  ln.enter(blockIdx.x, blockIdx.z);
  const Grid g = ln.g;
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5, k0 = blockIdx.y * 32;
  long long p;
  int i, j, k, kk;
  Val* mine = reinterpret_cast<Val*>(rows_raw) + wp * (32 * NS);
#pragma unroll 1
  for (int c = 0; c < 4; ++c) {
    const bool ok = ln.at(wp + 8 * c, k0 + lane, p, i, j, k);
    if (!__any_sync(0xffffffffu, ok)) continue;
    const Val* a = A + p * NS;
    if constexpr (ResidualCfg<PK, NS>::STAGE) {
      // forward stream: lanes are consecutive k, lane 0 of a column is on the grid
      const int n = min(32, g.nz - k0) * NS;
      const Val* run = A + __shfl_sync(0xffffffffu, p, 0) * NS;
      __syncwarp();
#pragma unroll
      for (int q = 0; q < NS; ++q)
        if (q * 32 + lane < n) mine[q * 32 + lane] = run[q * 32 + lane];
      __syncwarp();
      a = mine + lane * NS;
    }
    if (!ok) continue;
    V acc = V(0);
#pragma unroll
    for (int e = 0; e < NS; ++e) {
      const int a0 = i + Shape<NS>::o(e, 0), a1 = j + Shape<NS>::o(e, 1), a2 = k + Shape<NS>::o(e, 2);
      const bool in = (unsigned)a0 < (unsigned)g.nx && (unsigned)a1 < (unsigned)g.ny && (unsigned)a2 < (unsigned)g.nz;
      const V xv = in ? x[p + s.lin[e]] : V(0);
      acc = fma((V)to_c(a[e]), xv, acc);
    }
    if (PK == KBF) acc = __fmul_rn(scale[p], (float)acc);
    t[lane][wp + 8 * c] = b[p] - acc;
  }
  __syncthreads();
  for (int q = wp; q < 32 + 31 * ln.SL; q += 8)
    if (ln.slot(lane, k0, q, kk, p)) out[p] = t[kk][lane];
}

// Half product in natural order: the entries after (PART +1) or before (-1)
// the centre, outwards from it (the order in which the sweep that has them
// old takes them).  y = their product with x, or, given b, b minus it, the
// terms subtracted one by one.
template <int PK, int NS, int PART>
__global__ void __launch_bounds__(256) k_half(Grid g, Stencil s, const typename Prec<PK>::val* __restrict__ A,
                                              const float* __restrict__ scale,
                                              const typename Prec<PK>::vec* __restrict__ x,
                                              const typename Prec<PK>::vec* __restrict__ b,
                                              typename Prec<PK>::vec* __restrict__ y) {
  using V = typename Prec<PK>::vec;
  constexpr int EC = Shape<NS>::EC;
  const long long p = (long long)blockIdx.x * 256 + threadIdx.x;
  if (p >= g.n) return;
  const int k = (int)(p % g.nz), j = (int)((p / g.nz) % g.ny), i = (int)(p / ((long long)g.ny * g.nz));
  const typename Prec<PK>::val* a = A + p * NS;
  const bool fold = PK != KBF && b;
  V acc = fold ? b[p] : V(0);
  const V sg = fold ? V(-1) : V(1);
#pragma unroll
  for (int q = 0; q < EC; ++q) {
    const int e = PART > 0 ? EC + 1 + q : EC - 1 - q;
    const int a0 = i + Shape<NS>::o(e, 0), a1 = j + Shape<NS>::o(e, 1), a2 = k + Shape<NS>::o(e, 2);
    const bool in = (unsigned)a0 < (unsigned)g.nx && (unsigned)a1 < (unsigned)g.ny && (unsigned)a2 < (unsigned)g.nz;
    const V xv = in ? x[p + s.lin[e]] : V(0);
    acc = fma(sg * (V)to_c(a[e]), xv, acc);
  }
  if (PK == KBF) {
    acc = __fmul_rn(scale[p], (float)acc);
    if (b) acc = b[p] - acc;
  }
  y[p] = acc;
}

// Stream d0 = f - h and d1 = h.
template <typename T>
__global__ void __launch_bounds__(256) k_shear_split(Line ln, const T* __restrict__ f, const T* __restrict__ h,
                                                     T* __restrict__ d0, T* __restrict__ d1) {
  __shared__ T tf[32][33], th[32][33];
  ln.enter(blockIdx.x, blockIdx.z);
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5, k0 = blockIdx.y * 32;
  long long p;
  int i, j, k, kk;
#pragma unroll
  for (int c = 0; c < 4; ++c)
    if (ln.at(wp + 8 * c, k0 + lane, p, i, j, k)) {
      tf[lane][wp + 8 * c] = f[p];
      th[lane][wp + 8 * c] = h[p];
    }
  __syncthreads();
  for (int q = wp; q < 32 + 31 * ln.SL; q += 8)
    if (ln.slot(lane, k0, q, kk, p)) {
      const T hv = th[kk][lane];
      d0[p] = tf[kk][lane] - hv;
      d1[p] = hv;
    }
}

Line line_of(const Grid& g, const TriShape& t, int dir) {
  const int SP = t.ns == 27 ? Shear<27>::SP : t.ns == 19 ? Shear<19>::SP : Shear<7>::SP;
  const int SL = t.ns == 27 ? Shear<27>::SL : t.ns == 19 ? Shear<19>::SL : Shear<7>::SL;
  return Line{g, SP, SL, t.G, t.groups, t.rows, dir, 0, 0, 0, 0};
}

// Strips by chunks of steps by planes of a strip.
dim3 tiles(const TriShape& t, int steps, int chunk, int ny) {
  return dim3((unsigned)t.strips, (unsigned)((steps + chunk - 1) / chunk), (unsigned)(ny + 31));
}

}  // namespace

#define BY_NS(PK, F)                 \
  do {                               \
    if (ns == 27) F(PK, 27);         \
    else if (ns == 19) F(PK, 19);    \
    else F(PK, 7);                   \
  } while (0)
#define BY_PK(F)                     \
  do {                               \
    if (pk == K64) BY_NS(K64, F);    \
    else if (pk == K32) BY_NS(K32, F); \
    else BY_NS(KBF, F);              \
  } while (0)

cudaError_t launch_tri_records_ilu(const Grid& g, const TriShape& t, int pk, const double* LU, const double* udinv,
                                   void* Lrec, void* Urec, cudaStream_t st) {
  const int ns = t.ns;
  const Line f = line_of(g, t, +1), b = line_of(g, t, -1);
  const dim3 nb = tiles(t, g.nz + 31 * f.SL, 8, g.ny);
#define F_(PK, NS)                                                                    \
  do {                                                                                \
    k_records<PK, NS, false><<<nb, 256, 0, st>>>(f, 0, LU, nullptr, (char*)Lrec);     \
    k_records<PK, NS, true><<<nb, 256, 0, st>>>(b, 0, LU, udinv, (char*)Urec);        \
  } while (0)
  BY_PK(F_);
#undef F_
  smg_count_launch(2);
  return cudaGetLastError();
}

cudaError_t launch_tri_records_gs(const Grid& g, const TriShape& t, int pk, const double* A, const double* dinv,
                                  void* Lrec, void* Urec, cudaStream_t st) {
  const int ns = t.ns;
  const Line f = line_of(g, t, +1), b = line_of(g, t, -1);
  const dim3 nb = tiles(t, g.nz + 31 * f.SL, 8, g.ny);
#define F_(PK, NS)                                                                    \
  do {                                                                                \
    k_records<PK, NS, true><<<nb, 256, 0, st>>>(f, 1, A, dinv, (char*)Lrec);          \
    k_records<PK, NS, true><<<nb, 256, 0, st>>>(b, 1, A, dinv, (char*)Urec);          \
  } while (0)
  BY_PK(F_);
#undef F_
  smg_count_launch(2);
  return cudaGetLastError();
}

cudaError_t launch_shear_copy(const Grid& g, const TriShape& t, int dir, int vb, bool to_stream, const void* src,
                              void* dst, bool add, cudaStream_t st) {
  const Line ln = line_of(g, t, dir);
  constexpr int KCT = 64;
  const bool tall = ln.SL > 0 && g.nz > 32;  // SL = 0: every row is full
  const dim3 nb = tiles(t, ln.g.nz, tall ? KCT : 32, ln.g.ny);
#define C_(T)                                                                                        \
  do {                                                                                               \
    if (tall) k_shear_copy<T, KCT><<<nb, 256, 0, st>>>(ln, to_stream, (const T*)src, (T*)dst, add);  \
    else k_shear_copy<T, 32><<<nb, 256, 0, st>>>(ln, to_stream, (const T*)src, (T*)dst, add);        \
  } while (0)
  if (vb == 8) C_(double);
  else C_(float);
#undef C_
  smg_count_launch(1);
  return cudaGetLastError();
}

cudaError_t launch_shear_residual(const LevelView& L, const TriShape& t, const void* x, const void* b, void* out,
                                  cudaStream_t st) {
  const int ns = L.s.ns, pk = L.pk;
  const Line ln = line_of(L.g, t, +1);
  const dim3 nb = tiles(t, ln.g.nz, 32, ln.g.ny);
#define F_(PK, NS)                                                                                        \
  do {                                                                                                    \
    constexpr size_t sm = ResidualCfg<PK, NS>::rows;                                                     \
    const cudaError_t e =                                                                                 \
        cudaFuncSetAttribute(k_shear_residual<PK, NS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm); \
    if (e != cudaSuccess) return e;                                                                       \
    k_shear_residual<PK, NS><<<nb, 256, sm, st>>>(ln, L.s, (const Prec<PK>::val*)L.A, L.scale,            \
                                                  (const Prec<PK>::vec*)x, (const Prec<PK>::vec*)b,       \
                                                  (Prec<PK>::vec*)out);                                   \
  } while (0)
  BY_PK(F_);
#undef F_
  smg_count_launch(1);
  return cudaGetLastError();
}

cudaError_t launch_half(const LevelView& L, int part, const void* x, const void* b, void* y, cudaStream_t st) {
  const int ns = L.s.ns, pk = L.pk;
  const int nb = div_up(L.g.n, 256);
#define H_(PK, NS, PT)                                                                                         \
  k_half<PK, NS, PT><<<nb, 256, 0, st>>>(L.g, L.s, (const Prec<PK>::val*)L.A, L.scale, (const Prec<PK>::vec*)x, \
                                         (const Prec<PK>::vec*)b, (Prec<PK>::vec*)y)
#define F_(PK, NS)             \
  do {                         \
    if (part > 0) H_(PK, NS, 1); \
    else H_(PK, NS, -1);       \
  } while (0)
  BY_PK(F_);
#undef F_
#undef H_
  smg_count_launch(1);
  return cudaGetLastError();
}

cudaError_t launch_shear_split(const Grid& g, const TriShape& t, int vb, const void* f, const void* h, void* d0,
                               void* d1, cudaStream_t st) {
  const Line ln = line_of(g, t, +1);
  const dim3 nb = tiles(t, ln.g.nz, 32, ln.g.ny);
  if (vb == 8)
    k_shear_split<double><<<nb, 256, 0, st>>>(ln, (const double*)f, (const double*)h, (double*)d0, (double*)d1);
  else
    k_shear_split<float><<<nb, 256, 0, st>>>(ln, (const float*)f, (const float*)h, (float*)d0, (float*)d1);
  smg_count_launch(1);
  return cudaGetLastError();
}
