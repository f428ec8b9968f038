// Dense inverse of the coarsest level: in-place Gauss-Jordan elimination with
// partial pivoting, in blocks of kNb columns.
//
// What bounds it: n^3 FP64 FMAs on the whole chip, and n pivot searches one
// after another.  Column by column (two grid barriers each, the whole matrix
// through L2) a pivot took 17 us at n = 840 and 36 us at n = 2048: 14.9 and
// 73.9 ms.  In blocks the searches only see a panel of kNb columns:
//  (1) k_panel, one cluster of 8 CTAs: the panel's rows in shared memory, one
//      cluster barrier per column.  Every CTA offers its best row and that
//      row's values; all take the largest (the lowest row among equals) and
//      run one in-place Gauss-Jordan step on their rows.  The result is
//      N = [D^-1; -E D^-1] for the pivot block D and the other rows E;
//  (2) k_gather: W = the pivot rows of the other columns, and the rows that
//      lose their place to a pivot moved to the vacated ones;
//  (3) k_update, all SMs: A = A + N W (pivot rows: N W alone).
// The rows end up as those of the inverse of P A; k_unpermute undoes P on the
// columns.  Measured: a set-up with n = 2048 went from 76 to 29.5 ms, with
// n = 840 from 36.5 to 28.6 ms; with candidates compared as integers and pushed
// to the peers before the barrier, and one division a CTA, n = 2048 to 26.9.
// What is left is the panels' chain, 4 us a column: a search, a cluster barrier,
// a division and a step over the panel.
#include <cooperative_groups.h>

#include <algorithm>

#include "smg_internal.cuh"

namespace cg = cooperative_groups;

namespace {

constexpr int kNb = 16;       // columns of a panel
constexpr int kCluster = 8;   // CTAs of a panel
constexpr int kThreads = 256;
constexpr int kTi = 32, kTj = 64;  // tile of the update

// Row moves of a block: pivot row of each column, and the displaced rows with
// the places they move to.
struct Moves {
  int piv[kNb];
  int count;
  int from[kNb], to[kNb];
};

// Pivot candidates are compared as integers (the bits of |v| order like |v|; a
// comparison of doubles takes the FP64 pipe 64 cycles a warp): larger first, the
// lower row among equals.  NaN is no candidate.
__device__ __forceinline__ long long pivot_key(double v) {
  const long long k = __double_as_longlong(v) & 0x7fffffffffffffffLL;
  return k > 0x7ff0000000000000LL ? -1 : k;
}
__device__ __forceinline__ void better(long long& v, int& r, long long v2, int r2) {
  if (v2 > v || (v2 == v && r2 < r)) {
    v = v2;
    r = r2;
  }
}
template <int W>
__device__ __forceinline__ void best_of(long long& v, int& r) {  // of W neighbouring lanes
#pragma unroll
  for (int o = W / 2; o > 0; o >>= 1) {
    const long long v2 = __shfl_xor_sync(0xffffffffu, v, o);
    const int r2 = __shfl_xor_sync(0xffffffffu, r, o);
    better(v, r, v2, r2);
  }
}

__global__ void __launch_bounds__(kThreads) k_panel(int n, int k0, double* __restrict__ M, Moves* moves,
                                                    int* __restrict__ perm, int* err) {
  extern __shared__ double a[];  // [rows of this CTA][kNb + 1]
  constexpr int LD = kNb + 1, kWarps = kThreads / 32;
  // every CTA's candidate of a column: its key, row and values, written by its owner
  __shared__ long long c_key[2][kCluster];
  __shared__ int c_idx[2][kCluster];
  __shared__ double c_row[2][kCluster][kNb];
  __shared__ long long w_key[kWarps];
  __shared__ int w_idx[kWarps];
  __shared__ double prow[kNb], pinv;
  __shared__ int pivot;
  __shared__ Moves mv;
  cg::cluster_group cl = cg::this_cluster();
  const int rank = (int)cl.block_rank(), tid = threadIdx.x, lane = tid & 31, wp = tid >> 5;
  const int nb = min(kNb, n - k0);
  const int per = (n + kCluster - 1) / kCluster, r0 = rank * per, rows = max(0, min(n, r0 + per) - r0);
  unsigned char* used = reinterpret_cast<unsigned char*>(a + (size_t)per * LD);  // pivot row of this block
  for (int q = tid; q < rows * kNb; q += kThreads) {
    const int r = q / kNb, c = q % kNb;
    a[r * LD + c] = c < nb ? M[(long long)(r0 + r) * n + k0 + c] : 0.0;
  }
  for (int r = tid; r < rows; r += kThreads) used[r] = 0;
  cl.sync();  // every CTA runs before its candidates are written to
  bool singular = false;
  for (int t = 0; t < nb; ++t) {
    const int buf = t & 1;
    long long bv = -1;
    int bi = n;
    for (int r = tid; r < rows; r += kThreads)
      if (r0 + r >= k0 && !used[r]) better(bv, bi, pivot_key(a[r * LD + t]), r0 + r);
    best_of<32>(bv, bi);
    if (lane == 0) {
      w_key[wp] = bv;
      w_idx[wp] = bi;
    }
    __syncthreads();
    if (wp == 0) {
      bv = w_key[lane % kWarps];
      bi = w_idx[lane % kWarps];
      best_of<kWarps>(bv, bi);  // the same in every lane
      // to every CTA of the cluster, two at a time
#pragma unroll
      for (int h = 0; h < kCluster; h += 2) {
        const int to = h + lane / kNb, c = lane % kNb;
        cl.map_shared_rank(&c_row[buf][rank][0], to)[c] = bi < n ? a[(bi - r0) * LD + c] : 0.0;
      }
      if (lane < kCluster) {
        *cl.map_shared_rank(&c_key[buf][rank], lane) = bv;
        *cl.map_shared_rank(&c_idx[buf][rank], lane) = bi;
      }
    }
    cl.sync();
    if (wp == 0) {
      bv = c_key[buf][lane % kCluster];
      bi = c_idx[buf][lane % kCluster];
      best_of<kCluster>(bv, bi);
      if (bv > 0) {
        const double* pr = c_row[buf][bi / per];
        if (lane < kNb) prow[lane] = pr[lane];
        const double inv = 1.0 / pr[t];
        if (lane == 0) pinv = inv;
      }
      if (lane == 0) {
        pivot = bv > 0 ? bi : -1;
        mv.piv[t] = bi;
      }
    }
    __syncthreads();
    const int p = pivot;
    if (p < 0) {  // the same in every CTA
      singular = true;
      break;
    }
    const double inv = pinv;
    for (int r = tid; r < rows; r += kThreads) {
      double* row = a + r * LD;
      if (r0 + r == p) {
#pragma unroll
        for (int c = 0; c < kNb; ++c) row[c] = c == t ? inv : prow[c] * inv;
        used[r] = 1;
      } else {
        const double f = -row[t] * inv;
#pragma unroll
        for (int c = 0; c < kNb; ++c) row[c] = c == t ? f : fma(f, prow[c], row[c]);
      }
    }
    __syncthreads();
  }
  cl.sync();
  if (singular) {
    if (rank == 0 && tid == 0) atomicCAS(err, 0, SMG_EBREAKDOWN);
    return;
  }
  if (tid == 0) {
    // rows of the block that were not chosen move to the places of chosen
    // rows from outside it
    int m = 0, v = 0;
    for (int q = 0; q < nb; ++q) {
      bool chosen = false;
      for (int t = 0; t < nb; ++t) chosen |= mv.piv[t] == k0 + q;
      if (!chosen) mv.from[m++] = k0 + q;
      if (mv.piv[q] >= k0 + nb) mv.to[v++] = mv.piv[q];
    }
    mv.count = m;
  }
  __syncthreads();
  for (int q = tid; q < rows * kNb; q += kThreads) {
    const int r = q / kNb, c = q % kNb;
    if (c >= nb) continue;
    int at = r0 + r;
    for (int t = 0; t < nb; ++t)
      if (mv.piv[t] == r0 + r) at = k0 + t;
    for (int t = 0; t < mv.count; ++t)
      if (mv.from[t] == r0 + r) at = mv.to[t];
    M[(long long)at * n + k0 + c] = a[r * LD + c];
  }
  if (rank == 0 && tid == 0) {
    int pv[kNb], fr[kNb];
    for (int t = 0; t < nb; ++t) pv[t] = perm[mv.piv[t]];
    for (int t = 0; t < mv.count; ++t) fr[t] = perm[mv.from[t]];
    for (int t = 0; t < nb; ++t) perm[k0 + t] = pv[t];
    for (int t = 0; t < mv.count; ++t) perm[mv.to[t]] = fr[t];
    *moves = mv;
  }
}

// Columns outside the panel: W[t] = pivot row t, displaced rows moved.
__global__ void __launch_bounds__(64) k_gather(int n, int k0, double* __restrict__ M, const Moves* __restrict__ moves,
                                               double* __restrict__ W, const int* __restrict__ err) {
  __shared__ Moves mv;
  if (*err) return;
  for (int q = threadIdx.x; q < (int)(sizeof(Moves) / sizeof(int)); q += 64)
    reinterpret_cast<int*>(&mv)[q] = reinterpret_cast<const int*>(moves)[q];
  __syncthreads();
  const int c = blockIdx.x * 64 + threadIdx.x, nb = min(kNb, n - k0);
  if (c >= n || (c >= k0 && c < k0 + nb)) return;
  double w[kNb], d[kNb];
#pragma unroll
  for (int t = 0; t < kNb; ++t) {
    w[t] = t < nb ? M[(long long)mv.piv[t] * n + c] : 0.0;
    d[t] = t < mv.count ? M[(long long)mv.from[t] * n + c] : 0.0;
  }
#pragma unroll
  for (int t = 0; t < kNb; ++t) {
    W[(long long)t * n + c] = w[t];
    if (t < mv.count) M[(long long)mv.to[t] * n + c] = d[t];
  }
}

// Columns outside the panel: A[i][c] = (i in the block ? 0 : A[i][c]) +
// sum_t N[i][t] W[t][c], N the panel's columns of A.  Tiles of kTi x kTj, a
// thread 2 x 4 of it.
__global__ void __launch_bounds__(kThreads) k_update(int n, int k0, double* __restrict__ M,
                                                     const double* __restrict__ W, const int* __restrict__ err) {
  __shared__ double sn[kTi][kNb + 1], sw[kNb][kTj];
  if (*err) return;
  const int nb = min(kNb, n - k0);
  const int i0 = blockIdx.y * kTi, j0 = blockIdx.x * kTj;
  for (int q = threadIdx.x; q < kTi * kNb; q += kThreads) {
    const int i = i0 + q / kNb, t = q % kNb;
    sn[q / kNb][t] = i < n && t < nb ? M[(long long)i * n + k0 + t] : 0.0;
  }
  for (int q = threadIdx.x; q < kNb * kTj; q += kThreads) {
    const int t = q / kTj, c = j0 + q % kTj;
    sw[t][q % kTj] = c < n && !(c >= k0 && c < k0 + nb) ? W[(long long)t * n + c] : 0.0;
  }
  const int tj = threadIdx.x % 16, ti = threadIdx.x / 16;  // columns tj + 16 q, rows ti + 16 p
  double acc[2][4];
#pragma unroll
  for (int p = 0; p < 2; ++p)
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int i = i0 + ti + 16 * p, c = j0 + tj + 16 * q;
      acc[p][q] = i < n && c < n && !(i >= k0 && i < k0 + nb) ? M[(long long)i * n + c] : 0.0;
    }
  __syncthreads();
#pragma unroll
  for (int t = 0; t < kNb; ++t) {
    const double n0 = sn[ti][t], n1 = sn[ti + 16][t];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const double wv = sw[t][tj + 16 * q];
      acc[0][q] = fma(n0, wv, acc[0][q]);
      acc[1][q] = fma(n1, wv, acc[1][q]);
    }
  }
#pragma unroll
  for (int p = 0; p < 2; ++p)
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int i = i0 + ti + 16 * p, c = j0 + tj + 16 * q;
      if (i < n && c < n && !(c >= k0 && c < k0 + nb)) M[(long long)i * n + c] = acc[p][q];
    }
}

__global__ void k_identity_perm(int n, int* perm) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) perm[i] = i;
}

// Minv[i][perm[j]] = M[i][j]
__global__ void k_unpermute(int n, const double* __restrict__ M, const int* __restrict__ perm,
                            double* __restrict__ Minv) {
  const long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= (long long)n * n) return;
  const long long i = q / n;
  Minv[i * n + perm[q % n]] = M[q];
}

}  // namespace

size_t dense_scratch_bytes(int n) {
  return sizeof(double) * (size_t)kNb * n + sizeof(int) * (size_t)n + sizeof(Moves) + 64;
}

cudaError_t launch_dense_inverse(int n, double* M, double* Minv, void* scratch, int* err, cudaStream_t st) {
  double* W = (double*)scratch;
  int* perm = (int*)(W + (size_t)kNb * n);
  Moves* mv = (Moves*)(perm + (n + 15) / 16 * 16);
  const int per = (n + kCluster - 1) / kCluster;
  const size_t smem = sizeof(double) * (size_t)per * (kNb + 1) + (size_t)per;
  cudaError_t e = cudaFuncSetAttribute(k_panel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  k_identity_perm<<<div_up(n, 256), 256, 0, st>>>(n, perm);
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(kCluster);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = kCluster;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  const dim3 tiles((unsigned)((n + kTj - 1) / kTj), (unsigned)((n + kTi - 1) / kTi));
  long long launches = 2;
  for (int k0 = 0; k0 < n; k0 += kNb) {
    e = cudaLaunchKernelEx(&cfg, k_panel, n, k0, M, mv, perm, err);
    if (e != cudaSuccess) return e;
    ++launches;
    if (n > kNb) {
      k_gather<<<div_up(n, 64), 64, 0, st>>>(n, k0, M, mv, W, err);
      k_update<<<tiles, kThreads, 0, st>>>(n, k0, M, W, err);
      launches += 2;
    }
  }
  k_unpermute<<<div_up((long long)n * n, 256), 256, 0, st>>>(n, M, perm, Minv);
  smg_count_launch(launches);
  return cudaGetLastError();
}
