// What the wavefront kernels with mailboxes share: shared-memory counters,
// mbarriers with bulk copies, and the mailbox words themselves.
#pragma once
#include <algorithm>

#include "smg_internal.cuh"

namespace tri {

constexpr unsigned long long kCopyWaitNs = 100ull * 1000 * 1000;  // bound on a copy in flight

__device__ __forceinline__ unsigned smem_u32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ int ld_acq_cta(const int* p) {
  int v;
  asm volatile("ld.acquire.cta.shared.s32 %0, [%1];" : "=r"(v) : "r"(smem_u32(p)) : "memory");
  return v;
}
__device__ __forceinline__ void st_rel_cta(int* p, int v) {
  asm volatile("st.release.cta.shared.s32 [%0], %1;" ::"r"(smem_u32(p)), "r"(v) : "memory");
}
__device__ __forceinline__ void st_relaxed_cta(int* p, int v) {
  asm volatile("st.relaxed.cta.shared.s32 [%0], %1;" ::"r"(smem_u32(p)), "r"(v) : "memory");
}
__device__ __forceinline__ void mbar_init(unsigned long long* bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(unsigned long long* bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(unsigned long long* bar, unsigned parity) {
  unsigned ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// The same without suspending the thread.
__device__ __forceinline__ bool mbar_test(unsigned long long* bar, unsigned parity) {
  unsigned ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ void bulk_copy_g2s(void* dst, const void* src, unsigned bytes, unsigned long long* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_u32(dst)),
               "l"(src), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}

// ---- thread-block clusters -------------------------------------------------
__device__ __forceinline__ int cluster_rank() {
  unsigned r;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return (int)r;
}
__device__ __forceinline__ int cluster_size() {
  unsigned r;
  asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
  return (int)r;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release;\nbarrier.cluster.wait.acquire;" ::: "memory");
}
// Address of p's counterpart in the shared memory of CTA rank of the cluster.
__device__ __forceinline__ unsigned peer_addr(const void* p, int rank) {
  unsigned a;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_u32(p)), "r"(rank));
  return a;
}
__device__ __forceinline__ void st_peer(unsigned a, int v) {
  asm volatile("st.relaxed.cluster.shared::cluster.s32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ int ld_peer(unsigned a) {
  int v;
  asm volatile("ld.relaxed.cluster.shared::cluster.s32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
  return v;
}
// A counter in this CTA's shared memory that a CTA of the cluster writes while
// this one runs: a type of its own, so that it is not read at CTA scope (such a
// load does not pair with a store from outside the CTA).
struct PeerCounter {
  int v;
};
// A load at cluster scope pairs with the stores of either kind of counter.
__device__ __forceinline__ int ld_acq_cluster(const int* p) {
  int v;
  asm volatile("ld.acquire.cluster.shared::cta.s32 %0, [%1];" : "=r"(v) : "r"(smem_u32(p)) : "memory");
  return v;
}

// Mailbox words, in global memory (put, get) or in the shared memory of the
// reader (put_peer, get_own).  FP64: {tag | low half, tag | high half}; FP32: tag | value.
template <typename V> struct Mail;
template <> struct Mail<double> {
  using word = ulonglong2;
  static __device__ __forceinline__ void put(word* p, double v, unsigned tag) {
    const unsigned long long t = (unsigned long long)tag << 32;
    asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(p), "l"(t | (unsigned)__double2loint(v)),
                 "l"(t | (unsigned)__double2hiint(v))
                 : "memory");
  }
  static __device__ __forceinline__ word get(const word* p) {
    word w;
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(w.x), "=l"(w.y) : "l"(p) : "memory");
    return w;
  }
  static __device__ __forceinline__ void put_peer(unsigned a, double v, unsigned tag) {
    const word w = value(v, tag);
    asm volatile("st.relaxed.cluster.shared::cluster.v2.u64 [%0], {%1, %2};" ::"r"(a), "l"(w.x), "l"(w.y) : "memory");
  }
  static __device__ __forceinline__ word get_own(const word* p) {
    word w;
    asm volatile("ld.relaxed.cluster.shared::cta.v2.u64 {%0, %1}, [%2];"
                 : "=l"(w.x), "=l"(w.y)
                 : "r"(smem_u32(p))
                 : "memory");
    return w;
  }
  static __device__ __forceinline__ word value(double v, unsigned tag) {
    const unsigned long long t = (unsigned long long)tag << 32;
    return make_ulonglong2(t | (unsigned)__double2loint(v), t | (unsigned)__double2hiint(v));
  }
  static __device__ __forceinline__ bool ok(const word& w, unsigned tag) {
    return (unsigned)(w.x >> 32) == tag && (unsigned)(w.y >> 32) == tag;
  }
  static __device__ __forceinline__ double val(const word& w) {
    return __hiloint2double((int)(unsigned)w.y, (int)(unsigned)w.x);
  }
};
template <> struct Mail<float> {
  using word = unsigned long long;
  static __device__ __forceinline__ void put(word* p, float v, unsigned tag) {
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(value(v, tag)) : "memory");
  }
  static __device__ __forceinline__ word get(const word* p) {
    word w;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(w) : "l"(p) : "memory");
    return w;
  }
  static __device__ __forceinline__ void put_peer(unsigned a, float v, unsigned tag) {
    asm volatile("st.relaxed.cluster.shared::cluster.u64 [%0], %1;" ::"r"(a), "l"(value(v, tag)) : "memory");
  }
  static __device__ __forceinline__ word get_own(const word* p) {
    word w;
    asm volatile("ld.relaxed.cluster.shared::cta.u64 %0, [%1];" : "=l"(w) : "r"(smem_u32(p)) : "memory");
    return w;
  }
  static __device__ __forceinline__ word value(float v, unsigned tag) {
    return (unsigned long long)tag << 32 | __float_as_uint(v);
  }
  static __device__ __forceinline__ bool ok(const word& w, unsigned tag) { return (unsigned)(w >> 32) == tag; }
  static __device__ __forceinline__ float val(const word& w) { return __uint_as_float((unsigned)w); }
};

// Launch in clusters of CL CTAs, one per unit of CL tiles but no more than the
// SMs hold (per: CTAs per SM the registers are cut for).  Units are claimed by
// ticket, so a cluster that finds no room waits and then finds no unit left:
// the number need not be exact, and asking the runtime for it costs more than
// the launch.
template <typename Kern, typename Params>
cudaError_t launch_clusters(Kern kern, int CL, int nunits, int threads, int per, size_t smem, const Params& P,
                            cudaStream_t st) {
  int dev = 0, nsm = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  constexpr size_t kSmSmem = 228 * 1024, kCtaSmem = 2048;  // what an SM has; a CTA's static part
  if (per * (smem + kCtaSmem) > kSmSmem) per = 1;
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = CL;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(CL * std::min(nunits, std::max(1, nsm * per / CL)));
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  e = cudaLaunchKernelEx(&cfg, kern, P);
  return e == cudaSuccess ? cudaGetLastError() : e;
}

}  // namespace tri
