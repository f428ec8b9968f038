// FP32 instantiations of the sheared wavefront solves (trisolve.cuh).
#include "trisolve.cuh"

using namespace tri;

namespace {

template <int NS, bool HD>
cudaError_t go(const TriParams& P, cudaStream_t st) {
  if constexpr (NS == 7) return launch_tri_kernel<K32, NS, HD, 4, 0, 16>(P, st);
  else return launch_tri_kernel<K32, NS, HD, 8, 0, 12>(P, st);
}

}  // namespace

cudaError_t tri_launch_k32(int ns, bool hd, const TriParams& P, cudaStream_t st) {
  if (ns == 27) return hd ? go<27, true>(P, st) : go<27, false>(P, st);
  if (ns == 19) return hd ? go<19, true>(P, st) : go<19, false>(P, st);
  return hd ? go<7, true>(P, st) : go<7, false>(P, st);
}
