// FP32 instantiations of the sheared wavefront solves (trisolve.cuh).
#include "trisolve.cuh"

using namespace tri;

namespace {

template <int NS, bool HD>
cudaError_t go(const TriShape& t, const TriParams& P, cudaStream_t st) {
  if constexpr (NS != 7)
    if (t.G == 8) return launch_tri_kernel<K32, NS, HD, 8, 0, 12>(t.CL, P, st);
  return launch_tri_kernel<K32, NS, HD, 4, 0, 16>(t.CL, P, st);
}

}  // namespace

cudaError_t tri_launch_k32(int ns, bool hd, const TriShape& t, const TriParams& P, cudaStream_t st) {
  if (ns == 27) return hd ? go<27, true>(t, P, st) : go<27, false>(t, P, st);
  if (ns == 19) return hd ? go<19, true>(t, P, st) : go<19, false>(t, P, st);
  return hd ? go<7, true>(t, P, st) : go<7, false>(t, P, st);
}
