// Per-position kernels instantiated for the 64 x 64 window.
#include "kernels_pair.cuh"
#include "launch.h"
#include "pass2.cuh"

namespace ptycho {
template <>
cudaError_t launch_pass1<64>(const BatchArgs& a, cudaStream_t s, int) {
  return a.opr_U ? launch_pass1_pair<PairGeo<64>, true>(a, s) : launch_pass1_pair<PairGeo<64>, false>(a, s);
}
template cudaError_t launch_pass2<64>(const Pass2Args&, cudaStream_t, int);
}  // namespace ptycho
