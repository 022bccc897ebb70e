// Per-position kernels instantiated for the 256 x 256 window.
#include "kernels_pair.cuh"
#include "launch.h"
#include "pass2.cuh"

namespace ptycho {
template <>
cudaError_t launch_pass1<256>(const BatchArgs& a, cudaStream_t s, int) {
  return a.opr_U ? launch_pass1_pair<PairGeo<256>, true>(a, s) : launch_pass1_pair<PairGeo<256>, false>(a, s);
}
template cudaError_t launch_pass2<256>(const Pass2Args&, cudaStream_t, int);
}  // namespace ptycho
