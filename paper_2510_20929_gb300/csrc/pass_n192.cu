// Per-position kernels instantiated for the 192 x 192 window.
#include "kernels_pair.cuh"
#include "launch.h"
#include "pass2.cuh"

namespace ptycho {
template <>
cudaError_t launch_pass1<192>(const BatchArgs& a, cudaStream_t s, int) {
  return a.opr_U ? launch_pass1_pair<PairGeo<192>, true>(a, s) : launch_pass1_pair<PairGeo<192>, false>(a, s);
}
template cudaError_t launch_pass2<192>(const Pass2Args&, cudaStream_t, int);
}  // namespace ptycho
