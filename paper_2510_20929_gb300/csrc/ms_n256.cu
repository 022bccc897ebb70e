// Multislice per-position pass instantiated for the 256 x 256 window.
#include "kernels_ms.cuh"
#include "launch.h"

namespace ptycho {
template cudaError_t launch_pass1_ms<256>(const MsArgs&, cudaStream_t);
template cudaError_t launch_step_ms<256>(const MsStepArgs&, cudaStream_t);
}  // namespace ptycho
