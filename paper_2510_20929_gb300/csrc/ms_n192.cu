// Multislice per-position pass instantiated for the 192 x 192 window.
#include "kernels_ms.cuh"
#include "launch.h"

namespace ptycho {
template cudaError_t launch_pass1_ms<192>(const MsArgs&, cudaStream_t);
template cudaError_t launch_step_ms<192>(const MsStepArgs&, cudaStream_t);
}  // namespace ptycho
