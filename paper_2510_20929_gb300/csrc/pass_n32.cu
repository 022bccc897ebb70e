// Per-position kernels instantiated for the 32 x 32 window.
#include "kernels_pair.cuh"
#include "launch.h"
#include "pass2.cuh"

namespace ptycho {

// One line of a transform per lane group (k_pass1), or packed line pairs? With
// a position or two per SM all that counts is how long one position takes, and
// k_pass1 has twice its threads. Measured on GB300, k_pass1 <- or -> packed, us
// per launch:
//   gradients, 1 mode: 8 positions 16.2 <- 18.6, 152: 16.0 <- 19.8, 256: 18.4 <- 20.1, 400: 21.4 -> 20.7
//   gradients, 4 modes: 8: 22.9 <- 26.7, 152: 23.2 <- 28.1, 200: 31.4 -> 28.5
//   gradient of a given dL/dI, 1 mode: 152: 14.1 <- 18.0, 256: 15.1 <- 18.7, 400: 18.7 = 18.7
//   forward, 1 mode: 8: 8.4 <- 9.4, 304: 8.8 <- 9.4; 4 modes: 152: 11.8 <- 12.0, 200: 14.1 -> 12.8
//   relaxed probe, 8 eigenmodes, 64: forward 11.5 <- 13.0, gradients 19.7 <- 24.4, LSQML 18.5 <- 20.1
//   LSQML, 4 modes: 152: 21.6 <- 23.6, 200: 27.5 -> 24.5; 1 mode: 152: 15.5 -> 14.8
//     (with position sums 16.4 <- 18.4)
// k_pass1 reads the intensities in pairs.
static bool one_line(const BatchArgs& a) {
  if (((uintptr_t)a.meas & 7) != 0) return false;
  const bool lsqml = a.mode == MODE_LSQML_GAUSS || a.mode == MODE_LSQML_POISSON, single = a.M == 1;
  if (lsqml) return a.nb <= sm_count() && !(single && !a.opr_U && !a.possum);
  return a.nb <= (single ? 2 : 1) * sm_count();
}

template <>
cudaError_t launch_pass1<32>(const BatchArgs& a, cudaStream_t s, int) {
  if (one_line(a)) {
    constexpr int T = Threads<32>::T;
    return a.opr_U ? launch_pass1_t<32, T, true>(a, s) : launch_pass1_t<32, T, false>(a, s);
  }
  return a.opr_U ? launch_pass1_pair<PairGeo<32>, true>(a, s) : launch_pass1_pair<PairGeo<32>, false>(a, s);
}
template cudaError_t launch_pass2<32>(const Pass2Args&, cudaStream_t, int);
}  // namespace ptycho
