// Per-scan-position kernels of the LSQML hot path (templated on the window N).
//
// k_pass1: one CTA per position of a minibatch at window 16, and at 32 while a
//   launch has few positions per SM (kernels_pair.cuh holds the other windows; its
//   line pairs leave 16 too few threads: measured equal or slower, with a relaxed
//   probe 12 -> 16 us per 256 positions). For every incoherent probe mode k it extracts the sub-pixel object patch o_j = S_j(O) (bilinear),
//   forms the exit wave psi_jk = P_k o_j (Pty-Chi Sec. 2.1, the psi = p o of
//   Eq. 2), propagates it with the unitary 2-D FFT and accumulates the
//   incoherent intensity I_j = sum_k |Psi_jk|^2 (Eq. 4's forward model). It
//   then applies the data term (Eq. 1 amplitude loss, or the Poisson
//   likelihood), forms the far-field correction factor, back-propagates every
//   mode to chi_jk = F^-1[(rho - 1) Psi_jk] (= psi'_jk - psi_jk of Eq. 2), and
//   reduces g_j = sum_k conj(P_k) chi_jk and h_jk = conj(o_j) chi_jk. Finally
//   it scatter-adds S_j^T g_j and the illumination S_j^T sum_k |P_k|^2 into the
//   object-frame accumulators (the LSQML preconditioner) with vector atomics,
//   or, in gradient mode, S_j^T of the object gradient and the position
//   gradient through the bilinear weights.
// The step-size pass is in pass2.cuh.
#pragma once
#include <cooperative_groups.h>
#include "common.cuh"
#include "tc.cuh"

namespace ptycho {
namespace cg = cooperative_groups;

// CTA sizes of k_pass1 (a thread per line slot N*R1): the default, and the
// alternative the autotuner may pick (half of it, two lines per thread).
template <int N> struct Threads;
template <> struct Threads<16> { static constexpr int T = 64, ALT = 32; };
template <> struct Threads<32> { static constexpr int T = 128; };

template <int N>
struct Pass1Smem {
  static constexpr int RP = N + 16;  // row pitch of the intensity/factor plane (floats)
  static constexpr size_t red = 0;
  static constexpr size_t tile = red + 256 * sizeof(double);
  static constexpr size_t tw = tile + (size_t)N * N * sizeof(float2);
  static constexpr size_t rI = tw + (size_t)Twiddles<N>::COUNT * sizeof(float2);
  static constexpr size_t bytes = rI + (size_t)N * RP * sizeof(float);
};

// 2-D forward transform of the tile (natural layout on entry). Column pass
// first, then rows; `out(row, v)` receives each row's unnormalised transform in
// the line "out" layout: v[m] = X[row][Fft2<N>::out_index(n, m)].
template <int N, int T, class Out>
__device__ __forceinline__ void fft2_forward(float2* tile, const float2* tw, Out&& out) {
  using F = Fft2<N>;
  constexpr int R1 = F::R1, R2 = F::R2, L = T / R1, ITER = N / L;
  const int n = F::line_lane(), gid = F::line_slot();
#pragma unroll 1
  for (int it = 0; it < ITER; ++it) {
    const int col = gid + it * L;
    float2 v[R2];
    F::template load_in<false>(v, tile, col, n);
    F::template line_fwd<false>(v, tile, col, n, tw);
    F::template store_out<false>(v, tile, col, n);
  }
  __syncthreads();
#pragma unroll 1
  for (int it = 0; it < ITER; ++it) {
    const int row = gid + it * L;
    float2 v[R2];
    F::template load_in<true>(v, tile, row, n);
    F::template line_fwd<true>(v, tile, row, n, tw);
    out(row, v);
  }
}

// 2-D inverse (unnormalised). `in(row, v)` supplies each row in the "out"
// layout; `out(col, v)` receives each column with v[n2] = x[n + R1*n2][col].
// The tile must be free on entry.
template <int N, int T, class In, class Out>
__device__ __forceinline__ void fft2_inverse(float2* tile, const float2* tw, In&& in, Out&& out) {
  using F = Fft2<N>;
  constexpr int R1 = F::R1, R2 = F::R2, L = T / R1, ITER = N / L;
  const int n = F::line_lane(), gid = F::line_slot();
#pragma unroll 1
  for (int it = 0; it < ITER; ++it) {
    const int row = gid + it * L;
    float2 v[R2];
    in(row, v);
    F::template line_inv<true>(v, tile, row, n, tw);
    F::template store_in<true>(v, tile, row, n);
  }
  __syncthreads();
#pragma unroll 1
  for (int it = 0; it < ITER; ++it) {
    const int col = gid + it * L;
    float2 v[R2];
    F::template load_out<false>(v, tile, col, n);
    F::template line_inv<false>(v, tile, col, n, tw);
    out(col, v);
  }
}

// S_j^T of a patch of LR x N pixels (the whole patch, or a band of its rows)
// onto its (LR+1) x (N+1) object tile, evaluated separably:
// h_y(x) = (1-fx) p(y, x) + fx p(y, x-1) and out(y, x) = (1-fy) h_y(x) + fy h_{y-1}(x),
// with p = 0 outside. A thread owns one of the tile columns 0 .. N-1 and a run
// of rows (lanes of a warp emit consecutive x, so the atomics coalesce; the
// runs keep every thread busy), four rows of loads in flight (one at a time
// the walk took 27,000 cycles of a 512-thread CTA at N = 128); the tile's last
// column follows, a row per thread. `load(y, x)` returns the patch value as a
// float4 (unused components zero), `emit(y, x, v)` consumes the tile value.
template <int N, int LR, int T, class Load, class Emit>
__device__ __forceinline__ void bilinear_scatter(float fy, float fx, Load&& load, Emit&& emit) {
  constexpr int L1 = LR + 1, CH = 4;
  constexpr int SEG = T / N > 0 ? T / N : (N % T != 0 && 2 * N % T == 0) ? 2 : 1;
  constexpr int RS = (L1 + SEG - 1) / SEG;
  const float gx = 1.f - fx, gy = 1.f - fy;
  const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
  auto lerp = [](float wa, float4 a, float wb, float4 b) {   // wa a + wb b
    return make_float4(fmaf(wa, a.x, wb * b.x), fmaf(wa, a.y, wb * b.y), fmaf(wa, a.z, wb * b.z),
                       fmaf(wa, a.w, wb * b.w));
  };
  for (int item = threadIdx.x; item < N * SEG; item += T) {
    const int y0 = item / N * RS, x = item % N, y1 = min(L1, y0 + RS);
    auto rowh = [&](int y) {
      return lerp(fx, (y < LR && x > 0) ? load(y, x - 1) : zero, gx, y < LR ? load(y, x) : zero);
    };
    float4 hp = y0 > 0 ? rowh(y0 - 1) : zero;
    for (int y = y0; y < y1; y += CH) {
      float4 h[CH];
#pragma unroll
      for (int c = 0; c < CH; ++c) h[c] = rowh(y + c);
#pragma unroll
      for (int c = 0; c < CH; ++c) {
        if (y + c < y1) emit(y + c, x, lerp(gy, h[c], fy, hp));
        hp = h[c];
      }
    }
  }
  for (int y = threadIdx.x; y < L1; y += T) {
    const float4 a = y < LR ? load(y, N - 1) : zero, b = y > 0 ? load(y - 1, N - 1) : zero;
    emit(y, N, lerp(gy, lerp(fx, a, 0.f, zero), fy, lerp(fx, b, 0.f, zero)));
  }
}

// The end of the per-position pass: g_j (read with getg(y, x), in shared
// memory; every thread's writes are in flight on entry) and, for LSQML, the
// probe intensity are scattered into the object frame, then the position
// gradient or the sums of the position step are reduced. The CTA holds rows
// y0 .. y0 + LR - 1 of the patch (getg's y counts from y0). `spS` is LR * N
// floats of shared memory that are free on entry. FP64_SUMS: the position
// gradient goes to a.gsum. On a cluster (the other callers with several CTAs per
// position) a position marked invalid meanwhile is left out.
template <int N, int LR, int T, bool OPR, bool FP64_SUMS = false, class Get>
__device__ __forceinline__ void overlap_add(const BatchArgs& a, int slot, int j, int y0, int ty, int tx, float fy,
                                            float fx, const float2* p0, float* spS, double* red, Get&& getg) {
  constexpr int LNN = LR * N;
  const int tid = threadIdx.x, mode = a.mode, pb = y0 * N;
  const bool lsqml = (mode == MODE_LSQML_GAUSS || mode == MODE_LSQML_POISSON);
  constexpr bool CLUSTER = N > LR && !FP64_SUMS;
  int live = 1;
  if constexpr (CLUSTER) live = *(const volatile int*)(a.valid + slot);
  // LSQML: the probe intensity sum_k |P_k|^2 of every pixel into shared memory
  // (the intensity/factor plane is free by now), so that the scatter's row walk
  // waits on shared memory rather than on L2
  if (lsqml) {
#pragma unroll 2
    for (int p = 4 * tid; p < LNN; p += 4 * T) {
      float4 v = __ldg((const float4*)(a.Sp + pb + p));
      if (OPR && p0) {
        const float4 q0 = *(const float4*)(p0 + pb + p), q1 = *(const float4*)(p0 + pb + p + 2);
        v.x += q0.x * q0.x + q0.y * q0.y; v.y += q0.z * q0.z + q0.w * q0.w;
        v.z += q1.x * q1.x + q1.y * q1.y; v.w += q1.z * q1.z + q1.w * q1.w;
      }
      *(float4*)(spS + p) = v;
    }
  }
  if constexpr (CLUSTER) {
    if (!__syncthreads_and(live)) return;
  } else {
    __syncthreads();
  }
  if (lsqml) {
    bilinear_scatter<N, LR, T>(
        fy, fx,
        [&](int y, int x) {
          const float2 g = getg(y, x);
          return make_float4(g.x, g.y, spS[y * N + x], 0.f);
        },
        [&](int y, int x, float4 v) {
          atomicAdd(a.acc + (size_t)(ty + y0 + y) * a.W + (tx + x), make_float4(v.x, v.y, v.z, 0.f));
        });
  } else {
    bilinear_scatter<N, LR, T>(
        fy, fx,
        [&](int y, int x) {
          const float2 g = getg(y, x);
          return make_float4(g.x, g.y, 0.f, 0.f);
        },
        [&](int y, int x, float4 v) {
          atomicAdd(a.gobj + (size_t)(ty + y0 + y) * a.W + (tx + x), make_float2(v.x, v.y));
        });
  }

  // ---- position gradient through the bilinear weights (gradient modes), or the
  // ---- sums of the least-squares position step (LSQML position correction)
  if (a.gpos || a.possum) {
    const bool ls = a.possum != nullptr;
    float gy = 0.f, gx = 0.f, a11 = 0.f, a12 = 0.f, a22 = 0.f;
    // four pixels' loads in flight: the smaller CTAs' threads take many each (512
    // threads gain 1 % from four and lose as much when no sums are wanted)
#pragma unroll (T < 512 ? 4 : 2)
    for (int p = tid; p < LNN; p += T) {
      const int r = p / N, c = p % N;
      const float2* o = a.obj + (size_t)(ty + y0 + r) * a.W + (tx + c);
      const float2 O00 = __ldg(o), O01 = __ldg(o + 1), O10 = __ldg(o + a.W), O11 = __ldg(o + a.W + 1);
      const float2 dy = make_float2((1.f - fx) * (O10.x - O00.x) + fx * (O11.x - O01.x),
                                    (1.f - fx) * (O10.y - O00.y) + fx * (O11.y - O01.y));
      const float2 dx = make_float2((1.f - fy) * (O01.x - O00.x) + fy * (O11.x - O10.x),
                                    (1.f - fy) * (O01.y - O00.y) + fy * (O11.y - O10.y));
      const float2 g = getg(r, c);
      gy += g.x * dy.x + g.y * dy.y;  // Re(conj(g) dy)
      gx += g.x * dx.x + g.y * dx.y;
      if (ls) {   // sum_k abs(P_k)^2 times the derivative products
        const float sp = __ldg(a.Sp + pb + p) + ((OPR && p0) ? cabs2(p0[pb + p]) : 0.f);
        a11 = fmaf(sp, cabs2(dy), a11);
        a12 = fmaf(sp, dy.x * dx.x + dy.y * dx.y, a12);
        a22 = fmaf(sp, cabs2(dx), a22);
      }
    }
    if (ls) {
      double v[5] = {(double)a11, (double)a12, (double)a22, (double)gy, (double)gx};
      block_sum<5>(v, red);
      if (tid == 0)
        for (int q = 0; q < 5; ++q) atomicAdd(a.possum + (size_t)slot * 5 + q, v[q]);
    } else {
      double v[2] = {(double)gy, (double)gx};
      block_sum<2>(v, red);
      if (tid == 0) {
        if constexpr (FP64_SUMS) {
          atomicAdd(a.gsum + 2 * slot, v[0]);
          atomicAdd(a.gsum + 2 * slot + 1, v[1]);
        } else {
          atomicAdd(a.gpos + 2 * j, (float)v[0]);
          atomicAdd(a.gpos + 2 * j + 1, (float)v[1]);
        }
      }
    }
  }
}

// OPR: the primary probe mode is synthesised per position (a separate
// instantiation, so that the shared-probe kernel carries none of it).
template <int N, int T, bool OPR>
__global__ void __launch_bounds__(T, 1) k_pass1(BatchArgs a) {
  using F = Fft2<N>;
  using SM = Pass1Smem<N>;
  constexpr int R1 = F::R1, R2 = F::R2, NN = N * N, RP = SM::RP;
  extern __shared__ __align__(16) unsigned char smem[];
  wait_prior_grid();
  double* red = (double*)(smem + SM::red);
  float2* tile = (float2*)(smem + SM::tile);
  float2* tw = (float2*)(smem + SM::tw);
  float* rI = (float*)(smem + SM::rI);

  const int slot = blockIdx.x;
  const int tid = threadIdx.x, n = F::line_lane();
  const int e = a.b0 + slot;
  const int j = a.order ? a.order[e] : e;
  int ty = 0, tx = 0;
  float fy = 0.f, fx = 0.f;
  bool ok = (j >= 0 && j < a.J);
  if (ok) ok = tile_of(a.pos[2 * j], a.pos[2 * j + 1], N, a.H, a.W, ty, tx, fy, fx);
  if (!ok) {
    if (tid == 0) {
      atomicOr(a.status, FLAG_BOUNDS);
      if (a.valid) a.valid[slot] = 0;
    }
    return;
  }
  if (tid == 0 && a.valid) a.valid[slot] = 1;
  // the measured intensities are first read by the data term, after the forward
  // transforms: fetch them into L2 meanwhile (they may live in host memory)
  if (tid == 0 && a.meas && a.mode != MODE_FWD)
    prefetch_l2_bulk(a.meas + (size_t)j * N * N, (uint32_t)(N * N * sizeof(float)));
  make_twiddles<N>(tw);

  const int M = a.M;
  const float invN = 1.0f / (float)N;
  const size_t slotNN = (size_t)slot * NN;
  float* wj = (float*)(red + 128);   // this position's eigenmode weights (OPR)
  float2* p0 = (OPR && a.p0_s) ? a.p0_s + slotNN : nullptr;
  if (OPR) {
    if (tid < a.K) wj[tid] = a.opr_w[(size_t)j * a.K + tid];
    __syncthreads();
  }
  float2* psi_s = a.psi_s ? a.psi_s + slotNN * M : nullptr;
  float2* o_s = a.o_s ? a.o_s + slotNN : nullptr;

  // ---- forward model: I_j = sum_k |F(P_k o_j)|^2 -------------------------------
#pragma unroll 1
  for (int k = 0; k < M; ++k) {
    const float2* Pk = shared_mode<OPR>(a, k, NN);
    // psi_k = P_k o_j into the tile, two adjacent pixels per thread and iteration
    const NatPairs<N, T> np;
#pragma unroll 4
    for (int q = 0; q < NatPairs<N, T>::STEPS; ++q) {
      const int r = np.row(q), c = np.c, p = np.pix(q);
      float2 o0, o1;
      if (k == 0 || !o_s) {
        bilinear2(a.obj, a.W, ty + r, tx + c, fy, fx, o0, o1);
        if (k == 0 && o_s) *(float4*)(o_s + p) = make_float4(o0.x, o0.y, o1.x, o1.y);
      } else {
        const float4 o2 = *(const float4*)(o_s + p);
        o0 = make_float2(o2.x, o2.y);
        o1 = make_float2(o2.z, o2.w);
      }
      float4 P2;
      if (!OPR || Pk) {
        P2 = __ldg((const float4*)(Pk + p));
      } else {   // relaxed primary mode of this position
        P2 = opr_pair(a.opr_U, wj, a.K, NN, p);
        if (p0) *(float4*)(p0 + p) = P2;
      }
      const float2 x0 = cmul(make_float2(P2.x, P2.y), o0), x1 = cmul(make_float2(P2.z, P2.w), o1);
      store_pair(tile, np.phys(q), x0, x1);
    }
    __syncthreads();
    // the last mode's far field stays in the tile (each row in its own line's
    // storage, free once the row transform is done): the first inverse
    // transform reads it there instead of from the scratch
    const bool keep = k == M - 1 && a.mode != MODE_FWD && !a.loss_only;
    fft2_forward<N, T>(tile, tw, [&](int row, float2 (&v)[R2]) {
#pragma unroll
      for (int m = 0; m < R2; ++m) v[m] = cscale(v[m], invN);
      if constexpr (F::S == 2) {
        // registers (2q, 2q+1) hold two adjacent columns: 8-byte intensity and
        // 16-byte far-field accesses
#pragma unroll
        for (int q = 0; q < R2 / 2; ++q) {
          float2* ri = (float2*)(rI + row * RP + F::out_index(n, 2 * q));
          const float2 i2 = make_float2(cabs2(v[2 * q]), cabs2(v[2 * q + 1]));
          *ri = (k == 0) ? i2 : make_float2(ri->x + i2.x, ri->y + i2.y);
        }
      } else {
#pragma unroll
        for (int m = 0; m < R2; ++m) {
          float* ri = rI + row * RP + F::out_index(n, m);
          *ri = (k == 0) ? cabs2(v[m]) : *ri + cabs2(v[m]);
        }
      }
      if (keep) {
        F::template store_out<true>(v, tile, row, n);
      } else if (psi_s) {
        if constexpr (F::S == 2) {
#pragma unroll
          for (int q = 0; q < R2 / 2; ++q)
            *(float4*)(psi_s + (size_t)k * NN + row * N + F::out_index(n, 2 * q)) =
                make_float4(v[2 * q].x, v[2 * q].y, v[2 * q + 1].x, v[2 * q + 1].y);
        } else {
#pragma unroll
          for (int m = 0; m < R2; ++m) psi_s[(size_t)k * NN + row * N + F::out_index(n, m)] = v[m];
        }
      }
    });
    __syncthreads();
  }

  const int mode = a.mode;
  // ---- data term: loss and the far-field factor (same thread owns each pixel) ----
  const float eps = a.eps;
  const float* meas = a.meas + (size_t)j * NN;
  float lsum = 0.f;
  bool bad = false;
  {
    constexpr int L = T / R1, ITER = N / L;
    const int gid = F::line_slot();
#pragma unroll 1
    for (int it = 0; it < ITER; ++it) {
      const int row = gid + it * L;
      // the row's measured intensities, all loads issued before any use
      // (registers 2q, 2q+1 are adjacent columns when S = 2: 8-byte loads)
      float Imv[R2];
      if (mode != MODE_FWD) {
        if constexpr (F::S == 2) {
#pragma unroll
          for (int q = 0; q < R2 / 2; ++q) {
            const float2 t = __ldg((const float2*)(meas + row * N + F::out_index(n, 2 * q)));
            Imv[2 * q] = t.x;
            Imv[2 * q + 1] = t.y;
          }
        } else {
#pragma unroll
          for (int m = 0; m < R2; ++m) Imv[m] = __ldg(meas + row * N + F::out_index(n, m));
        }
      }
#pragma unroll
      for (int m = 0; m < R2; ++m) {
        const int col = F::out_index(n, m);
        const int pix = row * N + col;
        const float I = rI[row * RP + col];
        if (a.ipred) a.ipred[(size_t)j * NN + pix] = I;
        if (mode == MODE_FWD) continue;
        const float Im = Imv[m];
        float fac;
        if (mode == MODE_VJP) {
          bad |= !isfinite(Im);
          fac = 2.f * Im;
        } else {
          bad |= !(Im >= 0.f) || !isfinite(Im);
          const float Ie = I + eps;
          if (mode == MODE_LSQML_GAUSS || mode == MODE_GRAD_GAUSS) {
            const float sIe = sqrtf(Ie), sIm = sqrtf(Im);
            const float d = sIe - sIm;
            lsum = fmaf(d, d, lsum);
            const float rho = sIm / sIe;
            fac = (mode == MODE_LSQML_GAUSS) ? rho - 1.f : 2.f * (1.f - rho);
          } else {
            lsum += I - Im * logf(Ie);
            const float q = Im / Ie;
            fac = (mode == MODE_LSQML_POISSON) ? 0.5f * (q - 1.f) : 2.f * (1.f - q);
          }
        }
        rI[row * RP + col] = fac * invN;
      }
    }
  }
  if (bad) atomicOr(a.status, FLAG_NONFINITE);
  if (a.loss && mode != MODE_FWD && mode != MODE_VJP) {
    double v[1] = {(double)lsum};
    block_sum<1>(v, red);
    if (tid == 0) atomicAdd(a.loss, v[0]);
  }
  if (mode == MODE_FWD || a.loss_only) return;

  // ---- back-propagation: chi_k = F^-1[fac Psi_k], g = sum_k conj(P_k) chi_k, h_k ----
  // The modes run last to first: the far fields written last are read first,
  // while they are still in L2.
  float2* g_s = a.g_s + slotNN;
  float2* h_s = a.h_s + slotNN * M;
#pragma unroll 1
  for (int k = M - 1; k >= 0; --k) {
    const float2* Pk = shared_mode<OPR>(a, k, NN);
    __syncthreads();
    fft2_inverse<N, T>(
        tile, tw,
        [&](int row, float2 (&v)[R2]) {
          if (k == M - 1) {   // the last mode's far field was kept in the tile
            F::template load_out<true>(v, tile, row, n);
            __syncwarp();     // every lane of the line has read before the exchange writes
          } else if constexpr (F::S == 2) {
#pragma unroll
            for (int q = 0; q < R2 / 2; ++q) {
              const float4 X = *(const float4*)(psi_s + (size_t)k * NN + row * N + F::out_index(n, 2 * q));
              v[2 * q] = make_float2(X.x, X.y);
              v[2 * q + 1] = make_float2(X.z, X.w);
            }
          } else {
#pragma unroll
            for (int m = 0; m < R2; ++m) v[m] = psi_s[(size_t)k * NN + row * N + F::out_index(n, m)];
          }
          if constexpr (F::S == 2) {
#pragma unroll
            for (int q = 0; q < R2 / 2; ++q) {
              const float2 f = *(const float2*)(rI + row * RP + F::out_index(n, 2 * q));
              v[2 * q] = cscale(v[2 * q], f.x);
              v[2 * q + 1] = cscale(v[2 * q + 1], f.y);
            }
          } else {
#pragma unroll
            for (int m = 0; m < R2; ++m) v[m] = cscale(v[m], rI[row * RP + F::out_index(n, m)]);
          }
        },
        [&](int col, float2 (&v)[R2]) { F::template store_in<false>(v, tile, col, n); });
    __syncthreads();
    // chi_k (natural layout) is in the tile:
    // g += conj(P_k) chi_k, h_k = conj(o) chi_k
    const NatPairs<N, T> np;
#pragma unroll 2
    for (int q = 0; q < NatPairs<N, T>::STEPS; ++q) {
      const int p = np.pix(q);
      float2 x0, x1;
      load_pair(tile, np.phys(q), x0, x1);
      const float4 P2 = (!OPR || Pk) ? __ldg((const float4*)(Pk + p)) : *(const float4*)(p0 + p);
      const float4 o2 = *(const float4*)(o_s + p);
      const float2 g0 = cmulc(make_float2(P2.x, P2.y), x0), g1 = cmulc(make_float2(P2.z, P2.w), x1);
      float4 gv = make_float4(g0.x, g0.y, g1.x, g1.y);
      if (k < M - 1) {
        const float4 gp = *(const float4*)(g_s + p);
        gv = make_float4(gv.x + gp.x, gv.y + gp.y, gv.z + gp.z, gv.w + gp.w);
      }
      *(float4*)(g_s + p) = gv;
      const float2 h0 = cmulc(make_float2(o2.x, o2.y), x0), h1 = cmulc(make_float2(o2.z, o2.w), x1);
      __stcs((float4*)(h_s + (size_t)k * NN + p), make_float4(h0.x, h0.y, h1.x, h1.y));
    }
  }
  __syncthreads();

  // ---- scatter S_j^T g (and the illumination) into the object frame ----------------
  const NatPairs<N, T> np;
#pragma unroll 1
  for (int q = 0; q < NatPairs<N, T>::STEPS; ++q) {
    const float4 g2 = *(const float4*)(g_s + np.pix(q));
    store_pair(tile, np.phys(q), make_float2(g2.x, g2.y), make_float2(g2.z, g2.w));
  }
  overlap_add<N, N, T, OPR>(a, slot, j, 0, ty, tx, fy, fx, p0, rI, red, [&](int y, int x) { return tile[tix<N>(y, x)]; });
}


// Bilinear sample of dO_hat = dO_acc / (illum + damp) at the patch pixel whose
// four corners start at q (the quotient is taken per corner, then interpolated).
__device__ __forceinline__ float2 dohat(const float4* q, int W, float w00, float w01, float w10, float w11,
                                        float damp) {
  const float4 q00 = __ldg(q), q01 = __ldg(q + 1), q10 = __ldg(q + W), q11 = __ldg(q + W + 1);
  const float i00 = w00 / (q00.z + damp), i01 = w01 / (q01.z + damp);
  const float i10 = w10 / (q10.z + damp), i11 = w11 / (q11.z + damp);
  return make_float2(q00.x * i00 + q01.x * i01 + q10.x * i10 + q11.x * i11,
                     q00.y * i00 + q01.y * i01 + q10.y * i10 + q11.y * i11);
}

// Opts a kernel into more than 48 KB of dynamic shared memory, once per device
// (so that no attribute call happens while a stream is being captured).
template <class K>
cudaError_t smem_optin(K kernel, size_t bytes, unsigned long long* done_mask) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const unsigned long long bit = 1ull << (dev & 63);
  if (__atomic_load_n(done_mask, __ATOMIC_ACQUIRE) & bit) return cudaSuccess;
  e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (e == cudaSuccess) __atomic_fetch_or(done_mask, bit, __ATOMIC_ACQ_REL);
  return e;
}

template <int N, int T, bool OPR>
cudaError_t launch_pass1_t(const BatchArgs& a, cudaStream_t s) {
  constexpr size_t sm = Pass1Smem<N>::bytes;
  static unsigned long long done = 0;
  cudaError_t e = smem_optin(k_pass1<N, T, OPR>, sm, &done);
  if (e != cudaSuccess) return e;
  if (a.nb <= 0) return cudaSuccess;
  return launch_pdl(k_pass1<N, T, OPR>, dim3(a.nb), dim3(T), sm, s, a);
}

// variant 0: default CTA size, 1: the alternative (the relaxed-probe form has
// the default only)
template <int N>
cudaError_t launch_pass1(const BatchArgs& a, cudaStream_t s, int variant) {
  if (a.opr_U) return launch_pass1_t<N, Threads<N>::T, true>(a, s);
  return variant == 1 ? launch_pass1_t<N, Threads<N>::ALT, false>(a, s)
                      : launch_pass1_t<N, Threads<N>::T, false>(a, s);
}

}  // namespace ptycho
