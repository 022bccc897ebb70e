// Far-field stage of the per-position pass with the 2-D DFT evaluated as
// dense complex GEMMs on the 5th-generation tensor cores, in split BF16:
// every FP32 operand x is carried as x_hi + x_lo (x_hi = bf16(x),
// x_lo = bf16(x - x_hi)), and each real product keeps the three terms
// A_hi B_hi + A_lo B_hi + A_hi B_lo, accumulated in FP32 in tensor memory.
//
// The unitary 2-D DFT of an N x N tile X is F X F^T with F[m][c] =
// exp(-2 pi i m c / N) / sqrt(N) (Sec. 2.1, Eq. 4's far-field propagator).
// With D[m][n] = sum_c A[m][c] B[n][c] (A and B both K-major) it is two
// passes with the DFT matrix as A:
//   pass 1: D1[f][r] = sum_c F[f][c] X[r][c]       (B = X: rows r, K = columns c)
//   pass 2: D2[f'][f] = sum_r F[f'][r] D1[f][r]    (B = D1: rows f, K = r)
// so D2 = F X F^T with the row index in the TMEM lane and no transpose in
// between: the thread that owns TMEM lane f after pass 1 writes row f of the
// next B operand. The inverse uses conj(F). A complex product is four real
// products on separate re/im planes, the sign of the Fi terms chosen by the
// instruction descriptor's negate-A bit.
//
// k_exit (below) writes the exit waves psi_jk of a minibatch to the scratch.
//
// k_far_tc: per minibatch position (persistent CTAs): the exit waves psi_jk
// are transformed mode by mode; the far fields overwrite them in the scratch and their intensities
// accumulate per thread; the data term (Eq. 1 amplitude loss or the Poisson
// likelihood) gives the loss and the far-field factor; every mode is then
// scaled and transformed back, and chi_jk = F^-1[(rho - 1) Psi_jk] overwrites
// the scratch for the overlap-add part of the pass.
//
// Warp roles: groups of four producer warps (four groups at N = 128, else two)
// take the K steps in turn and write the step's B operand (a
// 16-wide K slice of four BF16 planes) into a ring of shared-memory slots;
// one MMA warp streams the DFT-matrix chunks and issues the MMAs as slices
// land; one TMA warp stages the exit waves and the measured intensities from
// global memory into a second ring with tiled tensor copies (128-byte
// swizzle). Pass-1 slices come from the staged exit waves, from the last
// forward far field still in TMEM (the first inverse transform) or from the
// far fields, staged again (the other inverse transforms); pass-2 slices from the
// pass-1 accumulator in TMEM. Pass 1 accumulates in TMEM buffer A, pass 2 in
// buffer B, so an image's pass-2 result drains while the next image's pass 1
// runs.
//
// Bound by the MMAs' operand reads from shared memory (about 1200 cycles per K
// step at N = 128, where the MMAs themselves take 768) and, for the rest, by the
// producers' chains. Measured on GB300, 256 positions: N = 128, 5 modes 453 ->
// 295 us, 1 mode 126 -> 84; N = 64, 4 modes 143 -> 118; N = 32, 2 modes, 512
// positions 94 -> 78 (before: eight warps on every slice, far fields stored and
// read back 16 bytes per line).
#pragma once
#include <cuda_bf16.h>

#include "kernels_pair.cuh"
#include "tc.cuh"

namespace ptycho {

template <int N>
struct FarTc {
  static_assert(N == 32 || N == 64 || N == 128, "DFT-GEMM windows");
  static constexpr int G = N == 128 ? 4 : 2;      // groups of four producer warps; group g takes the slices s % G = g
  static constexpr int PW = 4 * G;                // producer warps: TMEM lane quarter w % 4, group w / 4
  static constexpr int T = 32 * (PW + 2);         // and the MMA warp (PW) and the TMA warp (PW + 1)
  static constexpr int COLS_T = N / G;            // columns per producer thread: 16 (G u + g) + [0, 16)
  static constexpr int NCH = N / 16;              // K steps of one pass (= DFT chunks)
  static constexpr int NSF = 4;                   // ring slots of DFT chunks
  static constexpr int NSB = 4;                   // ring slots of B slices
  static constexpr int NSS = 4;                   // ring slots of staged tiles
  static constexpr int MT = 128;                  // MMA tile rows (DFT rows beyond N are zero)
  static constexpr uint32_t APLANE = MT * 16 * 2;            // one 128 x 16 BF16 plane of a chunk
  static constexpr uint32_t CHUNK = 4 * APLANE;              // Fr_hi, Fr_lo, Fi_hi, Fi_lo
  static constexpr uint32_t ASBO = 256;                      // 8-row groups of a 16-wide K slice
  static constexpr uint32_t BPLANE = (uint32_t)N * 16 * 2;   // one N x 16 BF16 plane of a B slice
  static constexpr uint32_t SLICE = 4 * BPLANE;              // Xr_hi, Xr_lo, Xi_hi, Xi_lo
  static constexpr uint32_t BSBO = 256;
  static constexpr uint32_t SSLOT = 128u * N;                // a staged tile: N rows x 32 floats
  static constexpr size_t fring = 0;
  static constexpr size_t sring = fring + (size_t)NSF * CHUNK;   // 1024-byte aligned (swizzled tiles)
  static constexpr size_t bring = sring + (size_t)NSS * SSLOT;
  static constexpr uint32_t WTILE = 16 * 128;                // a producer warp's tile: 16 rows of a slice
  static constexpr size_t wtile = bring + (size_t)NSB * SLICE;
  static constexpr size_t bars = wtile + (size_t)PW * WTILE;
  static constexpr int NBAR = 2 * NSF + 2 * NSB + 2 * NSS + 4 + PW;   // F, B and staging rings, p1, p2, drained, stored,
                                                                      // and a hand-over per producer warp
  static constexpr size_t misc = bars + 8 * (size_t)NBAR;
  static constexpr size_t mail = misc + 16;                     // running losses of each row
  static constexpr size_t bytes = mail + 128 * 8 + 1024;   // + alignment of the base to 1024 bytes
  static constexpr uint32_t COLS = 4 * N;                    // buffer A [0, 2N), buffer B [2N, 4N)
  static constexpr size_t dft_bytes = (size_t)NCH * CHUNK;
  static_assert(bytes <= 232448, "shared memory per CTA");
  static_assert(COLS >= 32 && COLS <= 512 && (COLS & (COLS - 1)) == 0, "TMEM allocation: a power of two <= 512");
  static_assert(sring % 1024 == 0 && SSLOT % 1024 == 0, "128-byte swizzled tiles need 1024-byte alignment");
  static_assert(CHUNK % 16 == 0 && SLICE % 16 == 0, "bulk copies move multiples of 16 bytes");
};

// An encoded tensor map (CUtensorMap), passed by value as a kernel parameter.
struct alignas(64) TmaDesc {
  unsigned long long v[16];
};

struct FarArgs {
  int H, W, M, J;
  const float* pos;
  const int* order;
  int b0, nb, mode;
  float eps;
  const float* meas;      // measured intensities, or dL/dI in MODE_VJP
  float2* psi_s;          // [B, M, N, N]: exit waves in, chi out (natural layout)
  const uint16_t* dft;    // DFT chunks written by k_dft_planes
  float* ipred;           // [J, N, N] or null
  double* loss;           // or null
  int* status;
};

// Exit waves of the split-BF16 form, one CTA per 32 rows of a position: the
// bilinear patch o_j = S_j(O) (Sec. 2.1) and psi_jk = P_k o_j of every mode go to
// the scratch, a pixel pair per thread. Bound by the stores (M + 1 planes of a
// position, 29 us at window 128, 5 modes, 256 positions: 42 us; with one CTA per
// position and its object tile staged by a tensor copy 56 us).
constexpr int BAND_T = 256;
template <int N>
struct DftBands {
  static constexpr int ROWS = 32, NUM = N / ROWS, PAIRS = ROWS * N / 2, PP = PAIRS / BAND_T;
  static constexpr size_t bytes = (size_t)ROWS * N * 12;   // g and the probe intensity of a band
  static_assert(PP * BAND_T == PAIRS, "whole pairs per thread");
};
template <int N>
__global__ void __launch_bounds__(BAND_T, 4) k_exit(BatchArgs a) {
  using C = DftBands<N>;
  constexpr int NN = N * N;
  wait_prior_grid();
  const int slot = blockIdx.x / C::NUM, p0 = (blockIdx.x % C::NUM) * C::PAIRS * 2, tid = threadIdx.x;
  const int e = a.b0 + slot, j = a.order ? a.order[e] : e;
  int ty = 0, tx = 0;
  float fy = 0.f, fx = 0.f;
  const bool ok = j >= 0 && j < a.J && tile_of(a.pos[2 * j], a.pos[2 * j + 1], N, a.H, a.W, ty, tx, fy, fx);
  if (tid == 0 && p0 == 0) {
    if (!ok) atomicOr(a.status, FLAG_BOUNDS);
    if (a.valid) a.valid[slot] = ok;
    if (a.gsum) a.gsum[2 * slot] = a.gsum[2 * slot + 1] = 0.0;
  }
  if (!ok) return;
  float2* psi = a.psi_s + (size_t)slot * a.M * NN;
#pragma unroll 2
  for (int i = 0; i < C::PP; ++i) {
    const int p = p0 + 2 * (i * BAND_T + tid);
    float2 o0, o1;
    bilinear2(a.obj, a.W, ty + p / N, tx + p % N, fy, fx, o0, o1);
    if (a.o_s) *(float4*)(a.o_s + (size_t)slot * NN + p) = make_float4(o0.x, o0.y, o1.x, o1.y);
    for (int k = 0; k < a.M; ++k) {
      const float4 P2 = __ldg((const float4*)(a.probe + (size_t)k * NN + p));
      const float2 x0 = cmul(make_float2(P2.x, P2.y), o0), x1 = cmul(make_float2(P2.z, P2.w), o1);
      *(float4*)(psi + (size_t)k * NN + p) = make_float4(x0.x, x0.y, x1.x, x1.y);
    }
  }
}

// The pass after the far field, one CTA per 32 rows of a position: g += conj(P_k)
// chi_k (in registers over the modes, last mode first as the FP32 pass) and
// h_k = conj(o) chi_k, then the overlap-add and the position sums of the band. The
// bands of a position add their shares of its gradient in FP64; k_gpos rounds
// the sum, once. (With the last band to arrive doing that, behind a fence that
// waits for the band's scatter, this kernel took 105 us instead of 95.)
// Bound by DRAM (2 M + 3 planes of a position, about 59 us at window 128, 5
// modes, 256 positions): 95 us there; one CTA of 1024 threads per position, g in
// global memory between the modes, took 155 us.
template <int N>
__global__ void __launch_bounds__(BAND_T, 3) k_overlap(BatchArgs a) {
  using C = DftBands<N>;
  constexpr int NN = N * N, U = C::PP < 4 ? C::PP : 4;   // pairs in flight
  extern __shared__ __align__(16) float2 gS[];           // the band of g, then of the probe intensity
  __shared__ double red[32 * 5];
  wait_prior_grid();
  const int slot = blockIdx.x / C::NUM, y0 = (blockIdx.x % C::NUM) * C::ROWS, tid = threadIdx.x;
  const int e = a.b0 + slot, j = a.order ? a.order[e] : e;
  int ty = 0, tx = 0;
  float fy = 0.f, fx = 0.f;
  if (!(j >= 0 && j < a.J) || !tile_of(a.pos[2 * j], a.pos[2 * j + 1], N, a.H, a.W, ty, tx, fy, fx)) return;   // (flagged)
  const size_t base = (size_t)slot * NN;
  const int M = a.M;
#pragma unroll 1
  for (int i0 = 0; i0 < C::PP; i0 += U) {
    const int l = 2 * (i0 * BAND_T + tid), p = y0 * N + l;   // in the band, in the patch
    float4 o[U], g[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      o[u] = *(const float4*)(a.o_s + base + p + 2 * u * BAND_T);
      g[u] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
#pragma unroll 1
    for (int k = M - 1; k >= 0; --k) {
      const size_t at = (base * M + (size_t)k * NN) + p;
      float4 c[U], P[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        c[u] = __ldcs((const float4*)(a.psi_s + at + 2 * u * BAND_T));
        P[u] = __ldg((const float4*)(a.probe + (size_t)k * NN + p + 2 * u * BAND_T));
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const float2 x0 = make_float2(c[u].x, c[u].y), x1 = make_float2(c[u].z, c[u].w);
        const float2 g0 = cmulc(make_float2(P[u].x, P[u].y), x0), g1 = cmulc(make_float2(P[u].z, P[u].w), x1);
        g[u] = k == M - 1 ? make_float4(g0.x, g0.y, g1.x, g1.y)
                          : make_float4(g0.x + g[u].x, g0.y + g[u].y, g1.x + g[u].z, g1.y + g[u].w);
        const float2 h0 = cmulc(make_float2(o[u].x, o[u].y), x0), h1 = cmulc(make_float2(o[u].z, o[u].w), x1);
        __stcs((float4*)(a.h_s + at + 2 * u * BAND_T), make_float4(h0.x, h0.y, h1.x, h1.y));
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      *(float4*)(a.g_s + base + p + 2 * u * BAND_T) = g[u];
      *(float4*)(gS + l + 2 * u * BAND_T) = g[u];
    }
  }
  overlap_add<N, C::ROWS, BAND_T, false, true>(a, slot, j, y0, ty, tx, fy, fx, nullptr, (float*)(gS + C::ROWS * N), red,
                                               [&](int y, int x) { return gS[y * N + x]; });
}

// gpos += the position gradient's FP64 sums of the valid slots.
__global__ void __launch_bounds__(BAND_T) k_gpos(BatchArgs a) {
  wait_prior_grid();
  const int i = blockIdx.x * BAND_T + threadIdx.x, slot = i / 2;
  if (slot >= a.nb || !a.valid[slot]) return;
  const int e = a.b0 + slot, j = a.order ? a.order[e] : e;
  atomicAdd(a.gpos + 2 * j + i % 2, (float)a.gsum[i]);
}

__device__ __forceinline__ uint16_t bf16_bits(float v) { return __bfloat16_as_ushort(__float2bfloat16_rn(v)); }
__device__ __forceinline__ float bf16_value(uint16_t b) { return __bfloat162float(__ushort_as_bfloat16(b)); }
// x = hi + lo to within 2^-16 |x| (BF16 keeps 8 significant bits)
// Two values as their hi and lo BF16 parts, packed (x in the low half).
__device__ __forceinline__ void split2_bf16(float x, float y, uint32_t& hi, uint32_t& lo) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(x, y);
  hi = *(const uint32_t*)&h;
  const __nv_bfloat162 l = __floats2bfloat162_rn(x - __uint_as_float(hi << 16), y - __uint_as_float(hi & 0xffff0000u));
  lo = *(const uint32_t*)&l;
}

// The DFT matrix of one pass as NCH chunks (one per 16-wide K slice), each the
// four planes Fr_hi, Fr_lo, Fi_hi, Fi_lo of 128 rows x 16 BF16 in the
// operand's shared-memory image (core matrices of 8 rows x 16 bytes, K-adjacent
// ones 128 bytes apart, 8-row groups 256 bytes apart). F[m][c] =
// exp(-2 pi i m c / N), rows m >= N zero; evaluated in FP64 from m c mod N.
template <int N>
__global__ void k_dft_planes(uint16_t* out) {
  using C = FarTc<N>;
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= C::NCH * C::MT * 16) return;
  const int s = idx / (C::MT * 16), m = (idx / 16) % C::MT, kk = idx % 16, c = 16 * s + kk;
  double re = 0.0, im = 0.0;
  if (m < N) {
    const int r = (int)(((long long)m * c) % N);
    double sn, cs;
    sincospi(2.0 * (double)r / (double)N, &sn, &cs);
    re = cs;
    im = -sn;
  }
  const size_t e = (size_t)s * (C::CHUNK / 2) + (size_t)(m / 8) * (C::ASBO / 2) + (kk / 8) * 64 + (m % 8) * 8 + (kk % 8);
  constexpr size_t P = C::APLANE / 2;
  const float reh = (float)re, imh = (float)im;
  const uint16_t rh = bf16_bits(reh), ih = bf16_bits(imh);
  out[e] = rh;
  out[e + P] = bf16_bits((float)(re - (double)bf16_value(rh)));
  out[e + 2 * P] = ih;
  out[e + 3 * P] = bf16_bits((float)(im - (double)bf16_value(ih)));
}

// Eight consecutive K values (K offset 8 h of a 16-wide slice) of operand
// row `row` into the four planes of a B slice (hi/lo of re and im).
template <int N>
__device__ __forceinline__ void put8(unsigned char* slice, int row, int h, const float* re, const float* im) {
  using C = FarTc<N>;
  uint32_t rh[4], rl[4], ih[4], il[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    split2_bf16(re[2 * q], re[2 * q + 1], rh[q], rl[q]);
    split2_bf16(im[2 * q], im[2 * q + 1], ih[q], il[q]);
  }
  unsigned char* p = slice + (size_t)(row / 8) * C::BSBO + h * 128 + (row % 8) * 16;
  *(uint4*)p = make_uint4(rh[0], rh[1], rh[2], rh[3]);
  *(uint4*)(p + C::BPLANE) = make_uint4(rl[0], rl[1], rl[2], rl[3]);
  *(uint4*)(p + 2 * C::BPLANE) = make_uint4(ih[0], ih[1], ih[2], ih[3]);
  *(uint4*)(p + 3 * C::BPLANE) = make_uint4(il[0], il[1], il[2], il[3]);
}

// Bounded wait that also gives up when another role has aborted; the
// outcome is made uniform over the warp.
__device__ __forceinline__ bool role_wait(uint64_t* b, uint32_t parity, volatile int* abort_s) {
  bool ok = tc::mbar_try_wait(b, parity);
  if (!ok) {
    const long long t0 = clock64();
    while (!(ok = tc::mbar_try_wait(b, parity))) {
      if (*abort_s) break;
      if (clock64() - t0 > (1ll << 31)) {
        *abort_s = 1;
        break;
      }
    }
  }
  return !__any_sync(0xffffffffu, !ok);
}

// Staged-tile element of row `row`, 16-byte chunk `c` (of 8), in the
// 128-byte swizzle the tensor copies write: chunk c of row r sits at c ^ (r % 8).
__device__ __forceinline__ float4 staged_chunk(const unsigned char* tile, int row, int c) {
  return *(const float4*)(tile + (size_t)row * 128 + ((c ^ (row & 7)) << 4));
}

template <int N>
__global__ void __launch_bounds__(FarTc<N>::T, 1)
    k_far_tc(FarArgs a, const __grid_constant__ TmaDesc tm_psi, const __grid_constant__ TmaDesc tm_meas) {
  using C = FarTc<N>;
  constexpr int NN = N * N, G = C::G, NU = C::NCH / G, NCH = C::NCH, NSB = C::NSB, NSS = C::NSS;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  wait_prior_grid();
  unsigned char* smem = smem_raw + ((1024u - (tc::smem_u32(smem_raw) & 1023u)) & 1023u);
  unsigned char* fring = smem + C::fring;
  unsigned char* sring = smem + C::sring;
  unsigned char* bring = smem + C::bring;
  uint64_t* fullF = (uint64_t*)(smem + C::bars);
  uint64_t* emptyF = fullF + C::NSF;
  uint64_t* fullB = emptyF + C::NSF;
  uint64_t* emptyB = fullB + NSB;
  uint64_t* fullS = emptyB + NSB;
  uint64_t* emptyS = fullS + NSS;
  uint64_t* p1done = emptyS + NSS;
  uint64_t* p2done = p1done + 1;
  uint64_t* drained = p2done + 1;
  uint64_t* stored = drained + 1;
  uint64_t* handed = stored + 1;
  uint32_t* holder = (uint32_t*)(smem + C::misc);
  volatile int* abort_s = (volatile int*)(holder + 1);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid == 0) {
    for (int s = 0; s < C::NSF; ++s) {
      tc::mbar_init(&fullF[s], 1);
      tc::mbar_init(&emptyF[s], 1);
    }
    for (int s = 0; s < NSB; ++s) {
      tc::mbar_init(&fullB[s], 4);
      tc::mbar_init(&emptyB[s], 1);
    }
    for (int s = 0; s < NSS; ++s) {
      tc::mbar_init(&fullS[s], 1);
      tc::mbar_init(&emptyS[s], 4);
    }
    tc::mbar_init(p1done, 1);
    tc::mbar_init(p2done, 1);
    tc::mbar_init(drained, C::PW);
    tc::mbar_init(stored, C::PW);
    for (int w = 0; w < C::PW; ++w) tc::mbar_init(&handed[w], 1);
    *abort_s = 0;
    tc::fence_mbar_init();
  }
  if (warp == 0) {
    tc::tmem_alloc(holder, C::COLS);
    tc::tmem_relinquish();
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = *holder;
  const uint32_t bufA = tmem, bufB = tmem + 2 * N;

  // The image sequence every role walks: per valid slot, M forward transforms,
  // then (unless only intensities are wanted) M inverse ones.
  auto slot_j = [&](int slot) -> int {
    const int e = a.b0 + slot;
    const int j = a.order ? a.order[e] : e;
    int ty, tx;
    float fy, fx;
    if (!(j >= 0 && j < a.J) || !tile_of(a.pos[2 * j], a.pos[2 * j + 1], N, a.H, a.W, ty, tx, fy, fx)) return -1;
    return j;   // an invalid slot is flagged by the first part of the pass
  };
  const bool backward = a.mode != MODE_FWD;

  if (warp == C::PW) {
    // ================================ MMA warp ====================================
    if (lane == 0) {
      const unsigned char* dft = (const unsigned char*)a.dft;
      uint32_t qc = 0, issued = 0, cb = 0;
      int64_t last_mma = -1;   // the last chunk whose MMAs were issued (and committed)
      for (int s = 0; s < C::NSF; ++s) {
        tc::mbar_expect_tx(&fullF[s], C::CHUNK);
        tc::bulk_g2s(fring + (size_t)s * C::CHUNK, dft + (size_t)(s % NCH) * C::CHUNK, C::CHUNK, &fullF[s]);
      }
      issued = C::NSF;
      constexpr uint32_t I_POS = tc::idesc_bf16(C::MT, N, false), I_NEG = tc::idesc_bf16(C::MT, N, true);
      bool ok = true;
      // one pass into the accumulator at `d` (re at d, im at d + N)
      auto pass = [&](uint32_t d, bool inverse, uint64_t* done) {
        const uint32_t i_re = inverse ? I_POS : I_NEG;   // Fi Xi into D_re: minus forward, plus inverse
        const uint32_t i_im = inverse ? I_NEG : I_POS;   // Fi Xr into D_im: plus forward, minus inverse
        for (int s = 0; s < NCH && ok; ++s, ++qc, ++cb) {
          const int sf = (int)(qc % C::NSF), sb = (int)(cb % NSB);
          if (!tc::mbar_wait(&fullF[sf], (uint32_t)((qc / C::NSF) & 1)) ||
              !tc::mbar_wait(&fullB[sb], (uint32_t)((cb / NSB) & 1))) {
            ok = false;
            break;
          }
          tc::fence_after_sync();
          const uint32_t sa = tc::smem_u32(fring + (size_t)sf * C::CHUNK);
          const uint64_t aRh = tc::sdesc(sa, 128, C::ASBO), aRl = tc::sdesc(sa + C::APLANE, 128, C::ASBO);
          const uint64_t aIh = tc::sdesc(sa + 2 * C::APLANE, 128, C::ASBO);
          const uint64_t aIl = tc::sdesc(sa + 3 * C::APLANE, 128, C::ASBO);
          const uint32_t sbase = tc::smem_u32(bring + (size_t)sb * C::SLICE);
          const uint64_t bRh = tc::sdesc(sbase, 128, C::BSBO), bRl = tc::sdesc(sbase + C::BPLANE, 128, C::BSBO);
          const uint64_t bIh = tc::sdesc(sbase + 2 * C::BPLANE, 128, C::BSBO);
          const uint64_t bIl = tc::sdesc(sbase + 3 * C::BPLANE, 128, C::BSBO);
          const uint32_t acc0 = s > 0 ? 1u : 0u, dre = d, dim = d + N;
          tc::mma_bf16(dre, aRh, bRh, I_POS, acc0);
          tc::mma_bf16(dre, aRl, bRh, I_POS, 1u);
          tc::mma_bf16(dre, aRh, bRl, I_POS, 1u);
          tc::mma_bf16(dre, aIh, bIh, i_re, 1u);
          tc::mma_bf16(dre, aIl, bIh, i_re, 1u);
          tc::mma_bf16(dre, aIh, bIl, i_re, 1u);
          tc::mma_bf16(dim, aRh, bIh, I_POS, acc0);
          tc::mma_bf16(dim, aRl, bIh, I_POS, 1u);
          tc::mma_bf16(dim, aRh, bIl, I_POS, 1u);
          tc::mma_bf16(dim, aIh, bRh, i_im, 1u);
          tc::mma_bf16(dim, aIl, bRh, i_im, 1u);
          tc::mma_bf16(dim, aIh, bRl, i_im, 1u);
          tc::mma_commit(&emptyF[sf]);
          tc::mma_commit(&emptyB[sb]);
          last_mma = qc;
          if (qc >= 1) {   // refill the previous chunk's slot once its MMAs are done
            const uint32_t qp = qc - 1, qn = qp + C::NSF;
            const int sp = (int)(qp % C::NSF);
            if (!tc::mbar_wait(&emptyF[sp], (uint32_t)((qp / C::NSF) & 1))) {
              ok = false;
              break;
            }
            tc::mbar_expect_tx(&fullF[sp], C::CHUNK);
            tc::bulk_g2s(fring + (size_t)sp * C::CHUNK, dft + (size_t)(qn % NCH) * C::CHUNK, C::CHUNK,
                         &fullF[sp]);
            ++issued;
          }
        }
        if (ok) tc::mma_commit(done);
      };
      uint32_t n = 0;
      for (int slot = blockIdx.x; slot < a.nb && ok && !*abort_s; slot += gridDim.x) {
        if (slot_j(slot) < 0) continue;
        for (int t = 0; t < (backward ? 2 * a.M : a.M) && ok && !*abort_s; ++t, ++n) {
          const bool inverse = t >= a.M;
          pass(bufA, inverse, p1done);
          if (ok && n >= 1 && !tc::mbar_wait(drained, (uint32_t)((n - 1) & 1))) ok = false;
          if (ok) pass(bufB, inverse, p2done);
        }
      }
      if (!ok) *abort_s = 1;
      // copies still in flight land before the CTA exits
      for (; qc < issued; ++qc)
        if (!tc::mbar_wait(&fullF[(int)(qc % C::NSF)], (uint32_t)((qc / C::NSF) & 1))) {
          *abort_s = 1;
          break;
        }
      // after an abort, the MMAs already issued finish (their last commit
      // completes) before the tensor memory is released
      if (*abort_s && last_mma >= 0)
        tc::mbar_wait(&emptyF[(int)(last_mma % C::NSF)], (uint32_t)((last_mma / C::NSF) & 1));
    }
  } else if (warp == C::PW + 1) {
    // ================================ TMA warp ====================================
    // Stages, in the order the producers consume them, the exit waves of the
    // forward transforms (N x 32-float tiles, 16 complex columns each), the
    // measured intensities of the data term (N x 16-float tiles) and, once the
    // producers have stored them, the far fields of the inverse transforms but
    // the first.
    if (lane == 0) {
      uint32_t ps = 0, np = 0;
      bool ok = true;
      auto stage = [&](const TmaDesc* map, int x, int z) {
        const int sl = (int)(ps % NSS);
        if (ps >= NSS && !tc::mbar_wait(&emptyS[sl], (uint32_t)(((ps / NSS) - 1) & 1))) {
          ok = false;
          return;
        }
        tc::mbar_expect_tx(&fullS[sl], map == &tm_meas ? C::SSLOT / 2 : C::SSLOT);
        tc::tma_load_3d(sring + (size_t)sl * C::SSLOT, map, x, 0, z, &fullS[sl]);
        ++ps;
      };
      for (int slot = blockIdx.x; slot < a.nb && ok && !*abort_s; slot += gridDim.x) {
        const int j = slot_j(slot);
        if (j < 0) continue;
        for (int k = 0; k < a.M && ok; ++k)
          for (int s = 0; s < NCH && ok; ++s) stage(&tm_psi, 32 * s, slot * a.M + k);
        if (backward)
          for (int s = 0; s < NCH && ok; ++s) stage(&tm_meas, 16 * s, j);
        if (backward && a.M > 1 && ok) {
          if (!tc::mbar_wait(stored, np++ & 1)) ok = false;
          for (int k = a.M - 2; k >= 0 && ok; --k)
            for (int s = 0; s < NCH && ok; ++s) stage(&tm_psi, 32 * s, slot * a.M + k);
        }
      }
      if (!ok) *abort_s = 1;
      // tiles still in flight land before the CTA exits (the last fill of each slot)
      for (uint32_t p = ps - (ps < (uint32_t)NSS ? ps : (uint32_t)NSS); p < ps; ++p)
        if (!tc::mbar_wait(&fullS[(int)(p % NSS)], (uint32_t)((p / NSS) & 1))) {
          *abort_s = 1;
          break;
        }
    }
  } else {
    // ============================= producer warps =================================
    // Each group of four warps takes whole slices in turn: a slice's chain (wait,
    // load, split, store, publish) is long, and eight warps on one slice after
    // the other left the tensor cores waiting for it.
    const int q4 = warp & 3, g = warp >> 2;
    const int row = 32 * q4 + lane;           // TMEM lane = operand row
    const bool act = row < N;                  // warp-uniform
    const uint32_t lrow = (uint32_t)(32 * q4) << 16;
    const float invN = 1.0f / (float)N;
    uint32_t pb = g, ps = g, n = 0, nd = 0, nh = 0;
    float acc[C::COLS_T];                      // I, then the far-field factor, of columns 16 (G u + g) + [0, 16)
#pragma unroll
    for (int i = 0; i < C::COLS_T; ++i) acc[i] = 0.f;
    bool alive = true;

    // takes B slot pb (waiting for it to be free), fills it, publishes it
    auto publish = [&](auto&& fill) {
      const int sb = (int)(pb % NSB);
      if (pb >= NSB && !role_wait(&emptyB[sb], (uint32_t)(((pb / NSB) - 1) & 1), abort_s)) {
        alive = false;
        return;
      }
      if (act) fill(bring + (size_t)sb * C::SLICE);
      tc::fence_async_smem();
      tc::fence_before_sync();
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&fullB[sb]);
      pb += G;
    };
    // waits for staged tile ps; returns it (null if a wait gave up)
    auto staged = [&]() -> const unsigned char* {
      const int sl = (int)(ps % NSS);
      if (!role_wait(&fullS[sl], (uint32_t)((ps / NSS) & 1), abort_s)) {
        alive = false;
        return nullptr;
      }
      return sring + (size_t)sl * C::SSLOT;
    };
    auto release_staged = [&]() {
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&emptyS[(int)(ps % NSS)]);
      ps += G;
    };
    // pass-1 slice G u + g from the staged tile of an exit wave or a far field,
    // times the factors
    auto produce_slice = [&](int u, auto scale) {
      const unsigned char* tile = staged();
      if (!alive) return;
      publish([&](unsigned char* slice) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          float re[8], im[8];
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const float4 v = staged_chunk(tile, row, 4 * h + i);
            const float f0 = scale(u, 8 * h + 2 * i), f1 = scale(u, 8 * h + 2 * i + 1);
            re[2 * i] = v.x * f0; im[2 * i] = v.y * f0;
            re[2 * i + 1] = v.z * f1; im[2 * i + 1] = v.w * f1;
          }
          put8<N>(slice, row, h, re, im);
        }
      });
      if (alive) release_staged();
    };
    auto produce_staged = [&]() {
#pragma unroll 1
      for (int u = 0; u < NU && alive; ++u) produce_slice(u, [](int, int) { return 1.f; });
    };
    auto produce_scaled = [&]() {
#pragma unroll
      for (int u = 0; u < NU; ++u)
        if (alive) produce_slice(u, [&](int v, int i) { return acc[16 * v + i]; });
    };
    // slices from an accumulator in TMEM: pass-2 slices from buffer A, or
    // (SCALE) the first inverse transform's pass-1 slices from the last forward
    // far field in buffer B, times 1/N and the factors
    auto tmem_slice = [&](uint32_t buf, int u, auto scale) {
      float re[16], im[16];
      if (act) {
        const uint32_t col = buf + lrow + 16 * (G * u + g);
        tc::tmem_ld16x2_wait(col, re, col + N, im);
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          const float f = scale(u, i);
          re[i] *= f;
          im[i] *= f;
        }
      }
      publish([&](unsigned char* slice) {
        put8<N>(slice, row, 0, re, im);
        put8<N>(slice, row, 1, re + 8, im + 8);
      });
    };
    auto produce_tmem = [&]() {   // (rolled: straight-line code runs at the rate of its fetch)
#pragma unroll 1
      for (int u = 0; u < NU && alive; ++u) tmem_slice(bufA, u, [](int, int) { return 1.f; });
    };
    auto produce_tmem_scaled = [&]() {
#pragma unroll
      for (int u = 0; u < NU; ++u)
        if (alive) tmem_slice(bufB, u, [&](int v, int i) { return acc[16 * v + i] * invN; });
    };
    // 16-byte chunk c of row r of the warp's tile, of 16 rows of 128 or 32 rows of
    // 64 bytes; chunks permuted so that rows and columns of it are free of bank
    // conflicts
    unsigned char* wtile = smem + C::wtile + warp * C::WTILE;
    auto chunk128 = [&](int r, int c) { return (float4*)(wtile + r * 128 + ((c ^ (r & 7)) << 4)); };
    auto chunk64 = [&](int r, int c) { return (float4*)(wtile + r * 64 + ((c ^ ((r >> 1) & 3)) << 4)); };
    // the pass-2 accumulator (buffer B) times `scale` to global memory (unless
    // dst is null); with `accumulate` its squared modulus is stored into
    // (first) or added to acc. A thread owns a row of the accumulator: stored
    // from there a warp's store touches 32 lines, 16 bytes each, and the rate of
    // these requests bound the kernel; turned through the warp's tile it writes
    // four whole lines.
    auto drain = [&](float2* dst, bool accumulate, bool first, float scale) {
      if (act) {
#pragma unroll
        for (int u = 0; u < NU; ++u) {
          const int col = 16 * (G * u + g);
          float re[16], im[16];
          tc::tmem_ld16x2_wait(bufB + lrow + col, re, bufB + lrow + N + col, im);
#pragma unroll
          for (int i = 0; i < 16; ++i) {
            re[i] *= scale;
            im[i] *= scale;
            if (accumulate) {
              const float a0 = fmaf(re[i], re[i], im[i] * im[i]);
              acc[16 * u + i] = first ? a0 : acc[16 * u + i] + a0;
            }
          }
          if (dst) {
#pragma unroll
            for (int t = 0; t < 2; ++t) {
              __syncwarp();   // the rows before have left the tile
              if ((lane >> 4) == t)
#pragma unroll
                for (int i = 0; i < 8; ++i)
                  *chunk128(lane & 15, i) = make_float4(re[2 * i], im[2 * i], re[2 * i + 1], im[2 * i + 1]);
              __syncwarp();
#pragma unroll
              for (int k = 0; k < 4; ++k) {
                const int r = 4 * k + lane / 8;
                *(float4*)(dst + (size_t)(32 * q4 + 16 * t + r) * N + col + 2 * (lane % 8)) = *chunk128(r, lane % 8);
              }
            }
          }
        }
      }
    };
    auto arrive_drained = [&]() {
      tc::fence_before_sync();
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(drained);
    };
    // the data term of position j from the intensities in acc: loss, ipred, and
    // the far-field factor (times 1/N for the unnormalised inverse) into acc;
    // the measured values come from the staged tiles (none in the forward mode).
    // The loss of a row is two running FP32 sums in column order, one per half
    // of the slices; the warps that share the row hand them over from slice to
    // slice.
    auto data_term = [&](int j) {
      float2 lsum = make_float2(0.f, 0.f);
      bool bad = false;
      const bool sums = backward && a.mode != MODE_VJP;
      float2* mail = (float2*)(smem + C::mail) + row;
      float* ip = (a.ipred && act) ? a.ipred + (size_t)j * NN + (size_t)(32 * q4) * N : nullptr;
      const bool vec = ((uintptr_t)a.ipred & 15) == 0;
#pragma unroll
      for (int u = 0; u < NU; ++u) {
        const int s = G * u + g;
        if (ip) {   // 8 rows x 64 bytes per store, through the warp's tile
          __syncwarp();
#pragma unroll
          for (int i = 0; i < 4; ++i)
            *chunk64(lane, i) = make_float4(acc[16 * u + 4 * i], acc[16 * u + 4 * i + 1], acc[16 * u + 4 * i + 2],
                                            acc[16 * u + 4 * i + 3]);
          __syncwarp();
#pragma unroll
          for (int t = 0; t < 4; ++t) {
            const int r = 8 * t + lane / 4;
            const float4 v = *chunk64(r, lane % 4);
            float* d = ip + (size_t)r * N + 16 * s + 4 * (lane % 4);
            if (vec) {
              *(float4*)d = v;
            } else {
              d[0] = v.x; d[1] = v.y; d[2] = v.z; d[3] = v.w;
            }
          }
        }
        if (!backward) continue;
        const unsigned char* tile = staged();
        if (!alive) break;
        float4 t[4];   // what the loss adds
        if (act) {
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const float4 Im = *(const float4*)(tile + row * 64 + ((i ^ ((row >> 1) & 3)) << 4));
            float* A = acc + 16 * u + 4 * i;
            float4 f;
            if (a.mode == MODE_VJP) {
              bad |= !isfinite(Im.x) || !isfinite(Im.y) || !isfinite(Im.z) || !isfinite(Im.w);
              f = make_float4(2.f * Im.x, 2.f * Im.y, 2.f * Im.z, 2.f * Im.w);
            } else {
              auto off = [](float x) { return !(x >= 0.f) || !isfinite(x); };
              bad |= off(Im.x) || off(Im.y) || off(Im.z) || off(Im.w);
              f = data_factor(a.mode, make_float4(A[0], A[1], A[2], A[3]), Im, a.eps, t[i]);
            }
            A[0] = f.x * invN; A[1] = f.y * invN; A[2] = f.z * invN; A[3] = f.w * invN;
          }
        }
        release_staged();
        if (!sums) continue;
        if (s > 0) {   // the sums up to the slice before
          if (!role_wait(&handed[q4 + 4 * ((g + G - 1) % G)], nh & 1, abort_s)) {
            alive = false;
            break;
          }
          ++nh;
          lsum = *mail;
        }
        if (act) {
          const bool sq = a.mode == MODE_LSQML_GAUSS || a.mode == MODE_GRAD_GAUSS;
          auto add = [&](float& l, const float4& v) {
            if (sq) {
              l = fmaf(v.x, v.x, l); l = fmaf(v.y, v.y, l); l = fmaf(v.z, v.z, l); l = fmaf(v.w, v.w, l);
            } else {
              l += v.x; l += v.y; l += v.z; l += v.w;
            }
          };
          add(lsum.x, t[0]); add(lsum.x, t[1]);
          add(lsum.y, t[2]); add(lsum.y, t[3]);
        }
        if (s < NCH - 1) {
          *mail = lsum;
          __syncwarp();
          if (lane == 0) tc::mbar_arrive(&handed[warp]);
        }
      }
      if (bad) atomicOr(a.status, FLAG_NONFINITE);
      if (a.loss && sums && g == G - 1) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          double v = (double)(h ? lsum.y : lsum.x);
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
          if (lane == 0 && v != 0.0) atomicAdd(a.loss, v);
        }
      }
    };

    // the previous image, drained once the next image's pass-1 slices are out
    float2* prev_dst = nullptr;
    bool have_prev = false, prev_fwd = false, prev_first = false, prev_last_fwd = false, prev_before_last = false;
    int prev_j = -1;
    auto drain_prev = [&]() {
      if (!role_wait(p2done, (uint32_t)(nd & 1), abort_s)) {
        alive = false;
        return;
      }
      tc::fence_after_sync();
      // forward far fields are kept for the inverse transforms (not needed
      // when only intensities are computed); inverse results are chi
      drain(prev_fwd && !backward ? nullptr : prev_dst, prev_fwd, prev_first, prev_fwd ? invN : 1.f);
      arrive_drained();
      ++nd;
      if (backward && prev_before_last) {   // every far field that is read again has been stored
        asm volatile("fence.proxy.async;\n" ::: "memory");   // (the copies that read them are asynchronous)
        __syncwarp();
        if (lane == 0) tc::mbar_arrive(stored);
      }
      if (prev_fwd && prev_last_fwd && !backward) data_term(prev_j);
      have_prev = false;
    };

    for (int slot = blockIdx.x; slot < a.nb && alive; slot += gridDim.x) {
      const int j = slot_j(slot);
      if (j < 0) continue;
      float2* psi = a.psi_s + (size_t)slot * a.M * NN;
      for (int t = 0; t < (backward ? 2 * a.M : a.M) && alive; ++t, ++n) {
        const bool fwd = t < a.M;
        const int k = fwd ? t : 2 * a.M - 1 - t;
        float2* io = psi + (size_t)k * NN;
        if (fwd) {
          produce_staged();
          if (have_prev && alive) drain_prev();
        } else if (k == a.M - 1) {
          // first inverse transform: the last forward far field is still in
          // buffer B; its intensities complete I, then the data term gives the
          // factor, then its pass-1 slices come straight from TMEM
          if (!role_wait(p2done, (uint32_t)(nd & 1), abort_s)) {
            alive = false;
            break;
          }
          tc::fence_after_sync();
          drain(nullptr, true, a.M == 1, invN);
          ++nd;
          data_term(j);
          if (alive) produce_tmem_scaled();
          arrive_drained();
          have_prev = false;
        } else {
          produce_scaled();
          if (have_prev && alive) drain_prev();
        }
        if (!alive) break;
        if (!role_wait(p1done, (uint32_t)(n & 1), abort_s)) {
          alive = false;
          break;
        }
        tc::fence_after_sync();
        produce_tmem();
        prev_dst = io;
        have_prev = true;
        prev_fwd = fwd;
        prev_first = fwd && k == 0;
        prev_last_fwd = fwd && k == a.M - 1;
        prev_before_last = fwd && k == a.M - 2;
        prev_j = j;
      }
    }
    if (alive && have_prev) drain_prev();
    if (!alive) *abort_s = 1;
  }

  if (tid == 0 && *abort_s) atomicOr(a.status, FLAG_TIMEOUT);
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  if (warp == 0) tc::tmem_dealloc(tmem, C::COLS);
}

}  // namespace ptycho
