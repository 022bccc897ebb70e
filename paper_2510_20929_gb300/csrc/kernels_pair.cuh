// The per-position pass on the packed line-pair transforms: windows 32 (but for
// launches of few positions, see pass_n32.cu), 64 and 128 in one CTA
// (fft_pair.cuh), 192 and 256 on a cluster of CTAs with 32 rows each
// (fft_cluster.cuh). It computes what k_pass1 (kernels.cuh) describes; what
// differs is where the data lives:
//   * every thread owns the same pixel pairs (two neighbours of one row, or, on
//     a cluster, of one column) when a mode's exit wave is built and when its chi comes back, so
//     psi_jk goes from the loads straight into the column transform's
//     registers and chi_jk from the registers into g and h, with no pass over
//     the tile on either side;
//   * the far field, the measured intensities and the factor of the data term
//     belong to one thread each, so the far-field scratch and the
//     intensity/factor plane hold one 16-byte unit per thread and step (every
//     access a whole coalesced run), and the last mode's far field stays in
//     registers through the data term into its inverse transform;
//   * the patch o_j and the running g_j of the thread's pixels stay in tensor
//     memory (windows 64 and up: 8 NP columns of the thread's TMEM lane).
// What bounds it: the transforms (about half the cycles; shared-memory
// wavefronts and issue slots), then the rate of L2 requests of the probe
// loads, the far-field scratch and the h stores (about 2.8 cycles per 128-byte
// request when all SMs stream), with one CTA of 512 threads filling an SM at
// window 128, and on the cluster windows the waits for the cluster.
// Straight-line code that a CTA runs once costs instruction fetches, so loops
// over a thread's pixels stay rolled where v is not indexed.
// Measured on GB300 against the one-line-per-lane-group passes it replaced (per
// launch): window 256, 8 modes, 256 positions 2423 -> 1705 us, 1 mode 496 ->
// 342; window 192, 4 modes 986 -> 673, 1 mode 406 -> 293; window 128, 5 modes,
// 256 positions 287 -> 249 us (1 mode: 101 -> 92, 1024 positions 1002 -> 860);
// window 64, 4 modes, 256 positions 63 -> 51, 1216 positions 227 -> 166, 1 mode,
// 16 positions 24.7 -> 20.7; window 32, 4 modes, 2000 positions 116 -> 72.
#pragma once
#include <type_traits>

#include "kernels.cuh"
#include "fft_cluster.cuh"

namespace ptycho {

// One thread's view of a window held by one CTA (ClFft is that of a cluster):
// pixel pair i = (row(i), col(i)) and the next column; far field of register i
// at rows far_y(i), far_y(i) + 1 of column far_x(i).
template <int N_>
struct OneCta {
  using F = fp::Fft<N_>;
  static constexpr int N = N_, R1 = F::R1, NP = F::R2, LR = N, Q = 1, T = F::T, TW = Twiddles<N>::COUNT;
  static constexpr bool VERT = false;
  __device__ __forceinline__ static void fill_twiddles(float2* tw) { make_twiddles<N>(tw); }
  float4* tile;
  const float2* tw;
  int p, n, pr, nr;
  __device__ __forceinline__ OneCta(float4* tile_, const float2* tw_)
      : tile(tile_), tw(tw_), p(F::col_pair()), n(F::col_lane()), pr(F::row_pair()), nr(F::row_lane()) {}
  static constexpr int q = 0;
  __device__ __forceinline__ int row(int i) const { return n + R1 * i; }
  __device__ __forceinline__ int col(int) const { return 2 * p; }
  __device__ __forceinline__ int far_y(int) const { return 2 * pr; }
  __device__ __forceinline__ int far_x(int i) const { return F::far_col(nr, i); }
  __device__ __forceinline__ static void pixel_sync() { F::col_sync(); }
  __device__ __forceinline__ void forward(fp::C2 (&v)[NP]) const {
    F::fwd_cols(v, tile, p, n, tw);
    __syncthreads();
    F::fwd_rows(v, tile, pr, nr, tw);
  }
  __device__ __forceinline__ void inverse(fp::C2 (&v)[NP]) const {
    F::inv_rows(v, tile, pr, nr, tw);
    __syncthreads();
    F::inv_cols(v, tile, p, n, tw);
  }
  // unit that holds pixel pair i once the line's lanes have read theirs, and
  // the 8-byte slot of local pixel (y, x) in those units
  __device__ __forceinline__ int pixel_unit(int i) const { return F::colu(row(i), p); }
  __device__ __forceinline__ static int pixel_slot(int y, int x) { return 2 * F::colu(y, x >> 1) + (x & 1); }
};

// What a CTA does about a copy whose wait gave up (`got` false in one of its
// threads): the status records it, and after a second bounded wait (copies in
// flight must not outlive the CTA) the position is dropped, with nothing of it
// scattered and its slot marked invalid. A CTA of a cluster cannot leave before
// the others, which write into its memory until the last transform, and goes on.
// After the forward transforms, whose barriers put that after the mark of the
// cluster's first CTA, it clears valid[slot] (settle_lost); after the inverse
// ones, whose barriers make that visible, every CTA of the cluster reads it
// before it scatters. The outputs of a forward model or of a loss alone are not
// held back on a cluster.
template <class G>
__device__ __forceinline__ bool copy_arrived(const G& geo, bool got, uint64_t* bar, uint32_t parity, int* status,
                                             int* valid, bool give_up) {
  if (give_up) got = got && geo.q < G::Q - 1;   // (self-test: in one CTA)
  if (__syncthreads_and(got)) return true;
  if (threadIdx.x == 0) {
    atomicOr(status, FLAG_TIMEOUT);
    if (G::Q == 1 && valid) *valid = 0;
    tc::mbar_wait(bar, parity);
  }
  __syncthreads();
  return false;
}
template <class G>
__device__ __forceinline__ void settle_lost(int* valid, bool lost) {
  if (G::Q > 1 && threadIdx.x == 0 && lost) *(volatile int*)valid = 0;
}

// Launch shape: CTAs per SM (shared memory at the windows 128 and up; the
// register budget, 80 and 128 a thread, at 64 and 32). On the cluster windows
// two CTAs of different clusters share an SM: one computes while the other
// waits on its cluster. Their 256 TMEM columns each fill it, and their shared
// memory (over a third of the SM's) keeps a third from fitting, so no CTA of
// a cluster can wait for tensor memory that another waiting cluster holds.
template <class G> struct PairCtas;
template <> struct PairCtas<OneCta<16>> { static constexpr int n = 16; };
template <> struct PairCtas<OneCta<32>> { static constexpr int n = 8; };
template <> struct PairCtas<OneCta<64>> { static constexpr int n = 3; };
template <> struct PairCtas<OneCta<128>> { static constexpr int n = 1; };
template <> struct PairCtas<fp::ClFft<192>> { static constexpr int n = 2; };
template <> struct PairCtas<fp::ClFft<256>> { static constexpr int n = 2; };

template <class G>
struct PairSmem {
  static constexpr int N = G::N, LNN = G::LR * G::N;   // pixels of the CTA
  static constexpr size_t red = 0;
  static constexpr size_t tile = red + 256 * sizeof(double);
  static constexpr size_t rI = tile + (size_t)LNN * sizeof(float2);
  static constexpr size_t tw = rI + (size_t)LNN * sizeof(float);
  static constexpr size_t o = tw + (size_t)G::TW * sizeof(float2);
  static constexpr size_t bytes = o + (N >= 64 ? 0 : (size_t)LNN * sizeof(float2));
  // the staged object tile: LR + 1 rows of up to N + 2 pixels, over the tile and
  // the intensity plane (free before the first transform). The pitch is 64
  // bytes off a multiple of 128: the rows of a half-warp's lanes alternate
  // between the two halves of the banks (window 16: what fits).
  static constexpr int opitch = N == 16 ? 160 : N * 8 + 64;
  static_assert((G::LR + 1) * opitch <= LNN * 12, "the object tile fits");
  static_assert(G::Q == 1 || 3 * (bytes + 1024) > 228 * 1024, "no third CTA (its tensor memory would not fit)");
};

// The data term of four pixels (Eq. 1, or the Poisson likelihood): adds the
// loss and returns the far-field factor. Square roots and quotients are
// formed from rsqrtf with one residual correction each (Markstein, IBM J. Res.
// Dev. 34, 1990: s += r y / 2 with the residual r = x - s^2 exact in one fused
// multiply-add; q += r / d likewise): sqrtf and the division leave the straight
// code for a zero operand, and most counts of a diffraction pattern are zero. The
// values were sqrtf's for every float in [1, 4) and the division's, for both
// likelihoods, in all of 2^24 pairs of a count and an intensity. Values outside
// 2^-96 .. 2^96 (zero counts aside) take the functions. `t` receives what the
// loss adds per pixel: the difference of the amplitudes (added squared), or
// the Poisson term; (x, z) and (y, w) are two rows.
__device__ __forceinline__ float4 data_factor(int mode, float4 I, float4 Im, float eps, float4& t) {
  constexpr float lo = 1.2621774e-29f, hi = 7.9228163e28f;   // 2^-96, 2^96
  const bool gauss = mode == MODE_LSQML_GAUSS || mode == MODE_GRAD_GAUSS;
  const bool lsqml = mode == MODE_LSQML_GAUSS || mode == MODE_LSQML_POISSON;
  const float2 I2[2] = {make_float2(I.x, I.y), make_float2(I.z, I.w)};
  const float2 M2[2] = {make_float2(Im.x, Im.y), make_float2(Im.z, Im.w)};
  float2 Ie[2], mx[2], rho[2], T2[2];
  bool in = true;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    Ie[h] = make_float2(I2[h].x + eps, I2[h].y + eps);
    mx[h] = make_float2(M2[h].x == 0.f ? 1.f : M2[h].x, M2[h].y == 0.f ? 1.f : M2[h].y);
    in = in && fminf(fminf(Ie[h].x, Ie[h].y), fminf(mx[h].x, mx[h].y)) >= lo &&
         fmaxf(fmaxf(Ie[h].x, Ie[h].y), fmaxf(mx[h].x, mx[h].y)) <= hi &&
         !(isnan(Ie[h].x) || isnan(Ie[h].y) || isnan(mx[h].x) || isnan(mx[h].y));
  }
  if (in) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const float2 y = make_float2(rsqrtf(Ie[h].x), rsqrtf(Ie[h].y));
      if (gauss) {
        const float2 half = fp::splat(0.5f);
        const float2 ym = make_float2(rsqrtf(mx[h].x), rsqrtf(mx[h].y));
        float2 s = fp::mul2(Ie[h], y), m = fp::mul2(mx[h], ym);
        s = fp::fma2(fp::mul2(half, y), fp::fma2(fp::neg2(s), s, Ie[h]), s);
        m = fp::fma2(fp::mul2(half, ym), fp::fma2(fp::neg2(m), m, mx[h]), m);
        if (M2[h].x == 0.f) m.x = 0.f;
        if (M2[h].y == 0.f) m.y = 0.f;
        T2[h] = fp::sub2(s, m);
        const float2 q = fp::mul2(m, y);
        rho[h] = fp::fma2(fp::fma2(fp::neg2(q), s, m), y, q);
      } else {
        float2 c = fp::mul2(y, y);   // 1 / Ie
        c = fp::fma2(c, fp::fma2(fp::neg2(Ie[h]), c, fp::splat(1.f)), c);
        const float2 q = fp::mul2(M2[h], c);
        rho[h] = fp::fma2(fp::fma2(fp::neg2(q), Ie[h], M2[h]), c, q);
        T2[h] = make_float2(I2[h].x - M2[h].x * logf(Ie[h].x), I2[h].y - M2[h].y * logf(Ie[h].y));
      }
    }
  } else {
    const float Iv[4] = {I.x, I.y, I.z, I.w}, Mv[4] = {Im.x, Im.y, Im.z, Im.w};
    float r[4], l[4];
#pragma unroll
    for (int h = 0; h < 4; ++h) {
      const float E = Iv[h] + eps;
      if (gauss) {
        const float s = sqrtf(E), m = sqrtf(Mv[h]);
        l[h] = s - m;
        r[h] = m / s;
      } else {
        l[h] = Iv[h] - Mv[h] * logf(E);
        r[h] = Mv[h] / E;
      }
    }
    T2[0] = make_float2(l[0], l[1]);
    T2[1] = make_float2(l[2], l[3]);
    rho[0] = make_float2(r[0], r[1]);
    rho[1] = make_float2(r[2], r[3]);
  }
  t = make_float4(T2[0].x, T2[0].y, T2[1].x, T2[1].y);
  const float w = lsqml ? (gauss ? 1.f : 0.5f) : -2.f;   // rho - 1, (q - 1) / 2, or 2 (1 - rho)
  return make_float4(w * (rho[0].x - 1.f), w * (rho[0].y - 1.f), w * (rho[1].x - 1.f), w * (rho[1].y - 1.f));
}

// A thread's pixel pair at p in a plane of the patch: loads (read-only data, and
// data this kernel writes) and stores.
template <class G>
__device__ __forceinline__ float4 ldg_pair(const float2* p) {
  if constexpr (G::VERT) {
    const float2 u = __ldg(p), v = __ldg(p + G::N);
    return make_float4(u.x, u.y, v.x, v.y);
  } else {
    return __ldg((const float4*)p);
  }
}
template <class G>
__device__ __forceinline__ float4 ld_pair(const float2* p) {
  if constexpr (G::VERT) {
    const float2 u = p[0], v = p[G::N];
    return make_float4(u.x, u.y, v.x, v.y);
  } else {
    return *(const float4*)p;
  }
}
template <class G>
__device__ __forceinline__ void st_pair(float2* p, float4 v) {
  if constexpr (G::VERT) {
    p[0] = make_float2(v.x, v.y);
    p[G::N] = make_float2(v.z, v.w);
  } else {
    *(float4*)p = v;
  }
}
template <class G>
__device__ __forceinline__ void stcs_pair(float2* p, float4 v) {
  if constexpr (G::VERT) {
    __stcs(p, make_float2(v.x, v.y));
    __stcs(p + G::N, make_float2(v.z, v.w));
  } else {
    __stcs((float4*)p, v);
  }
}
// The packed pair of a pixel pair, and its product with one.
__device__ __forceinline__ fp::C2 pack_pair(float2 a, float2 b) { return {make_float2(a.x, b.x), make_float2(a.y, b.y)}; }
__device__ __forceinline__ fp::C2 exit_wave(float4 P, float4 o) {
  return pack_pair(cmul(make_float2(P.x, P.y), make_float2(o.x, o.y)),
                   cmul(make_float2(P.z, P.w), make_float2(o.z, o.w)));
}

// Runs use(i, load(i)) for the NP pixel pairs with D loads ahead of their use
// (the wave of a thread fills half of its registers, so the loads of a whole
// plane do not fit beside it).
template <int NP, int D, class Load, class Use>
__device__ __forceinline__ void ahead(Load&& load, Use&& use) {
  decltype(load(0)) r[D];
#pragma unroll
  for (int i = 0; i < D; ++i) r[i] = load(i);
#pragma unroll
  for (int i = 0; i < NP; ++i) {
    const auto x = r[i % D];
    if (i + D < NP) r[i % D] = load(i + D);
    use(i, x);
  }
}

// The CTA's rows of the (N + 1)^2 object tile, staged in shared memory by one
// bulk copy per row, from the row's start rounded down to 16 bytes (row r then
// begins at pixel off(r)); rows of an unaligned object, and the one row whose
// copy would end past the plane, by plain loads.
template <class G>
struct ObjStage {
  static constexpr int N = G::N, LR = G::LR, T = G::T, PITCH = PairSmem<G>::opitch;
  unsigned char* stage;
  uint64_t* bar;
  const float2* tile0;   // first pixel of the CTA's rows in the plane
  int W;
  bool bulk, end;        // bulk copies; the last row ends the plane
  // plane: H x W pixels, `base` the (16-byte aligned, for bulk copies) array it lies in
  __device__ __forceinline__ ObjStage(void* smem, uint64_t* bar_, const void* base, const float2* plane, int H, int W_,
                                      int y, int x)
      : stage((unsigned char*)smem), bar(bar_), tile0(plane + (size_t)y * W_ + x), W(W_), bulk(((uintptr_t)base & 15) == 0),
        end((size_t)(y + LR) * W_ + x + N + 2 > (size_t)H * W_) {}
  __device__ __forceinline__ int off(int r) const {
    return bulk ? (int)(((uintptr_t)tile0 >> 3) + (uintptr_t)r * W) & 1 : 0;
  }
  __device__ __forceinline__ bool row_plain(int r) const { return !bulk || (r == LR && end && off(r) == 0); }
  // one thread, before any copy completes; then the whole CTA
  __device__ __forceinline__ void expect() const {
    if (bulk) tc::mbar_expect_tx(bar, (uint32_t)((row_plain(LR) ? LR : LR + 1) * (N + 2) * sizeof(float2)));
  }
  __device__ __forceinline__ void copy() const {
    for (int r = threadIdx.x; r < LR + 1; r += T)
      if (!row_plain(r))
        tc::bulk_g2s(stage + r * PITCH, tile0 + (size_t)r * W - off(r), (N + 2) * sizeof(float2), bar);
    if (!bulk) {
      for (int i = threadIdx.x; i < (LR + 1) * (N + 1); i += T) {
        const int r = i / (N + 1), c = i % (N + 1);
        ((float2*)(stage + r * PITCH))[c] = __ldg(tile0 + (size_t)r * W + c);
      }
    } else if (row_plain(LR)) {
      for (int c = threadIdx.x; c < N + 1; c += T) ((float2*)(stage + LR * PITCH))[c] = __ldg(tile0 + (size_t)LR * W + c);
    }
  }
  __device__ __forceinline__ bool wait(uint32_t parity) const { return !bulk || tc::mbar_wait(bar, parity); }
  // the bilinear patch at a pixel pair (staged rows and joined threads)
  __device__ __forceinline__ float4 patch(int r, int c, float fy, float fx) const {
    const float w00 = (1.f - fy) * (1.f - fx), w01 = (1.f - fy) * fx, w10 = fy * (1.f - fx), w11 = fy * fx;
    auto srow = [&](int y) { return (const float2*)(stage + y * PITCH) + off(y) + c; };
    auto mix = [&](float2 a, float2 b, float2 d, float2 e) {
      return make_float2(w00 * a.x + w01 * b.x + w10 * d.x + w11 * e.x, w00 * a.y + w01 * b.y + w10 * d.y + w11 * e.y);
    };
    const float2 *A = srow(r), *B = srow(r + 1);
    const float2 a0 = A[0], a1 = A[1], b0 = B[0], b1 = B[1];
    const float2 o0 = mix(a0, a1, b0, b1);
    float2 o1;
    if constexpr (G::VERT) {
      const float2* D = srow(r + 2);
      o1 = mix(b0, b1, D[0], D[1]);
    } else {
      o1 = mix(a1, A[2], b1, B[2]);
    }
    return make_float4(o0.x, o0.y, o1.x, o1.y);
  }
};

// The far field v (scaled to the unitary transform) into the intensity plane.
template <class G>
__device__ __forceinline__ void add_intensity(const fp::C2 (&v)[G::NP], float4* rI, bool first) {
#pragma unroll
  for (int i = 0; i < G::NP; i += 2) {
    float2 i0 = fp::fma2(v[i].re, v[i].re, fp::mul2(v[i].im, v[i].im));
    float2 i1 = fp::fma2(v[i + 1].re, v[i + 1].re, fp::mul2(v[i + 1].im, v[i + 1].im));
    float4* ri = rI + (i / 2) * G::T + threadIdx.x;
    if (!first) {
      const float4 s = *ri;
      i0 = fp::add2(make_float2(s.x, s.y), i0);
      i1 = fp::add2(make_float2(s.z, s.w), i1);
    }
    *ri = make_float4(i0.x, i0.y, i1.x, i1.y);
  }
}
// v times the factors of the intensity plane.
template <class G>
__device__ __forceinline__ void mul_factor(fp::C2 (&v)[G::NP], const float4* rI) {
#pragma unroll
  for (int i = 0; i < G::NP; i += 2) {
    const float4 f = rI[(i / 2) * G::T + threadIdx.x];
    v[i] = fp::pscale(v[i], make_float2(f.x, f.y));
    v[i + 1] = fp::pscale(v[i + 1], make_float2(f.z, f.w));
  }
}
// A thread's far field in its scratch plane: unit i at plane[i T].
template <class G>
__device__ __forceinline__ void put_far(const fp::C2 (&v)[G::NP], float4* plane) {
#pragma unroll
  for (int i = 0; i < G::NP; ++i) plane[i * G::T] = make_float4(v[i].re.x, v[i].re.y, v[i].im.x, v[i].im.y);
}
template <class G>
__device__ __forceinline__ void get_far(fp::C2 (&v)[G::NP], const float4* plane) {
#pragma unroll
  for (int i = 0; i < G::NP; ++i) {
    const float4 x = plane[i * G::T];
    v[i] = {make_float2(x.x, x.y), make_float2(x.z, x.w)};
  }
}

// The data term of the CTA's far-field pixels: the intensity plane rI becomes
// the plane of factors, `ipred` (when set) receives the intensities, `loss` the
// loss. The tile must be free; `arrived(got, bar)` joins the block after the
// wait for the pattern and says whether to go on. A rolled loop over the units
// of the plane: unrolled over the far field's registers it would be most of the
// kernel's code, and ran at the speed of instruction fetches.
template <class G, bool CHAIN, class Arrived>
__device__ __forceinline__ bool data_term(const G& geo, float4* rI, double* red, uint64_t* bar,
                                          const float* __restrict__ meas_all, int j, float* ipred, int mode, float eps,
                                          double* loss, int* status, Arrived&& arrived_all) {
  constexpr int N = G::N, T = G::T, NP = G::NP, NN = N * N, LR = G::LR, LNN = LR * N;
  const int tid = threadIdx.x, y0 = LR * geo.q;
  const float invN = 1.0f / (float)N;
  float4* tile = geo.tile;
  float2 ls = make_float2(0.f, 0.f);   // rows 2pr and 2pr + 1
  bool bad = false;
  const bool sq = mode == MODE_LSQML_GAUSS || mode == MODE_GRAD_GAUSS;
  auto add_loss = [&](float4 t) {
    if (sq)
      ls = fp::fma2(make_float2(t.z, t.w), make_float2(t.z, t.w),
                    fp::fma2(make_float2(t.x, t.y), make_float2(t.x, t.y), ls));
    else
      ls = fp::add2(fp::add2(ls, make_float2(t.x, t.y)), make_float2(t.z, t.w));
  };
  // The pattern into the tile, one bulk copy per row (loaded straight to its
  // threads, 32 bytes of a row per request, it took 6,000 cycles). The pitch
  // spreads the row pairs of a warp over the banks.
  constexpr int FW = G::VERT ? LR : N;   // far-field columns of the CTA
  constexpr int MP = FW + 4;
  float* mS = (float*)tile;
  const int x0 = G::VERT ? y0 : 0;       // its first column
  const float* meas = meas_all + (size_t)j * NN + x0;
  if (mode != MODE_FWD) {
    const bool mbulk = ((uintptr_t)meas_all & 15) == 0;
    tc::fence_async_smem();
    __syncthreads();   // the tile is free
    if (mbulk) {
      if (tid == 0) tc::mbar_expect_tx(bar, (uint32_t)(LNN * sizeof(float)));
      for (int r = tid; r < N; r += T) tc::bulk_g2s(mS + r * MP, meas + r * N, FW * sizeof(float), bar);
    } else {
      for (int i = tid; i < LNN; i += T) mS[i / FW * MP + i % FW] = __ldg(meas + i / FW * N + i % FW);
    }
    if (!arrived_all(!mbulk || tc::mbar_wait(bar, 0), bar)) return false;
  }
  // unit i of the intensity plane: registers 2i and 2i + 1 of v, two far-field
  // pixels each; their places in the staged pattern (and, with the pitch N,
  // in the whole one)
  struct At { int a, b, c, d; };
  auto at = [&](int i, int pitch) -> At {
    if constexpr (G::VERT) {
      const int p = geo.far_y(2 * i) * pitch + geo.far_x(), r = geo.far_y(2 * i + 1) * pitch + geo.far_x();
      return {p, p + 1, r, r + 1};
    } else {
      const int y = geo.far_y(0) * pitch, c = geo.far_x(2 * i), d = geo.far_x(2 * i + 1);
      return {y + c, y + pitch + c, y + d, y + pitch + d};
    }
  };
#pragma unroll 1
  for (int i = 0; i < NP / 2; ++i) {
    const float4 I = rI[i * T + tid];
    if (ipred) {
      float* d = ipred + (size_t)j * NN + x0;
      const At g = at(i, N);
      d[g.a] = I.x; d[g.b] = I.y; d[g.c] = I.z; d[g.d] = I.w;
    }
    if (mode == MODE_FWD) continue;
    const At m = at(i, MP);
    const float4 Im = make_float4(mS[m.a], mS[m.b], mS[m.c], mS[m.d]);
    float4 f;
    if (mode == MODE_VJP) {
      bad |= !isfinite(Im.x) || !isfinite(Im.y) || !isfinite(Im.z) || !isfinite(Im.w);
      f = make_float4(2.f * Im.x, 2.f * Im.y, 2.f * Im.z, 2.f * Im.w);
    } else {
      auto off = [](float x) { return !(x >= 0.f) || !isfinite(x); };
      bad |= off(Im.x) || off(Im.y) || off(Im.z) || off(Im.w);
      float4 t;
      f = data_factor(mode, I, Im, eps, t);
      add_loss(t);
      if constexpr (CHAIN) {   // kept for the upper rows' sum below
        mS[m.a] = t.x; mS[m.b] = t.y; mS[m.c] = t.z; mS[m.d] = t.w;
      }
    }
    rI[i * T + tid] = make_float4(f.x * invN, f.y * invN, f.z * invN, f.w * invN);
  }
  if (bad) atomicOr(status, FLAG_NONFINITE);
  if (loss && mode != MODE_FWD && mode != MODE_VJP) {
    // FP32 per row and lane (CHAIN: rows r and r + N / 2 in one sum; on a
    // cluster, per column and lane), a tree over the lanes and some rows (the
    // CTA's columns), FP64 from there: the loss keeps one order of summation,
    // whatever the packing
    int slots;
    bool mine = true;
    if constexpr (CHAIN) {
      float2* lo = (float2*)(mS + N * MP);
      static_assert(N * MP * 4 + T / 2 * 8 <= LNN * 8, "room beside the pattern");
      mine = tid >= T / 2;
      if (!mine) lo[tid] = ls;
      __syncthreads();
      if (mine) {
        ls = lo[tid - T / 2];
#pragma unroll 1
        for (int i = 0; i < NP / 2; ++i) {
          const At m = at(i, MP);
          add_loss(make_float4(mS[m.a], mS[m.b], mS[m.c], mS[m.d]));
        }
      }
      __syncthreads();
    }
    if constexpr (!G::VERT) {
      constexpr int LP = 32 / G::R1;   // line pairs per warp
      auto down = [](float x, int o) { return x + __shfl_down_sync(0xffffffffu, x, o); };
      float sum;
      if constexpr (N == 16) {   // rows first, then lanes
        ls = make_float2(down(down(ls.x, 2), 1), down(down(ls.y, 2), 1));
        sum = down(down(ls.x + ls.y, 16), 8);
      } else {
#pragma unroll
        for (int o = 16; o >= 1; o /= 2)
          if (o != LP / 2) ls = make_float2(down(ls.x, o), down(ls.y, o));
        sum = ls.x + ls.y;
      }
      const int lane = tid & 31;   // lanes 0 and LP / 2 hold LP rows each
      if ((lane & ~(LP / 2)) == 0) red[(tid >> 5) * 2 + (lane != 0)] = mine ? (double)sum : 0.0;
      slots = 2 * (T / 32);
    } else {
      float* col = mS + N * MP;   // [lane][column]
      *(float2*)(col + geo.n * LR + geo.far_x()) = ls;
      __syncthreads();
#pragma unroll
      for (int r = tid >> 5; r < G::R1; r += T / 32) {
        float s = col[r * LR + (tid & 31)];
#pragma unroll
        for (int o = 16; o >= 1; o /= 2) s += __shfl_down_sync(0xffffffffu, s, o);
        if ((tid & 31) == 0) red[r] = (double)s;
      }
      slots = G::R1;
    }
    __syncthreads();
    if (tid < 32) {
      double s = tid < slots ? red[tid] : 0.0;
      for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
      if (tid == 0) atomicAdd(loss, s);
    }
  }
  return true;
}

template <class G, bool OPR>
__global__ void __launch_bounds__(G::T, PairCtas<G>::n) k_pass1_pair(BatchArgs a) {
  using SM = PairSmem<G>;
  using fp::C2;
  constexpr int N = G::N, T = G::T, NP = G::NP, NN = N * N, LR = G::LR, Q = G::Q, LNN = LR * N;
  static_assert(NP % 4 == 0 && NP * T * 2 == LNN, "pixel pairs");
  constexpr int D = 6;   // probe loads in flight in the backward pass (its v fills half the registers)
  extern __shared__ __align__(16) unsigned char smem[];
  wait_prior_grid();
  double* red = (double*)(smem + SM::red);
  float4* tile = (float4*)(smem + SM::tile);
  float4* rI = (float4*)(smem + SM::rI);
  float2* tw = (float2*)(smem + SM::tw);

  const int slot = blockIdx.x / Q, tid = threadIdx.x;
  const G geo(tile, tw);
  const int y0 = LR * geo.q;   // first patch row of this CTA
  const bool first = tid == 0 && geo.q == 0;
  const int e = a.b0 + slot;
  const int j = a.order ? a.order[e] : e;
  int ty = 0, tx = 0;
  float fy = 0.f, fx = 0.f;
  bool ok = (j >= 0 && j < a.J);
  if (ok) ok = tile_of(a.pos[2 * j], a.pos[2 * j + 1], N, a.H, a.W, ty, tx, fy, fx);
  if (!ok) {   // (the same decision in every CTA of a cluster)
    if (first) {
      atomicOr(a.status, FLAG_BOUNDS);
      if (a.valid) a.valid[slot] = 0;
    }
    return;
  }
  if (first && a.valid) a.valid[slot] = 1;
  // the measured intensities are first read by the data term, after the forward
  // transforms: fetch them into L2 meanwhile (they may live in host memory)
  if (first && a.meas && a.mode != MODE_FWD)
    prefetch_l2_bulk(a.meas + (size_t)j * NN, (uint32_t)(NN * sizeof(float)));
  uint64_t* bar = (uint64_t*)(red + 252);
  const ObjStage<G> stage(tile, bar, a.obj, a.obj, a.H, a.W, ty + y0, tx);
  if (tid == 0) {
    tc::mbar_init(bar, 1);
    tc::mbar_init(bar + 1, 1);
    tc::fence_mbar_init();
    stage.expect();
  }
  constexpr bool TM = N >= 64;
  constexpr int TMN = T / 128 * 8 * NP, TMC = TMN == 192 ? 256 : TMN, TG = 4 * NP;   // columns of the CTA; g's offset
  uint32_t* tm_holder = (uint32_t*)(red + 250);   // beyond the block reductions' 160 doubles
  if constexpr (TM) {
    if (tid < 32) {
      tc::tmem_alloc(tm_holder, TMC);
      tc::tmem_relinquish();
    }
    tc::fence_before_sync();
  }
  __syncthreads();   // the barrier's state, the tensor-memory address
  if constexpr (TM) tc::fence_after_sync();
  stage.copy();
  G::fill_twiddles(tw);

  const int M = a.M, mode = a.mode;
  const float invN = 1.0f / (float)N;
  const size_t slotNN = (size_t)slot * NN;
  float* wj = (float*)(red + 128);   // this position's eigenmode weights (OPR)
  float2* p0 = (OPR && a.p0_s) ? a.p0_s + slotNN : nullptr;
  if (OPR && tid < a.K) wj[tid] = a.opr_w[(size_t)j * a.K + tid];
  // far field of mode k, unit i of this thread: psi[k NN / 2 + i T] (the CTA's
  // share of the plane is the memory of its own pixel rows)
  float4* oS = (float4*)(smem + SM::o) + tid;   // (window 32) pixel pair q at oS[q T]
  float4* psi = a.psi_s ? (float4*)(a.psi_s + slotNN * M + (size_t)y0 * N) + tid : nullptr;
  float2* o_s = a.o_s ? a.o_s + slotNN : nullptr;
  auto pix = [&](int i) { return (y0 + geo.row(i)) * N + geo.col(i); };   // pixel pair i in a plane

  // Tensor memory as per-thread storage: the thread's NP pixel pairs of o in
  // the first 4 NP of its columns, of g in the next 4 NP (warp w reaches lanes
  // 32 (w % 4) ..+31; every fourth warp shares them, 8 NP columns each). A CTA
  // holds TMC columns: the SM's 512 serve all the CTAs its shared memory admits.
  // (Window 32: o in shared memory, g in its scratch.)
  auto tm_o = [&]() -> uint32_t {
    const int w = (int)(threadIdx.x >> 5);
    return *tm_holder + ((uint32_t)(32 * (w & 3)) << 16) + (uint32_t)((w >> 2) * 8 * NP);
  };
  auto tm_release = [&]() {
    if constexpr (TM) {
      tc::fence_before_sync();
      __syncthreads();
      tc::fence_after_sync();
      if (threadIdx.x < 32) tc::tmem_dealloc(*tm_holder, TMC);
    }
  };
  // The pixel pairs of a probe mode. The relaxed primary mode is synthesised
  // eigenmode by eigenmode, half of the pairs' loads in flight (pair by pair,
  // each over all eigenmodes, 256 positions of the 192 window with 8
  // eigenmodes took 613 us instead of 435), and kept in p0 for the way back.
  // The one call that is slower for it than with the unpacked pass is the
  // forward model of a lone relaxed mode at window 256 (700 positions, 8
  // eigenmodes 524 -> 600 us, 1: 448 -> 466): two eigenmodes in flight (629 us),
  // quarters of the pairs with four (591, but 192 slower) and a prefetch of
  // the next eigenmode into L1 (632) did not mend it.
  auto probe_fwd = [&](const float2* Pk, float4 (&P)[NP]) {
    if (!OPR || Pk) {
#pragma unroll
      for (int i = 0; i < NP; ++i) P[i] = ldg_pair<G>(Pk + pix(i));
      return;
    }
#pragma unroll
    for (int i = 0; i < NP; ++i) P[i] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int h = 0; h < NP; h += NP / 2)
#pragma unroll 1
      for (int m = 0; m < a.K; ++m) {
        const float w = wj[m];
        const float2* U = a.opr_U + (size_t)m * NN;
#pragma unroll
        for (int i = h; i < h + NP / 2; ++i) {
          const float4 u = ldg_pair<G>(U + pix(i));
          P[i].x = fmaf(w, u.x, P[i].x); P[i].y = fmaf(w, u.y, P[i].y);
          P[i].z = fmaf(w, u.z, P[i].z); P[i].w = fmaf(w, u.w, P[i].w);
        }
      }
    if (p0)
#pragma unroll
      for (int i = 0; i < NP; ++i) st_pair<G>(p0 + pix(i), P[i]);
  };
  auto probe_back = [&](const float2* Pk, int i) -> float4 {
    return (!OPR || Pk) ? ldg_pair<G>(Pk + pix(i)) : ld_pair<G>(p0 + pix(i));
  };

  // ---- forward model: I_j = sum_k |F(P_k o_j)|^2 -------------------------------
  // Every pixel pair of a mode's probe is in flight at once: the loads are
  // issued before the barrier that frees the tile (the registers of v are
  // empty there).
  C2 v[NP];
  float4 P[NP];
  if (OPR) __syncthreads();   // the weights
  probe_fwd(shared_mode<OPR>(a, 0, NN), P);
  // joins the block after a wait for copies; false when a thread's wait gave up
  // (everything is released then, but on a cluster: see copy_arrived)
  auto arrived_all = [&](bool got, uint64_t* b) -> bool {
    if (copy_arrived(geo, got, b, 0, a.status, a.valid ? a.valid + slot : nullptr, (a.give_up >> (int)(b - bar)) & 1))
      return true;
    if (Q == 1) tm_release();
    return false;
  };
  bool lost = !arrived_all(stage.wait(0), bar);   // (also twiddles, plainly loaded rows)
  if (lost && Q == 1) return;
#pragma unroll
  for (int qg = 0; qg < NP / 4; ++qg) {   // the patch o_j and the first mode's exit wave
    float ov[16];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int i = 4 * qg + u;
      const float4 o = stage.patch(geo.row(i), geo.col(i), fy, fx);
      if (o_s) st_pair<G>(o_s + pix(i), o);
      *(float4*)(ov + 4 * u) = o;
      if constexpr (!TM) oS[i * T] = o;
      v[i] = exit_wave(P[i], o);
    }
    if constexpr (TM) tc::tmem_st16(tm_o() + 16 * qg, ov);
  }
  if constexpr (TM) tc::tmem_wait_st();
  __syncthreads();   // the staged object tile is read: its place belongs to the transforms
#pragma unroll 1
  for (int k = 0; k < M; ++k) {
    if (k > 0) {
#pragma unroll
      for (int qg = 0; qg < NP / 4; ++qg) {
        float ov[16];
        if constexpr (TM) tc::tmem_ld16_wait(tm_o() + 16 * qg, ov);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          if constexpr (!TM) *(float4*)(ov + 4 * u) = oS[(4 * qg + u) * T];
          v[4 * qg + u] = exit_wave(P[4 * qg + u], *(const float4*)(ov + 4 * u));
        }
      }
    }
    geo.forward(v);
#pragma unroll
    for (int q = 0; q < NP; ++q) v[q] = fp::pscale(v[q], fp::splat(invN));
    add_intensity<G>(v, rI, k == 0);
    if (k == M - 1) break;   // the last mode's far field stays in v
    if (psi) put_far<G>(v, psi + (size_t)k * (NN / 2));
    probe_fwd(shared_mode<OPR>(a, k + 1, NN), P);
    __syncthreads();   // the tile is free for the next mode
  }

  // ---- data term: loss and the far-field factor, on the thread's own pixels ------
  if (!data_term<G, N == 64>(geo, rI, red, bar + 1, a.meas, j, a.ipred, mode, a.eps, a.loss, a.status, arrived_all)) {
    if (Q == 1) return;
    lost = true;
  }
  if (mode == MODE_FWD || a.loss_only) {
    tm_release();
    return;
  }
  settle_lost<G>(a.valid + slot, lost);

  // ---- back-propagation: chi_k = F^-1[fac Psi_k], g = sum_k conj(P_k) chi_k, h_k ----
  // The modes run last to first: the far fields written last are read first,
  // while they are still in L2.
  float2* g_s = a.g_s + slotNN;
  float2* h_s = a.h_s + slotNN * M;
#pragma unroll 1
  for (int k = M - 1; k >= 0; --k) {
    const float2* Pk = shared_mode<OPR>(a, k, NN);
    if (k < M - 1) get_far<G>(v, psi + (size_t)k * (NN / 2));
    mul_factor<G>(v, rI);
    __syncthreads();   // the tile is free
    geo.inverse(v);
    if (k == 0) G::pixel_sync();   // the line's units are read: g may overwrite them
    float4 Pr[D];   // the probe pairs, D loads ahead
#pragma unroll
    for (int q = 0; q < D; ++q) Pr[q] = probe_back(Pk, q);
#pragma unroll
    for (int qg = 0; qg < NP / 2; ++qg) {
      float ov[8], gv[8];
      if constexpr (TM) {
        if (k < M - 1)
          tc::tmem_ld8x2_wait(tm_o() + 8 * qg, ov, tm_o() + TG + 8 * qg, gv);
        else
          tc::tmem_ld8_wait(tm_o() + 8 * qg, ov);
      } else {
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          *(float4*)(ov + 4 * u) = oS[(2 * qg + u) * T];
          if (k < M - 1) *(float4*)(gv + 4 * u) = ld_pair<G>(g_s + pix(2 * qg + u));
        }
      }
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int q = 2 * qg + u;
        const float4 P2 = Pr[q % D];
        if (q + D < NP) Pr[q % D] = probe_back(Pk, q + D);
        const float2 x0 = make_float2(v[q].re.x, v[q].im.x), x1 = make_float2(v[q].re.y, v[q].im.y);
        float2 g0 = cmulc(make_float2(P2.x, P2.y), x0), g1 = cmulc(make_float2(P2.z, P2.w), x1);
        if (k < M - 1) {
          g0.x += gv[4 * u]; g0.y += gv[4 * u + 1]; g1.x += gv[4 * u + 2]; g1.y += gv[4 * u + 3];
        }
        const float2 h0 = cmulc(make_float2(ov[4 * u], ov[4 * u + 1]), x0);
        const float2 h1 = cmulc(make_float2(ov[4 * u + 2], ov[4 * u + 3]), x1);
        stcs_pair<G>(h_s + (size_t)k * NN + pix(q), make_float4(h0.x, h0.y, h1.x, h1.y));
        const float4 g4 = make_float4(g0.x, g0.y, g1.x, g1.y);
        if (!TM || k == 0) st_pair<G>(g_s + pix(q), g4);
        if (k == 0) tile[geo.pixel_unit(q)] = g4;   // (re, im) pairs, for the scatter
        *(float4*)(gv + 4 * u) = g4;
      }
      if constexpr (TM)
        if (k > 0) tc::tmem_st8(tm_o() + TG + 8 * qg, gv);
    }
    if (TM && k > 0) tc::tmem_wait_st();
  }
  __syncthreads();
  const float2* gt = (const float2*)tile;
  overlap_add<N, LR, T, OPR>(a, slot, j, y0, ty, tx, fy, fx, p0, (float*)rI, red,
                             [&](int y, int x) { return gt[G::pixel_slot(y, x)]; });
  tm_release();
}

template <class G, bool OPR>
cudaError_t launch_pass1_pair(const BatchArgs& a, cudaStream_t s) {
  constexpr size_t sm = PairSmem<G>::bytes;
  static unsigned long long done = 0;
  cudaError_t e = smem_optin(k_pass1_pair<G, OPR>, sm, &done);
  if (e != cudaSuccess) return e;
  if (a.nb <= 0) return cudaSuccess;
  if constexpr (G::Q == 1) {
    return launch_pdl(k_pass1_pair<G, OPR>, dim3(a.nb), dim3(G::T), sm, s, a);
  } else {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(G::Q * a.nb));
    cfg.blockDim = dim3(G::T);
    cfg.dynamicSmemBytes = sm;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = G::Q;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_pass1_pair<G, OPR>, a);
  }
}

// The window's geometry.
template <int N>
using PairGeo = std::conditional_t<(N > 128), fp::ClFft<(N > 128 ? N : 256)>, OneCta<(N > 128 ? 128 : N)>>;

}  // namespace ptycho
