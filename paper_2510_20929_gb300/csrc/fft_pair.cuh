// Shared-memory 2-D FFT of one N x N complex64 tile per CTA, two lines at a
// time in packed FP32 (sm_103a).
//
// The far-field propagator of the ptychographic forward model (Pty-Chi,
// Sec. 2.1; Eq. 4's F(o, p, Lambda)) and its inverse, with the line transforms
// of fft.cuh (the same radices, twiddles and order of operations, so the same
// values), for the windows whose whole tile one CTA holds. What differs: every
// thread carries R2 points of TWO lines as packed pairs (re_a, re_b), (im_a,
// im_b), so each add, multiply and fused multiply-add is one f32x2 instruction
// for both (they share every twiddle), and each shared-memory access moves the
// 16 bytes of a pair. One line at a time the 1-D transforms were bound by issue
// slots (540 instructions per 16 points) and by shared-memory wavefronts.
//
// A line of N = R1 * R2 points belongs to R1 threads. The first half of a
// forward line transform is an R2-point DFT of x[n + R1 n2] and the twiddles
// W^(n k2) in thread n; the lanes of the line exchange; the second half is the
// R1-point DFT over n, giving X[k2 + R2 k1]. The inverse mirrors it. The
// packing may change at an exchange, where a thread holds 2 x 2 blocks (two
// lines x two neighbouring indices) and writes them transposed:
//   forward, columns: two columns packed; then two rows k2, k2 + 1 of one column;
//   forward, rows:    two rows packed throughout; the far field of a thread is
//                     rows 2p, 2p + 1 at columns S n + s + R2 k1 (S = R2 / R1);
//   inverse, rows:    two rows packed; then two columns n, n + 1 of one row;
//   inverse, columns: two columns packed throughout.
// So pixels enter and leave in registers by two adjacent columns of one row
// (16 bytes, natural order, for the caller's global accesses), the tile is
// never stored by the thread that reads it back, and a far-field element stays
// with the thread that made it: the far field can rest in any per-thread
// layout between the two transforms.
//
// The tile holds N * N / 2 units of 16 bytes: by rows, unit (rp, c) = pixels
// (2 rp, c), (2 rp + 1, c) as (re, re, im, im); by columns, unit (r, cp) =
// pixels (r, 2 cp), (r, 2 cp + 1). Every thread writes the second half's
// results over the units it read for it, and the exchange stays inside the
// units of the line pair, so one synchronisation of the line's own threads per
// pass is enough. By rows these are lanes of one warp; by columns a warp spans
// 8 line pairs (128 contiguous bytes of each pixel row, so that the caller's
// global accesses are whole lines: at half lines the pass was bound by the rate
// of its L2 requests), and at R1 = 8 the two warps of a line meet at a named
// barrier. Both unit maps XOR the low three bits with linear functions of
// the upper ones, chosen so that the quarter-warps (8 lanes of 16 bytes) of
// every access hit all eight 16-byte bank groups.
#pragma once
#include "fft.cuh"

namespace ptycho {
namespace fp {

struct C2 {   // two complex values: (re_a, re_b), (im_a, im_b)
  float2 re, im;
};

__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __fadd2_rn(a, neg2(b)); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 splat(float v) { return make_float2(v, v); }

__device__ __forceinline__ C2 padd(C2 a, C2 b) { return {add2(a.re, b.re), add2(a.im, b.im)}; }
__device__ __forceinline__ C2 psub(C2 a, C2 b) { return {sub2(a.re, b.re), sub2(a.im, b.im)}; }
__device__ __forceinline__ C2 pscale(C2 a, float2 s) { return {mul2(a.re, s), mul2(a.im, s)}; }
// a * (c + i s), the same twiddle for both lines
__device__ __forceinline__ C2 pmul(C2 a, float c, float s) {
  const float2 cc = splat(c), ss = splat(s);
  return {fma2(a.re, cc, neg2(mul2(a.im, ss))), fma2(a.re, ss, mul2(a.im, cc))};
}
// a * t and a * conj(t), with a twiddle per line
__device__ __forceinline__ C2 pmul(C2 a, C2 t) {
  return {fma2(a.re, t.re, neg2(mul2(a.im, t.im))), fma2(a.re, t.im, mul2(a.im, t.re))};
}
__device__ __forceinline__ C2 pmulc(C2 a, C2 t) {
  return {fma2(a.re, t.re, mul2(a.im, t.im)), fma2(a.im, t.re, neg2(mul2(a.re, t.im)))};
}
template <int DIR>
__device__ __forceinline__ C2 prot90(C2 a) {   // a * exp(DIR i pi / 2)
  return DIR < 0 ? C2{a.im, neg2(a.re)} : C2{neg2(a.im), a.re};
}
// a * exp(DIR i m pi / 8), m compile-time
template <int DIR, int m>
__device__ __forceinline__ C2 ptw16(C2 a) {
  constexpr int mm = m & 15;
  if constexpr (mm == 0) return a;
  else if constexpr (mm == 4) return prot90<DIR>(a);
  else {
    constexpr float cs[16] = {1.f, PT_C1, PT_C2, PT_S1, 0.f, -PT_S1, -PT_C2, -PT_C1,
                              -1.f, -PT_C1, -PT_C2, -PT_S1, 0.f, PT_S1, PT_C2, PT_C1};
    constexpr float sn[16] = {0.f, PT_S1, PT_C2, PT_C1, 1.f, PT_C1, PT_C2, PT_S1,
                              0.f, -PT_S1, -PT_C2, -PT_C1, -1.f, -PT_C1, -PT_C2, -PT_S1};
    return pmul(a, cs[mm], DIR < 0 ? -sn[mm] : sn[mm]);
  }
}

// In-register DFTs of R packed points, natural order, sign DIR.
template <int R, int DIR> struct PDft;
template <int DIR> struct PDft<2, DIR> {
  template <class V> __device__ __forceinline__ static void run(V& v) {
    const C2 a = v[0], b = v[1];
    v[0] = padd(a, b);
    v[1] = psub(a, b);
  }
};
template <int DIR> struct PDft<4, DIR> {
  template <class V> __device__ __forceinline__ static void run(V& v) {
    const C2 t0 = padd(v[0], v[2]), t1 = psub(v[0], v[2]);
    const C2 t2 = padd(v[1], v[3]), d = psub(v[1], v[3]);
    v[0] = padd(t0, t2);
    v[2] = psub(t0, t2);
    // t1 +- exp(DIR i pi/2) d
    const C2 p = {sub2(t1.re, d.im), add2(t1.im, d.re)}, m = {add2(t1.re, d.im), sub2(t1.im, d.re)};
    v[1] = DIR < 0 ? m : p;
    v[3] = DIR < 0 ? p : m;
  }
};
template <int DIR> struct PDft<8, DIR> {
  template <class V> __device__ __forceinline__ static void run(V& v) {
    C2 e[4] = {v[0], v[2], v[4], v[6]};
    C2 o[4] = {v[1], v[3], v[5], v[7]};
    PDft<4, DIR>::run(e);
    PDft<4, DIR>::run(o);
    o[1] = ptw16<DIR, 2>(o[1]);
    o[2] = ptw16<DIR, 4>(o[2]);
    o[3] = ptw16<DIR, 6>(o[3]);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      v[k] = padd(e[k], o[k]);
      v[k + 4] = psub(e[k], o[k]);
    }
  }
};
template <int DIR> struct PDft<16, DIR> {
  // n = b + 4a, k = k1 + 4k2: X[k] = sum_b W16^(b k1) W4^(b k2) sum_a W4^(a k1) v[b + 4a]
  template <class V> __device__ __forceinline__ static void run(V& v) {
    C2 y[4][4];
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      C2 t[4] = {v[b], v[b + 4], v[b + 8], v[b + 12]};
      PDft<4, DIR>::run(t);
#pragma unroll
      for (int k1 = 0; k1 < 4; ++k1) y[b][k1] = t[k1];
    }
    y[1][1] = ptw16<DIR, 1>(y[1][1]);
    y[1][2] = ptw16<DIR, 2>(y[1][2]);
    y[1][3] = ptw16<DIR, 3>(y[1][3]);
    y[2][1] = ptw16<DIR, 2>(y[2][1]);
    y[2][2] = ptw16<DIR, 4>(y[2][2]);
    y[2][3] = ptw16<DIR, 6>(y[2][3]);
    y[3][1] = ptw16<DIR, 3>(y[3][1]);
    y[3][2] = ptw16<DIR, 6>(y[3][2]);
    y[3][3] = ptw16<DIR, 9>(y[3][3]);
#pragma unroll
    for (int k1 = 0; k1 < 4; ++k1) {
      C2 t[4] = {y[0][k1], y[1][k1], y[2][k1], y[3][k1]};
      PDft<4, DIR>::run(t);
#pragma unroll
      for (int k2 = 0; k2 < 4; ++k2) v[k1 + 4 * k2] = t[k2];
    }
  }
};

// The twiddles of fft.cuh (W^(n k), k = 1..R2-1: four from the table, the rest
// as products) for lane indices n and n + 1, packed.
template <int R2>
__device__ __forceinline__ void pair_twiddles(C2 (&t)[R2], const float2* tw, int n) {
  constexpr int L4 = R2 - 1 < 4 ? R2 - 1 : 4;
#pragma unroll
  for (int k = 1; k <= L4; ++k) {
    const float2 a = tw[n * (R2 + 1) + k], b = tw[(n + 1) * (R2 + 1) + k];
    t[k] = {make_float2(a.x, b.x), make_float2(a.y, b.y)};
  }
#pragma unroll
  for (int k = 5; k < R2; ++k) {
    const int a = k & ~3, b = k & 3;
    t[k] = b == 0 ? pmul(t[a - 4], t[4]) : pmul(t[a], t[b]);
  }
}

// Line split (that of fft.cuh) and the unit maps' XOR terms. By columns a
// quarter warp covers 8 consecutive line pairs of one lane index n; by rows 8
// line pairs (R1 = 4), or 4 line pairs of two n that differ in bit 0 (R1 = 8).
template <int N> struct Cfg;
template <> struct Cfg<16> {
  static constexpr int R1 = 4, R2 = 4;
  __host__ __device__ static constexpr int rsw(int rp, int c) { return (rp & 7) ^ ((c >> 3) & 1); }
  __host__ __device__ static constexpr int csw(int r, int) { return (r >> 1) & 7; }
};
template <> struct Cfg<32> {
  static constexpr int R1 = 4, R2 = 8;
  __host__ __device__ static constexpr int rsw(int rp, int c) { return (rp & 7) ^ ((c >> 3) & 1); }
  __host__ __device__ static constexpr int csw(int r, int) { return (r >> 1) & 7; }
};
template <> struct Cfg<64> {
  static constexpr int R1 = 8, R2 = 8;
  __host__ __device__ static constexpr int rsw(int rp, int c) { return ((c >> 3) & 1) ^ ((rp & 3) << 1); }
  __host__ __device__ static constexpr int csw(int r, int) { return (r & 2) ^ (((r >> 2) & 1) * 5); }
};
template <> struct Cfg<128> {
  static constexpr int R1 = 8, R2 = 16;
  __host__ __device__ static constexpr int rsw(int rp, int c) { return (((c >> 3) ^ (c >> 4)) & 1) ^ ((rp & 3) << 1); }
  __host__ __device__ static constexpr int csw(int r, int cp) { return ((cp >> 3) & 1) ^ (r & 6); }
};

template <int N>
struct Fft {
  using C = Cfg<N>;
  static constexpr int R1 = C::R1, R2 = C::R2, S = R2 / R1, G = 32 / R1, T = N / 2 * R1;
  static_assert(R1 * R2 == N && S * R1 == R2 && R1 % 2 == 0 && T % 32 == 0, "line split");
  static_assert(R1 == FftCfg<N>::R1 && R2 == FftCfg<N>::R2, "the line split of fft.cuh");
  static constexpr int UNITS = N * N / 2;   // 16-byte units of the tile

  // this thread's index within its line, and its line pair, by rows and by columns
  __device__ __forceinline__ static int row_lane() { return (int)(threadIdx.x & 31) / G; }
  __device__ __forceinline__ static int row_pair() { return (int)(threadIdx.x >> 5) * G + (int)(threadIdx.x & 31) % G; }
  __device__ __forceinline__ static int col_lane() { return (int)threadIdx.x / 8 % R1; }
  __device__ __forceinline__ static int col_pair() { return (int)threadIdx.x / (8 * R1) * 8 + (int)(threadIdx.x & 7); }
  // joins the threads of a column line (8 line pairs: 8 R1 threads)
  __device__ __forceinline__ static void col_sync() {
    if constexpr (R1 == 4) __syncwarp();
    else asm volatile("bar.sync %0, %1;\n" ::"r"(1 + (int)threadIdx.x / (8 * R1)), "n"(8 * R1) : "memory");
  }
  // far-field column of register k1 S + s of row lane n
  __device__ __forceinline__ static int far_col(int n, int i) { return S * n + i % S + R2 * (i / S); }

  // unit of pixels (2 rp, c), (2 rp + 1, c); and of pixels (r, 2 cp), (r, 2 cp + 1)
  __host__ __device__ static constexpr int rowu(int rp, int c) { return rp * N + (c ^ C::rsw(rp, c)); }
  __host__ __device__ static constexpr int colu(int r, int cp) { return r * (N / 2) + (cp ^ C::csw(r, cp)); }
  // unit of the sum of two index pairs with disjoint bits, from the units of
  // the per-thread part and the compile-time part: the low three bits combine
  // by XOR, the rest by addition
  __device__ __forceinline__ static int at(int base, int ct) { return (base ^ (ct & 7)) + (ct & ~7); }

  __device__ __forceinline__ static void put(float4* t, int u, C2 v) {
    t[u] = make_float4(v.re.x, v.re.y, v.im.x, v.im.y);
  }
  __device__ __forceinline__ static C2 get(const float4* t, int u) {
    const float4 x = t[u];
    return {make_float2(x.x, x.y), make_float2(x.z, x.w)};
  }
  // the 2 x 2 block of packed values a, b transposed into two units
  __device__ __forceinline__ static void put_t(float4* t, int ux, int uy, C2 a, C2 b) {
    t[ux] = make_float4(a.re.x, b.re.x, a.im.x, b.im.x);
    t[uy] = make_float4(a.re.y, b.re.y, a.im.y, b.im.y);
  }

  // W^(n k), k = 1..R2-1: the first four from the table, the rest as products
  // (fft.cuh's); one lane index for both lines of the pack
  __device__ __forceinline__ static void twiddles(float2 (&t)[R2], const float2* tw, int n) {
    LineTwiddles<R1, R2>::twiddles(t, tw, n);
  }
  // Forward, first pass: columns. In: v[n2] = pixels (n + R1 n2, 2p), (.., 2p + 1).
  // Leaves the half-transformed tile in row units.
  __device__ __forceinline__ static void fwd_cols(C2 (&v)[R2], float4* tile, int p, int n, const float2* tw) {
    PDft<R2, -1>::run(v);
    {
      float2 t[R2];
      twiddles(t, tw, n);
#pragma unroll
      for (int k = 1; k < R2; ++k) v[k] = pmul(v[k], t[k].x, t[k].y);
    }
    const int wb = rowu(R2 / 2 * n, 2 * p);
#pragma unroll
    for (int m = 0; m < R2 / 2; ++m)
      put_t(tile, at(wb, rowu(m, 0)), at(wb, rowu(m, 0) ^ 1), v[2 * m], v[2 * m + 1]);
    col_sync();
    // column 2p + n % 2, rows k2 = 2m, 2m + 1 with m = n / 2 + R1 / 2 s
    const int rb = rowu(n >> 1, 2 * p + (n & 1));
#pragma unroll
    for (int s = 0; s < S; ++s) {
      C2 w[R1];
#pragma unroll
      for (int n1 = 0; n1 < R1; ++n1) w[n1] = get(tile, at(rb, rowu(R1 / 2 * s + R2 / 2 * n1, 0)));
      PDft<R1, -1>::run(w);
#pragma unroll
      for (int k1 = 0; k1 < R1; ++k1) put(tile, at(rb, rowu(R1 / 2 * s + R2 / 2 * k1, 0)), w[k1]);
    }
  }
  // Forward, second pass: rows. Out: v[k1 S + s] = far field of rows 2p, 2p + 1, column far_col(n, k1 S + s).
  __device__ __forceinline__ static void fwd_rows(C2 (&v)[R2], float4* tile, int p, int n, const float2* tw) {
    const int wb = rowu(p, n), rb = rowu(p, R1 * S * n);
#pragma unroll
    for (int n2 = 0; n2 < R2; ++n2) v[n2] = get(tile, at(wb, rowu(0, R1 * n2)));
    PDft<R2, -1>::run(v);
    {
      float2 t[R2];
      twiddles(t, tw, n);
#pragma unroll
      for (int k = 1; k < R2; ++k) v[k] = pmul(v[k], t[k].x, t[k].y);
    }
#pragma unroll
    for (int k2 = 0; k2 < R2; ++k2) put(tile, at(wb, rowu(0, R1 * k2)), v[k2]);
    __syncwarp();
#pragma unroll
    for (int s = 0; s < S; ++s) {
      C2 w[R1];
#pragma unroll
      for (int n1 = 0; n1 < R1; ++n1) w[n1] = get(tile, at(rb, rowu(0, n1 + R1 * s)));
      PDft<R1, -1>::run(w);
#pragma unroll
      for (int k1 = 0; k1 < R1; ++k1) v[k1 * S + s] = w[k1];
    }
  }
  // Inverse, first pass: rows, from the layout fwd_rows leaves.
  __device__ __forceinline__ static void inv_rows(C2 (&v)[R2], float4* tile, int p, int n, const float2* tw) {
    const int wb = colu(2 * p, R1 / 2 * S * n);
#pragma unroll
    for (int s = 0; s < S; ++s) {
      C2 w[R1];
#pragma unroll
      for (int k1 = 0; k1 < R1; ++k1) w[k1] = v[k1 * S + s];
      PDft<R1, 1>::run(w);
#pragma unroll
      for (int m = 0; m < R1 / 2; ++m) {
        const int ct = colu(0, m + R1 / 2 * s);
        put_t(tile, at(wb, ct), at(wb, ct ^ colu(1, 0)), w[2 * m], w[2 * m + 1]);
      }
    }
    __syncwarp();
    // row 2p + n / (R1 / 2), columns n1 = 2m, 2m + 1 with m = n % (R1 / 2)
    const int m = n % (R1 / 2), rb = colu(2 * p + n / (R1 / 2), m);
#pragma unroll
    for (int k2 = 0; k2 < R2; ++k2) v[k2] = get(tile, at(rb, colu(0, R1 / 2 * k2)));
    {
      C2 t[R2];
      pair_twiddles<R2>(t, tw, 2 * m);
#pragma unroll
      for (int k = 1; k < R2; ++k) v[k] = pmulc(v[k], t[k]);
    }
    PDft<R2, 1>::run(v);
#pragma unroll
    for (int n2 = 0; n2 < R2; ++n2) put(tile, at(rb, colu(0, R1 / 2 * n2)), v[n2]);
  }
  // Inverse, second pass: columns. Out: v[n2] = pixels (n + R1 n2, 2p), (.., 2p + 1), times N^2.
  __device__ __forceinline__ static void inv_cols(C2 (&v)[R2], float4* tile, int p, int n, const float2* tw) {
    const int wb = colu(S * n, p), rb = colu(R2 * n, p);
#pragma unroll
    for (int s = 0; s < S; ++s) {
      C2 w[R1];
#pragma unroll
      for (int k1 = 0; k1 < R1; ++k1) w[k1] = get(tile, at(wb, colu(s + R2 * k1, 0)));
      PDft<R1, 1>::run(w);
#pragma unroll
      for (int n1 = 0; n1 < R1; ++n1) put(tile, at(wb, colu(s + R2 * n1, 0)), w[n1]);
    }
    col_sync();
#pragma unroll
    for (int k2 = 0; k2 < R2; ++k2) v[k2] = get(tile, at(rb, colu(k2, 0)));
    {
      float2 t[R2];
      twiddles(t, tw, n);
#pragma unroll
      for (int k = 1; k < R2; ++k) v[k] = pmulc(v[k], {splat(t[k].x), splat(t[k].y)});
    }
    PDft<R2, 1>::run(v);
  }
};

}  // namespace fp
}  // namespace ptycho
