// The packed line-pair 2-D FFT of fft_pair.cuh for windows larger than one
// CTA's shared memory (192 and 256): a cluster of Q = N / 32 CTAs holds the
// tile, 32 rows each.
//
// The forward transform takes rows first, then columns (the inverse columns,
// then rows), with the line transforms and order of operations of fft.cuh. A
// row pass packs two rows until its exchange and two neighbouring columns
// after it, and writes every result straight into the shared memory of the CTA
// that owns its column (16 bytes through distributed shared memory): the
// transposition costs one remote write per unit instead of a local write, a
// remote read and a second local write, and its barriers overlap the
// R-point DFT between the exchange and that write. Per transform there are two
// cluster barriers: one after which every CTA's tile may be overwritten (its
// exchange is in registers), one after which every unit has arrived.
//   forward, rows:    pixels of two rows in registers -> remote column units
//   forward, columns: column units -> far field in registers: columns 2p,
//                     2p + 1 of the CTA's 32, rows n + R1 s + R2 k1
//   inverse:          the mirror image
// Against row passes over the tile, a transpose in rounds of remote reads, and
// row passes again (one line per lane group) a 256^2 transform needs half the
// shared-memory wavefronts and a quarter of the cluster barriers.
#pragma once
#include <cooperative_groups.h>

#include "fft_pair.cuh"

namespace ptycho {
namespace fp {
namespace cg = cooperative_groups;

template <int DIR> struct PDft<3, DIR> {
  // X0 = v0 + (v1 + v2); X1,2 = v0 - (v1 + v2)/2 +- i DIR sin(2 pi / 3) (v1 - v2)
  template <class V> __device__ __forceinline__ static void run(V& v) {
    const float2 s3 = splat(DIR * 0.86602540378443865f), mh = splat(-0.5f);
    const C2 t1 = padd(v[1], v[2]), t2 = psub(v[1], v[2]);
    const C2 m = {fma2(mh, t1.re, v[0].re), fma2(mh, t1.im, v[0].im)};
    v[0] = padd(v[0], t1);
    v[1] = {fma2(neg2(s3), t2.im, m.re), fma2(s3, t2.re, m.im)};
    v[2] = {fma2(s3, t2.im, m.re), fma2(neg2(s3), t2.re, m.im)};
  }
};

// a * exp(DIR i m pi / 12), m compile-time
template <int DIR, int m>
__device__ __forceinline__ C2 ptw24(C2 a) {
  constexpr int mm = m % 24;
  if constexpr (mm == 0) return a;
  else if constexpr (mm == 6) return prot90<DIR>(a);
  else if constexpr (mm == 12) return {neg2(a.re), neg2(a.im)};
  else {
    constexpr float c15 = 0.96592582628906829f, s15 = 0.25881904510252076f;
    constexpr float c30 = 0.86602540378443865f, c45 = 0.70710678118654752f;
    constexpr float cs[24] = {1.f,  c15,  c30,  c45,  0.5f,  s15,  0.f, -s15, -0.5f, -c45, -c30, -c15,
                              -1.f, -c15, -c30, -c45, -0.5f, -s15, 0.f, s15,  0.5f,  c45,  c30,  c15};
    constexpr float sn[24] = {0.f,  s15,  0.5f,  c45,  c30,  c15,  1.f,  c15,  c30,  c45,  0.5f,  s15,
                              0.f, -s15, -0.5f, -c45, -c30, -c15, -1.f, -c15, -c30, -c45, -0.5f, -s15};
    return pmul(a, cs[mm], DIR < 0 ? -sn[mm] : sn[mm]);
  }
}

template <int DIR> struct PDft<24, DIR> {
  // n = b + 3a, k = k1 + 8k2: X[k] = sum_b W3^(b k2) W24^(b k1) sum_a W8^(a k1) v[b + 3a]
  template <class V> __device__ __forceinline__ static void run(V& v) {
    C2 y[3][8];
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      C2 t[8];
#pragma unroll
      for (int a = 0; a < 8; ++a) t[a] = v[b + 3 * a];
      PDft<8, DIR>::run(t);
#pragma unroll
      for (int k1 = 0; k1 < 8; ++k1) y[b][k1] = t[k1];
    }
    y[1][1] = ptw24<DIR, 1>(y[1][1]); y[1][2] = ptw24<DIR, 2>(y[1][2]); y[1][3] = ptw24<DIR, 3>(y[1][3]);
    y[1][4] = ptw24<DIR, 4>(y[1][4]); y[1][5] = ptw24<DIR, 5>(y[1][5]); y[1][6] = ptw24<DIR, 6>(y[1][6]);
    y[1][7] = ptw24<DIR, 7>(y[1][7]);
    y[2][1] = ptw24<DIR, 2>(y[2][1]); y[2][2] = ptw24<DIR, 4>(y[2][2]); y[2][3] = ptw24<DIR, 6>(y[2][3]);
    y[2][4] = ptw24<DIR, 8>(y[2][4]); y[2][5] = ptw24<DIR, 10>(y[2][5]); y[2][6] = ptw24<DIR, 12>(y[2][6]);
    y[2][7] = ptw24<DIR, 14>(y[2][7]);
#pragma unroll
    for (int k1 = 0; k1 < 8; ++k1) {
      C2 t[3] = {y[0][k1], y[1][k1], y[2][k1]};
      PDft<3, DIR>::run(t);
#pragma unroll
      for (int k2 = 0; k2 < 3; ++k2) v[k1 + 8 * k2] = t[k2];
    }
  }
};

template <int N> struct ClCfg;
template <> struct ClCfg<192> { static constexpr int R1 = 8, R2 = 24, SH = 3; };
template <> struct ClCfg<256> { static constexpr int R1 = 16, R2 = 16, SH = 4; };

// One thread's view of the cluster's tile: line pair p of its CTA (rows 2p,
// 2p + 1 by rows; columns 2p, 2p + 1 of the CTA's by columns) and lane n of it.
template <int N_>
struct ClFft {
  using C = ClCfg<N_>;
  static constexpr int N = N_, R1 = C::R1, R2 = C::R2, S = R2 / R1, LR = 32, Q = N / LR, T = LR / 2 * R1;
  static constexpr int NP = R2;         // pixel pairs per thread
  static constexpr bool VERT = true;    // a pixel pair is two rows of one column
  static_assert(R1 * R2 == N && S * R1 == R2 && 32 % R1 == 0, "line split; a line's lanes share a warp");
  static constexpr int TW = R1 * (R2 + 1);
  __device__ __forceinline__ static void fill_twiddles(float2* tw) { make_line_twiddles<N, R1, R2>(tw); }

  float4* tile;
  const float2* tw;
  int p, n, q;
  __device__ __forceinline__ ClFft(float4* tile_, const float2* tw_)
      : tile(tile_), tw(tw_), p((int)threadIdx.x / R1), n((int)threadIdx.x % R1),
        q((int)cg::this_cluster().block_rank()) {}

  // pixel 0 of pair i (CTA-local row; pixel 1 is the row below), and the far
  // field of register i = k1 S + s (columns far_x() and far_x() + 1)
  __device__ __forceinline__ int row(int) const { return 2 * p; }
  __device__ __forceinline__ int col(int i) const { return n + R1 * i; }
  __device__ __forceinline__ int far_y(int i) const { return n + R1 * (i % S) + R2 * (i / S); }
  __device__ __forceinline__ int far_x() const { return 2 * p; }
  __device__ __forceinline__ int pixel_unit(int i) const { return unit(p, n, R1 * i); }
  __device__ __forceinline__ static int pixel_slot(int y, int x) { return 2 * unit(y >> 1, x) + (y & 1); }
  // joins the lanes that share the units of this thread's pixels
  __device__ __forceinline__ static void pixel_sync() { __syncwarp(); }

  // unit i of a line pair: 8 lanes that differ in the low three bits of i, or
  // in the next ones (SH upwards), or in bit 0 and the line, hit all bank groups
  __host__ __device__ static constexpr int unit(int line, int i) {
    return line * N + (i ^ ((i >> C::SH) & 7) ^ ((line & 3) << 1));
  }
  __device__ __forceinline__ static int unit(int line, int rt, int ct) {   // i = rt + ct
    if constexpr ((N & (N - 1)) == 0) {   // disjoint bits
      const int b = unit(line, rt), c = unit(0, ct);
      return (b ^ (c & 7)) + (c & ~7);
    } else {
      return unit(line, rt + ct);
    }
  }
  __device__ __forceinline__ C2 get(int u) const {
    const float4 x = tile[u];
    return {make_float2(x.x, x.y), make_float2(x.z, x.w)};
  }
  __device__ __forceinline__ static void put(float4* t, int u, C2 v) {
    t[u] = make_float4(v.re.x, v.re.y, v.im.x, v.im.y);
  }
  __device__ __forceinline__ void put_t(int ux, int uy, C2 a, C2 b) const {
    tile[ux] = make_float4(a.re.x, b.re.x, a.im.x, b.im.x);
    tile[uy] = make_float4(a.re.y, b.re.y, a.im.y, b.im.y);
  }
  // unit (line pair L of the whole window, i) in its owner's shared memory
  __device__ __forceinline__ void send(int L, int i, C2 v) const {
    put(cg::this_cluster().map_shared_rank(tile, L / (LR / 2)), unit(L % (LR / 2), i), v);
  }
  template <int DIR>   // v[k] *= exp(DIR 2 pi i n k / N)
  __device__ __forceinline__ void twiddle(C2 (&v)[R2]) const {
    float2 t[R2];
    LineTwiddles<R1, R2>::twiddles(t, tw, n);
#pragma unroll
    for (int k = 1; k < R2; ++k)
      v[k] = DIR < 0 ? pmul(v[k], t[k].x, t[k].y) : pmulc(v[k], {splat(t[k].x), splat(t[k].y)});
  }

  // In: v[i] = pixels (row(i), col(i)), (row(i) + 1, col(i)). Out: v[i] = the
  // unnormalised far field. The CTA's tile must be free on entry.
  __device__ __forceinline__ void forward(C2 (&v)[R2]) const {
    cg::cluster_group cluster = cg::this_cluster();
    PDft<R2, -1>::run(v);
    twiddle<-1>(v);
#pragma unroll
    for (int m = 0; m < R2 / 2; ++m)
      put_t(unit(p, R2 * n, 2 * m), unit(p, R2 * n, 2 * m + 1), v[2 * m], v[2 * m + 1]);
    __syncwarp();
    // row 2p + g % 2, columns k2 = 2 (g / 2) and the next, g = n + R1 s
    C2 w[S][R1];
#pragma unroll
    for (int s = 0; s < S; ++s)
#pragma unroll
      for (int n1 = 0; n1 < R1; ++n1) w[s][n1] = get(unit(p, n, R1 * s + R2 * n1));
    cluster.barrier_arrive();
#pragma unroll
    for (int s = 0; s < S; ++s) PDft<R1, -1>::run(w[s]);
    cluster.barrier_wait();
#pragma unroll
    for (int s = 0; s < S; ++s) {
      const int g = n + R1 * s;
#pragma unroll
      for (int k1 = 0; k1 < R1; ++k1) send((g >> 1) + R2 / 2 * k1, LR * q + 2 * p + (g & 1), w[s][k1]);
    }
    cluster.sync();
#pragma unroll
    for (int n2 = 0; n2 < R2; ++n2) v[n2] = get(unit(p, n, R1 * n2));
    PDft<R2, -1>::run(v);
    twiddle<-1>(v);
#pragma unroll
    for (int k2 = 0; k2 < R2; ++k2) put(tile, unit(p, n, R1 * k2), v[k2]);
    __syncwarp();
#pragma unroll
    for (int s = 0; s < S; ++s) {   // rows k2 = n + R1 s, + R2 k1
      C2 x[R1];
#pragma unroll
      for (int n1 = 0; n1 < R1; ++n1) x[n1] = get(unit(p, R1 * n, R1 * R1 * s + n1));
      PDft<R1, -1>::run(x);
#pragma unroll
      for (int k1 = 0; k1 < R1; ++k1) v[k1 * S + s] = x[k1];
    }
  }

  // The mirror image (times N^2), from the layout forward leaves to the one it takes.
  __device__ __forceinline__ void inverse(C2 (&v)[R2]) const {
    cg::cluster_group cluster = cg::this_cluster();
#pragma unroll
    for (int s = 0; s < S; ++s) {
      C2 x[R1];
#pragma unroll
      for (int k1 = 0; k1 < R1; ++k1) x[k1] = v[k1 * S + s];
      PDft<R1, 1>::run(x);
#pragma unroll
      for (int m = 0; m < R1 / 2; ++m)
        put_t(unit(p, R1 * n, R1 * R1 * s + 2 * m), unit(p, R1 * n, R1 * R1 * s + 2 * m + 1), x[2 * m], x[2 * m + 1]);
    }
    __syncwarp();
    // column 2p + n % 2, rows 2 (n / 2) + R1 n2 and the next
#pragma unroll
    for (int k2 = 0; k2 < R2; ++k2) v[k2] = get(unit(p, n, R1 * k2));
    cluster.barrier_arrive();
    {
      C2 t[R2];
      pair_twiddles<R2>(t, tw, n & ~1);
#pragma unroll
      for (int k = 1; k < R2; ++k) v[k] = pmulc(v[k], t[k]);
    }
    PDft<R2, 1>::run(v);
    cluster.barrier_wait();
#pragma unroll
    for (int n2 = 0; n2 < R2; ++n2) send((n >> 1) + R1 / 2 * n2, LR * q + 2 * p + (n & 1), v[n2]);
    cluster.sync();
#pragma unroll
    for (int s = 0; s < S; ++s) {
      C2 x[R1];
#pragma unroll
      for (int k1 = 0; k1 < R1; ++k1) x[k1] = get(unit(p, n, R1 * s + R2 * k1));
      PDft<R1, 1>::run(x);
#pragma unroll
      for (int n1 = 0; n1 < R1; ++n1) put(tile, unit(p, n, R1 * s + R2 * n1), x[n1]);
    }
    __syncwarp();
#pragma unroll
    for (int k2 = 0; k2 < R2; ++k2) v[k2] = get(unit(p, R2 * n, k2));
    twiddle<1>(v);
    PDft<R2, 1>::run(v);
  }
};

}  // namespace fp
}  // namespace ptycho
