// The step-size pass of one minibatch: the five sums of each position's
// least-squares step (LSQML's self-adaptive step sizes, Pty-Chi Sec. 2.2), the
// FP64 2x2 solve and the alpha-weighted object update.
//
// k_pass2 and k_pass2_cluster do it position by position: a CTA (or four) per
// position, each reading the minibatch's probe direction and the probe-frame
// planes again from L2. They take as long as one position does whenever the
// minibatch leaves the GPU unfilled (window 256: 118 us from 8 positions to 32).
//
// k_step_sums and k_step_update are two launches. The first turns the loops
// round: a CTA keeps 2 T pixels of the probe frame (in registers and shared
// memory) and walks over positions, so that only their own planes and the
// accumulator's corners are left to load, and a minibatch of any size fills the
// GPU. The partial sums of four positions at a time meet in one transposing
// shuffle tree, then in FP64. The update needs every position's alpha and
// follows in bands of rows. Both are bound by the latency of the loads (2.4
// TB/s of DRAM reads at a large minibatch; bulk copies, loads one position
// ahead and staged corners all measured the same).
#pragma once
#include "kernels.cuh"
#include "launch.h"

namespace ptycho {

// FP64 solve of the damped 2x2 step-size system (the fallbacks of each step alone).
__device__ __forceinline__ void solve_step(double a11, double a12, double a22, double r1, double r2, double lam,
                                           double& aO, double& aP) {
  const double tr = 0.5 * (a11 + a22);
  const double d11 = a11 + lam * tr, d22 = a22 + lam * tr;
  const double det = d11 * d22 - a12 * a12;
  if (det > 0.0) {
    aO = (d22 * r1 - a12 * r2) / det;
    aP = (d11 * r2 - a12 * r1) / det;
  } else {
    aO = d11 > 0.0 ? r1 / d11 : 0.0;
    aP = d22 > 0.0 ? r2 / d22 : 0.0;
  }
}

// One CTA per position, two of them per SM.
constexpr int PASS2_T = 512;

template <int N, int T, bool OPR>
__global__ void __launch_bounds__(T, 1024 / T) k_pass2(Pass2Args a) {
  constexpr int NN = N * N;
  wait_prior_grid();
  __shared__ double red[32 * 5];
  __shared__ double alpha_sh;
  const int slot = blockIdx.x, tid = threadIdx.x;
  if (!a.valid[slot]) return;
  const int e = a.b0 + slot;
  const int j = a.order ? a.order[e] : e;
  int ty, tx;
  float fy, fx;
  tile_of(a.pos[2 * j], a.pos[2 * j + 1], N, a.H, a.W, ty, tx, fy, fx);
  const float w00 = (1.f - fy) * (1.f - fx), w01 = (1.f - fy) * fx, w10 = fy * (1.f - fx), w11 = fy * fx;
  const float damp = a.delta_o * __uint_as_float(a.sc->max_illum);
  const size_t slotNN = (size_t)slot * NN;
  const int M = a.M;
  const float2* g_s = a.g_s + slotNN;
  const float2* o_s = a.o_s + slotNN;
  const float2* h_s = a.h_s + slotNN * M;
  // OPR: the primary mode P_j0 and its direction sum_m w_jm dU_m differ per
  // position; Sp, Cp, Sdp and dP then hold the shared modes only
  constexpr bool opr = OPR;
  __shared__ float wsh[OPR_KMAX];
  if (opr) {
    if (tid < a.K) wsh[tid] = a.opr_w[(size_t)j * a.K + tid];
    __syncthreads();
  }
  const float2* p0 = opr ? a.p0_s + slotNN : nullptr;

  float A11 = 0.f, A12 = 0.f, A22 = 0.f, b1 = 0.f, b2 = 0.f;
  {
    // two adjacent pixels per iteration: 16-byte loads of g, o and Cp, and the
    // six accumulator corners the pair shares (half the trips of this
    // latency-bound loop); with OPR also the pair's primary mode, its
    // direction sum_m w_jm dU_m (K 16-byte loads) and h_j0
#pragma unroll 1
    for (int p = 2 * tid; p < NN; p += 2 * T) {
      const int r = p / N, c = p % N;
      const float4 g2 = __ldg((const float4*)(g_s + p));   // kept in L2: the update reads g again
      const float4 o2 = __ldcs((const float4*)(o_s + p));
      float2 d0 = make_float2(0.f, 0.f), d1 = d0;
      if (a.update_object) {
        const float4* q = a.acc + (size_t)(ty + r) * a.W + (tx + c);
        const float4 qa = __ldg(q), qb = __ldg(q + 1), qc = __ldg(q + 2);
        const float4 qd = __ldg(q + a.W), qe = __ldg(q + a.W + 1), qf = __ldg(q + a.W + 2);
        const float ia = 1.f / (qa.z + damp), ib = 1.f / (qb.z + damp), ic = 1.f / (qc.z + damp);
        const float id = 1.f / (qd.z + damp), ie = 1.f / (qe.z + damp), iF = 1.f / (qf.z + damp);
        // dO_hat at the pixel: each corner's quotient, then the bilinear weights
        d0 = make_float2(w00 * ia * qa.x + w01 * ib * qb.x + w10 * id * qd.x + w11 * ie * qe.x,
                         w00 * ia * qa.y + w01 * ib * qb.y + w10 * id * qd.y + w11 * ie * qe.y);
        d1 = make_float2(w00 * ib * qb.x + w01 * ic * qc.x + w10 * ie * qe.x + w11 * iF * qf.x,
                         w00 * ib * qb.y + w01 * ic * qc.y + w10 * ie * qe.y + w11 * iF * qf.y);
      }
      float2 sp = __ldg((const float2*)(a.Sp + p)), sdp = __ldg((const float2*)(a.Sdp + p));
      float4 cp = __ldg((const float4*)(a.Cp + p));
      if constexpr (OPR) {
        const float4 P2 = *(const float4*)(p0 + p);
        const float2 Pa = make_float2(P2.x, P2.y), Pb = make_float2(P2.z, P2.w);
        sp.x += cabs2(Pa);
        sp.y += cabs2(Pb);
        if (a.update_probe) {
          const float4 D2 = opr_pair(a.opr_dU, wsh, a.K, NN, p);
          const float2 ea = make_float2(D2.x, D2.y), eb = make_float2(D2.z, D2.w);
          const float2 ca = cmulc(Pa, ea), cb = cmulc(Pb, eb);
          cp = make_float4(cp.x + ca.x, cp.y + ca.y, cp.z + cb.x, cp.w + cb.y);
          sdp.x += cabs2(ea);
          sdp.y += cabs2(eb);
          const float4 h2 = __ldcs((const float4*)(h_s + p));
          b2 += ea.x * h2.x + ea.y * h2.y + eb.x * h2.z + eb.y * h2.w;   // Re(conj(dP_j0) h_j0)
        }
      }
      const float2 g0 = make_float2(g2.x, g2.y), g1 = make_float2(g2.z, g2.w);
      const float2 o0 = make_float2(o2.x, o2.y), o1 = make_float2(o2.z, o2.w);
      A11 += cabs2(d0) * sp.x + cabs2(d1) * sp.y;
      const float2 od0 = cmulc(d0, o0), od1 = cmulc(d1, o1);   // conj(d) o
      A12 += od0.x * cp.x - od0.y * cp.y + od1.x * cp.z - od1.y * cp.w;   // Re(conj(d) o Cp)
      A22 += cabs2(o0) * sdp.x + cabs2(o1) * sdp.y;
      b1 += d0.x * g0.x + d0.y * g0.y + d1.x * g1.x + d1.y * g1.y;       // Re(conj(d) g)
    }
  }
  if (a.update_probe) {
    // b2 = Re sum_k <dP_k, h_k> over the shared modes: their planes are
    // contiguous, two pixels per 16-byte load
    const float4* h4 = (const float4*)(h_s + (opr ? NN : 0));
    const float4* d4 = (const float4*)a.dP;
    const int Q = (opr ? M - 1 : M) * NN / 2;
    int q = tid;
    for (; q + 3 * T < Q; q += 4 * T) {      // four independent 16-byte streams per thread
      float4 dp[4], h[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        dp[u] = __ldg(d4 + q + u * T);
        h[u] = __ldcs(h4 + q + u * T);
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) b2 += dp[u].x * h[u].x + dp[u].y * h[u].y + dp[u].z * h[u].z + dp[u].w * h[u].w;
    }
    for (; q < Q; q += T) {
      const float4 dp = __ldg(d4 + q);
      const float4 h = __ldcs(h4 + q);
      b2 += dp.x * h.x + dp.y * h.y + dp.z * h.z + dp.w * h.w;   // Re(conj(dP_k) h_k)
    }
  }
  double v[5] = {A11, A12, A22, b1, b2};
  block_sum<5>(v, red);
  if (tid == 0) {
    double aO, aP;
    solve_step(v[0], v[1], v[2], v[3], v[4], a.lam, aO, aP);
    alpha_sh = aO;
    if (a.alpha_out) {
      a.alpha_out[2 * j] = aO;
      a.alpha_out[2 * j + 1] = aP;
    }
    atomicAdd(&a.sc->sum_alpha_p, aP);
    atomicAdd(&a.sc->count, 1);
  }
  __syncthreads();
  if (!a.update_object) return;
  // O += alpha_O S_j^T g / (illum + delta_O): each object pixel of the (N+1)^2 tile
  // gathers its four patch neighbours and is divided by its own preconditioner
  const float aO = (float)alpha_sh;
  const float c00 = aO * w00, c01 = aO * w01, c10 = aO * w10, c11 = aO * w11;
  constexpr int N1 = N + 1;
  if (((uintptr_t)a.obj & 15) == 0 && (a.W & 1) == 0) {
    // pairs of object pixels at even object columns, one 16-byte vector atomic
    // each (half the atomic operations); per tile row N/2 pairs and one single
    // pixel (the first when tx is odd, else the last)
    constexpr int PR = N / 2 + 1;
    const int odd = tx & 1;
    auto gat = [&](int y, int x) {
      return (y >= 0 && y < N && x >= 0 && x < N) ? g_s[y * N + x] : make_float2(0.f, 0.f);
    };
    for (int i = tid; i < N1 * PR; i += T) {
      const int y = i / PR, k = i % PR;
      const size_t row = (size_t)(ty + y) * a.W + tx;
      if (k < N / 2) {
        const int x = 2 * k + odd;   // pixels x, x + 1 of the tile row
        const float2 gA = gat(y, x - 1), gB = gat(y, x), gC = gat(y, x + 1);
        const float2 hA = gat(y - 1, x - 1), hB = gat(y - 1, x), hC = gat(y - 1, x + 1);
        const float2 s0 = make_float2(c00 * gB.x + c01 * gA.x + c10 * hB.x + c11 * hA.x,
                                      c00 * gB.y + c01 * gA.y + c10 * hB.y + c11 * hA.y);
        const float2 s1 = make_float2(c00 * gC.x + c01 * gB.x + c10 * hC.x + c11 * hB.x,
                                      c00 * gC.y + c01 * gB.y + c10 * hC.y + c11 * hB.y);
        const float i0 = 1.f / (__ldg(&a.acc[row + x].z) + damp);
        const float i1 = 1.f / (__ldg(&a.acc[row + x + 1].z) + damp);
        atomicAdd((float4*)(a.obj + row + x), make_float4(s0.x * i0, s0.y * i0, s1.x * i1, s1.y * i1));
      } else {
        const int x = odd ? 0 : N;
        const float2 gA = gat(y, x - 1), gB = gat(y, x), hA = gat(y - 1, x - 1), hB = gat(y - 1, x);
        const float2 s0 = make_float2(c00 * gB.x + c01 * gA.x + c10 * hB.x + c11 * hA.x,
                                      c00 * gB.y + c01 * gA.y + c10 * hB.y + c11 * hA.y);
        const float i0 = 1.f / (__ldg(&a.acc[row + x].z) + damp);
        atomicAdd(a.obj + row + x, make_float2(s0.x * i0, s0.y * i0));
      }
    }
    return;
  }
  // each object pixel of the (N+1)^2 tile gathers its four patch neighbours
  // (independent outputs keep many global loads in flight)
  for (int q = tid; q < N1 * N1; q += T) {
    const int y = q / N1, x = q % N1;
    float2 sacc = make_float2(0.f, 0.f);
    if (y < N && x < N) { const float2 g = g_s[y * N + x]; sacc.x += c00 * g.x; sacc.y += c00 * g.y; }
    if (y < N && x > 0) { const float2 g = g_s[y * N + x - 1]; sacc.x += c01 * g.x; sacc.y += c01 * g.y; }
    if (y > 0 && x < N) { const float2 g = g_s[(y - 1) * N + x]; sacc.x += c10 * g.x; sacc.y += c10 * g.y; }
    if (y > 0 && x > 0) { const float2 g = g_s[(y - 1) * N + x - 1]; sacc.x += c11 * g.x; sacc.y += c11 * g.y; }
    const size_t oi = (size_t)(ty + y) * a.W + (tx + x);
    const float inv = 1.f / (__ldg(&a.acc[oi].z) + damp);
    atomicAdd(a.obj + oi, make_float2(sacc.x * inv, sacc.y * inv));
  }
}

// Cluster form of the step-size pass (N <= 128): the PASS2C_C CTAs of a
// cluster share one position. CTA q reduces rows [q N/C, (q+1) N/C) of the
// patch and chunk q of the h planes and keeps its rows of g in shared memory;
// the C partial sums meet over distributed shared memory and are added in
// rank order, so every CTA holds the same FP64 totals and solves the 2x2
// system itself; then CTA q scatters the object update of its band of the
// (N+1)^2 tile (rows q N/C .. (q+1) N/C - 1, the last band also row N) from
// its own rows of g and, for its first row, the row above from L2. Against
// one CTA per position: four times the CTAs (the minibatch no longer leaves
// some SMs with one position and others with two), the serial solve of one
// cluster overlaps the streams of the others, and g is read once.
constexpr int PASS2C_T = 256, PASS2C_C = 4;

template <int N, int MINB>
__global__ void __cluster_dims__(PASS2C_C, 1, 1) __launch_bounds__(PASS2C_T, MINB) k_pass2_cluster(Pass2Args a) {
  constexpr int NN = N * N, T = PASS2C_T, C = PASS2C_C, RB = N / C, N1 = N + 1;
  static_assert(N % C == 0 && N <= 128, "bands of whole rows, g band in static shared memory");
  wait_prior_grid();
  cg::cluster_group cluster = cg::this_cluster();
  __shared__ double red[32 * 5];
  __shared__ double part[5];
  __shared__ double alpha_sh;
  __shared__ __align__(16) float2 gsh[RB * N];
  const int q = (int)cluster.block_rank();
  const int slot = blockIdx.x / C, tid = threadIdx.x;
  if (!a.valid[slot]) return;   // the same decision in every CTA of the cluster
  const int e = a.b0 + slot;
  const int j = a.order ? a.order[e] : e;
  int ty, tx;
  float fy, fx;
  tile_of(a.pos[2 * j], a.pos[2 * j + 1], N, a.H, a.W, ty, tx, fy, fx);
  const float w00 = (1.f - fy) * (1.f - fx), w01 = (1.f - fy) * fx, w10 = fy * (1.f - fx), w11 = fy * fx;
  const float damp = a.delta_o * __uint_as_float(a.sc->max_illum);
  const size_t slotNN = (size_t)slot * NN;
  const int M = a.M;
  const float2* g_s = a.g_s + slotNN;
  const float2* o_s = a.o_s + slotNN;
  const float2* h_s = a.h_s + slotNN * M;

  const int p_lo = q * RB * N;
  float A11 = 0.f, A12 = 0.f, A22 = 0.f, b1 = 0.f, b2 = 0.f;
#pragma unroll 1
  for (int i = tid; i < RB * N; i += T) {
    const int p = p_lo + i, r = p / N, c = p % N;
    const float2 g = __ldcs(g_s + p);
    const float2 o = __ldcs(o_s + p);
    gsh[i] = g;
    float2 d = make_float2(0.f, 0.f);
    if (a.update_object) d = dohat(a.acc + (size_t)(ty + r) * a.W + (tx + c), a.W, w00, w01, w10, w11, damp);
    const float sp = __ldg(a.Sp + p), sdp = __ldg(a.Sdp + p);
    const float2 cp = __ldg(a.Cp + p);
    A11 += cabs2(d) * sp;
    const float2 od = cmulc(d, o);           // conj(d) o
    A12 += od.x * cp.x - od.y * cp.y;        // Re(conj(d) o Cp)
    A22 += cabs2(o) * sdp;
    b1 += d.x * g.x + d.y * g.y;             // Re(conj(d) g)
  }
  if (a.update_probe) {
    // b2 over chunk q of the h planes (contiguous pixel pairs)
    const float4* h4 = (const float4*)h_s;
    const float4* d4 = (const float4*)a.dP;
    const int Q = M * NN / 2;
    const int q_lo = (int)((long long)Q * q / C), q_hi = (int)((long long)Q * (q + 1) / C);
    int k = q_lo + tid;
    for (; k + 3 * T < q_hi; k += 4 * T) {   // four independent 16-byte streams per thread
      float4 dp[4], h[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        dp[u] = __ldg(d4 + k + u * T);
        h[u] = __ldcs(h4 + k + u * T);
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) b2 += dp[u].x * h[u].x + dp[u].y * h[u].y + dp[u].z * h[u].z + dp[u].w * h[u].w;
    }
    for (; k < q_hi; k += T) {
      const float4 dp = __ldg(d4 + k);
      const float4 h = __ldcs(h4 + k);
      b2 += dp.x * h.x + dp.y * h.y + dp.z * h.z + dp.w * h.w;   // Re(conj(dP_k) h_k)
    }
  }
  double v[5] = {A11, A12, A22, b1, b2};
  block_sum<5>(v, red);
  if (tid == 0)
#pragma unroll
    for (int i = 0; i < 5; ++i) part[i] = v[i];
  cluster.sync();   // every CTA's partials (and its g band) are written
  if (tid == 0) {
    double t[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
#pragma unroll
    for (int r = 0; r < C; ++r) {
      const double* pr = cluster.map_shared_rank(part, r);
#pragma unroll
      for (int i = 0; i < 5; ++i) t[i] += pr[i];
    }
    double aO, aP;
    solve_step(t[0], t[1], t[2], t[3], t[4], a.lam, aO, aP);
    alpha_sh = aO;
    if (q == 0) {
      if (a.alpha_out) {
        a.alpha_out[2 * j] = aO;
        a.alpha_out[2 * j + 1] = aP;
      }
      atomicAdd(&a.sc->sum_alpha_p, aP);
      atomicAdd(&a.sc->count, 1);
    }
  }
  cluster.sync();   // no CTA leaves while another reads its partials; alpha_sh is visible
  if (!a.update_object) return;
  const float aO = (float)alpha_sh;
  const float c00 = aO * w00, c01 = aO * w01, c10 = aO * w10, c11 = aO * w11;
  const int y0 = q * RB, y1 = y0 + RB + (q == C - 1 ? 1 : 0);
  // g at patch row yy (y0 - 1 <= yy < y0 + RB): the band from shared memory, the row above from L2
  auto gat = [&](int yy, int xx) { return yy >= y0 ? gsh[(yy - y0) * N + xx] : __ldg(g_s + yy * N + xx); };
  for (int i = tid; i < (y1 - y0) * N1; i += T) {
    const int y = y0 + i / N1, x = i % N1;
    float2 sacc = make_float2(0.f, 0.f);
    if (y < N && x < N) { const float2 g = gat(y, x); sacc.x += c00 * g.x; sacc.y += c00 * g.y; }
    if (y < N && x > 0) { const float2 g = gat(y, x - 1); sacc.x += c01 * g.x; sacc.y += c01 * g.y; }
    if (y > 0 && x < N) { const float2 g = gat(y - 1, x); sacc.x += c10 * g.x; sacc.y += c10 * g.y; }
    if (y > 0 && x > 0) { const float2 g = gat(y - 1, x - 1); sacc.x += c11 * g.x; sacc.y += c11 * g.y; }
    const size_t oi = (size_t)(ty + y) * a.W + (tx + x);
    const float inv = 1.f / (__ldg(&a.acc[oi].z) + damp);
    atomicAdd(a.obj + oi, make_float2(sacc.x * inv, sacc.y * inv));
  }
}

constexpr int STEP_T = 256, STEP_U = 4, STEP_GROUP = 96;   // threads, positions per tree, most positions per CTA

template <int N>
struct StepSums {
  static constexpr int T = N * N / 2 < STEP_T ? N * N / 2 : STEP_T;
  static constexpr int CHUNKS = N * N / 2 / T;
  static_assert(T * CHUNKS * 2 == N * N && T % 32 == 0, "a pixel pair per thread");
};

// Sums of `per` positions over one chunk's pixel pairs per CTA, added to
// a.part[slot][5] (zero on entry) by FP64 atomics: the last bits of a position's
// sums, and so of its alpha, depend on the order in which the chunks finish (one
// CTA per position adds in a fixed order). Dynamic shared memory: (M + K) T
// float4, the direction of each mode (OPR: of each eigenmode, then of the shared
// modes) at the thread's pair.
template <int N, bool OPR>
__global__ void __launch_bounds__(StepSums<N>::T, 3) k_step_sums(Pass2Args a, int per) {
  constexpr int NN = N * N, T = StepSums<N>::T, U = STEP_U, W = T / 32;
  extern __shared__ __align__(16) float4 dsm[];
  __shared__ float part[2][W][U * 5];
  __shared__ float4 where[STEP_GROUP];   // tile corner (int bits) and fractions
  __shared__ int live[STEP_GROUP];       // 0: a skipped position
  __shared__ float wsh[OPR ? STEP_GROUP * OPR_KMAX : 1];
  wait_prior_grid();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int chunk = blockIdx.x % StepSums<N>::CHUNKS, group = blockIdx.x / StepSums<N>::CHUNKS;
  const int p = (chunk * T + tid) * 2, r = p / N, c = p % N;   // this thread's pixels p, p + 1
  const int i0 = group * per, n = min(per, a.nb - i0);
  const int M = a.M, K = OPR ? a.K : 0, Ms = OPR ? M - 1 : M;       // shared modes
  const float damp = a.delta_o * __uint_as_float(a.sc->max_illum);
  for (int i = tid; i < n; i += T) {
    int ty = 0, tx = 0;   // (a skipped position's loads go to the object's first tile)
    float fy = 0.f, fx = 0.f;
    const bool ok = a.valid[i0 + i] != 0;
    live[i] = ok;
    if (ok) {
      const int e = a.b0 + i0 + i, j = a.order ? a.order[e] : e;
      tile_of(a.pos[2 * j], a.pos[2 * j + 1], N, a.H, a.W, ty, tx, fy, fx);
      if (OPR)
        for (int m = 0; m < K; ++m) wsh[i * OPR_KMAX + m] = a.opr_w[(size_t)j * K + m];
    }
    where[i] = make_float4(__int_as_float(ty), __int_as_float(tx), fy, fx);
  }
  if (a.update_probe) {
    for (int m = 0; m < K; ++m) dsm[m * T + tid] = __ldg((const float4*)(a.opr_dU + (size_t)m * NN + p));
    for (int k = 0; k < Ms; ++k) dsm[(K + k) * T + tid] = __ldg((const float4*)(a.dP + (size_t)k * NN + p));
  }
  const float2 Sp = __ldg((const float2*)(a.Sp + p)), Sd = __ldg((const float2*)(a.Sdp + p));
  const float4 Cp = __ldg((const float4*)(a.Cp + p));
  __syncthreads();

  // the five partial sums of position i at this thread's pair (no branch on the
  // position: the loads of several positions are in flight together)
  auto sums = [&](int i, float (&v)[5]) {
    const float4 w = where[i];
    const int ty = __float_as_int(w.x), tx = __float_as_int(w.y);
    const size_t base = (size_t)(i0 + i) * NN + p;
    const float4 g2 = __ldg((const float4*)(a.g_s + base));   // (read again by the update)
    const float4 o2 = __ldcs((const float4*)(a.o_s + base));
    const float2* h = a.h_s + (size_t)(i0 + i) * M * NN + p;
    float2 sp = Sp, sd = Sd;
    float4 cp = Cp;
    float b2 = 0.f;
    if (OPR) {
      const float4 P2 = __ldg((const float4*)(a.p0_s + base));
      const float2 Pa = make_float2(P2.x, P2.y), Pb = make_float2(P2.z, P2.w);
      sp.x += cabs2(Pa);
      sp.y += cabs2(Pb);
      if (a.update_probe) {   // the primary mode's direction sum_m w_jm dU_m
        const float4 h2 = __ldcs((const float4*)h);
        float4 D = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int m = 0; m < K; ++m) {
          const float4 u = dsm[m * T + tid];
          const float wm = wsh[i * OPR_KMAX + m];
          D.x = fmaf(wm, u.x, D.x); D.y = fmaf(wm, u.y, D.y); D.z = fmaf(wm, u.z, D.z); D.w = fmaf(wm, u.w, D.w);
        }
        const float2 ea = make_float2(D.x, D.y), eb = make_float2(D.z, D.w);
        const float2 ca = cmulc(Pa, ea), cb = cmulc(Pb, eb);
        cp = make_float4(cp.x + ca.x, cp.y + ca.y, cp.z + cb.x, cp.w + cb.y);
        sd.x += cabs2(ea);
        sd.y += cabs2(eb);
        b2 += D.x * h2.x + D.y * h2.y + D.z * h2.z + D.w * h2.w;   // Re(conj(dP_j0) h_j0)
      }
      h += NN;
    }
    if (a.update_probe)   // Re sum_k <dP_k, h_k> over the shared modes
#pragma unroll 4
      for (int k = 0; k < Ms; ++k) {
        const float4 x = __ldcs((const float4*)(h + (size_t)k * NN)), d = dsm[(K + k) * T + tid];
        b2 += d.x * x.x + d.y * x.y + d.z * x.z + d.w * x.w;
      }
    float2 d0 = make_float2(0.f, 0.f), d1 = d0;
    if (a.update_object) {
      const float fy = w.z, fx = w.w;
      const float w00 = (1.f - fy) * (1.f - fx), w01 = (1.f - fy) * fx, w10 = fy * (1.f - fx), w11 = fy * fx;
      const float4* q = a.acc + (size_t)(ty + r) * a.W + (tx + c);
      const float4 qa = __ldg(q), qb = __ldg(q + 1), qc = __ldg(q + 2);
      const float4 qd = __ldg(q + a.W), qe = __ldg(q + a.W + 1), qf = __ldg(q + a.W + 2);
      const float ia = 1.f / (qa.z + damp), ib = 1.f / (qb.z + damp), ic = 1.f / (qc.z + damp);
      const float id = 1.f / (qd.z + damp), ie = 1.f / (qe.z + damp), iF = 1.f / (qf.z + damp);
      // dO_hat at the pixel: each corner's quotient, then the bilinear weights
      d0 = make_float2(w00 * ia * qa.x + w01 * ib * qb.x + w10 * id * qd.x + w11 * ie * qe.x,
                       w00 * ia * qa.y + w01 * ib * qb.y + w10 * id * qd.y + w11 * ie * qe.y);
      d1 = make_float2(w00 * ib * qb.x + w01 * ic * qc.x + w10 * ie * qe.x + w11 * iF * qf.x,
                       w00 * ib * qb.y + w01 * ic * qc.y + w10 * ie * qe.y + w11 * iF * qf.y);
    }
    const float2 g0 = make_float2(g2.x, g2.y), g1 = make_float2(g2.z, g2.w);
    const float2 o0 = make_float2(o2.x, o2.y), o1 = make_float2(o2.z, o2.w);
    const float2 od0 = cmulc(d0, o0), od1 = cmulc(d1, o1);   // conj(d) o
    v[0] = cabs2(d0) * sp.x + cabs2(d1) * sp.y;
    v[1] = od0.x * cp.x - od0.y * cp.y + od1.x * cp.z - od1.y * cp.w;   // Re(conj(d) o Cp)
    v[2] = cabs2(o0) * sd.x + cabs2(o1) * sd.y;
    v[3] = d0.x * g0.x + d0.y * g0.y + d1.x * g1.x + d1.y * g1.y;       // Re(conj(d) g)
    v[4] = b2;
  };
  static_assert(U == 4, "the tree below splits four positions over the lanes");
#pragma unroll 1
  for (int t = 0, buf = 0; t < n; t += U, buf ^= 1) {
    float v[U][5];
#pragma unroll
    for (int u = 0; u < U; ++u) sums(min(t + u, n - 1), v[u]);
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (t + u >= n || !live[t + u])
#pragma unroll
        for (int q = 0; q < 5; ++q) v[u][q] = 0.f;
    // lanes 8u .. 8u + 7 end with position u: halves of the positions change
    // hands over lane bits 4 and 3, then eight lanes add up
    float x[5];
#pragma unroll
    for (int q = 0; q < 5; ++q) {
      const bool hi = lane & 16, hj = lane & 8;
      const float s0 = hi ? v[0][q] : v[2][q], s1 = hi ? v[1][q] : v[3][q];
      const float k0 = (hi ? v[2][q] : v[0][q]) + __shfl_xor_sync(0xffffffffu, s0, 16);
      const float k1 = (hi ? v[3][q] : v[1][q]) + __shfl_xor_sync(0xffffffffu, s1, 16);
      x[q] = (hj ? k1 : k0) + __shfl_xor_sync(0xffffffffu, hj ? k0 : k1, 8);
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) x[q] += __shfl_xor_sync(0xffffffffu, x[q], o);
    }
#pragma unroll
    for (int q = 0; q < 5; ++q)
      if ((lane & 7) == q) part[buf][warp][(lane >> 3) * 5 + q] = x[q];
    __syncthreads();   // (the other buffer is free: its readers joined here)
    if (tid < U * 5 && t + tid / 5 < n) {
      double s = 0.0;
      for (int k = 0; k < W; ++k) s += (double)part[buf][k][tid];
      atomicAdd(a.part + (size_t)(i0 + t + tid / 5) * 5 + tid % 5, s);
    }
  }
}

// Object update of rows band * 32 .. of one position's tile (the last band also
// row N): O += alpha_O S_j^T g / (illum + delta_O), each object pixel gathering
// its four patch neighbours and divided by its own preconditioner.
constexpr int UPD_T = 256;
template <int N>
struct Bands {
  static constexpr int ROWS = N < 32 ? N : 32, NUM = N / ROWS;
};
template <int N>
__device__ __forceinline__ void update_band(int band, const float2* __restrict__ g_s, const float4* __restrict__ acc,
                                            float2* obj, int W, int ty, int tx, float fy, float fx, float damp,
                                            float aO) {
  constexpr int T = UPD_T, RB = Bands<N>::ROWS, N1 = N + 1;
  const int tid = threadIdx.x;
  const float c00 = aO * ((1.f - fy) * (1.f - fx)), c01 = aO * ((1.f - fy) * fx);
  const float c10 = aO * (fy * (1.f - fx)), c11 = aO * (fy * fx);
  const int y0 = band * RB, y1 = y0 + RB + (band == Bands<N>::NUM - 1 ? 1 : 0);
  auto gat = [&](int y, int x) {
    return (y >= 0 && y < N && x >= 0 && x < N) ? __ldg(g_s + y * N + x) : make_float2(0.f, 0.f);
  };
  auto mix = [&](float2 gB, float2 gA, float2 hB, float2 hA, float inv) {
    return make_float2((c00 * gB.x + c01 * gA.x + c10 * hB.x + c11 * hA.x) * inv,
                       (c00 * gB.y + c01 * gA.y + c10 * hB.y + c11 * hA.y) * inv);
  };
  auto out = [&](int y, int x) { return (size_t)(ty + y) * W + tx + x; };
  auto pre = [&](size_t o) { return 1.f / (__ldg(&acc[o].z) + damp); };
  if (((uintptr_t)obj & 15) == 0 && (W & 1) == 0) {
    // pairs of object pixels at even object columns, one 16-byte vector atomic
    // each (half the atomic operations); per tile row N/2 pairs and one single
    // pixel (the first when tx is odd, else the last). A thread keeps one
    // column pair and walks down its rows: the row of g above stays in registers.
    const int odd = tx & 1;
    constexpr int RUNS = T / (N / 2) > 0 ? T / (N / 2) : 1;
    for (int item = tid; item < RUNS * (N / 2); item += T) {
      const int x = 2 * (item % (N / 2)) + odd, run = item / (N / 2);
      const int ya = y0 + (y1 - y0) * run / RUNS, yb = y0 + (y1 - y0) * (run + 1) / RUNS;
      float2 hA = gat(ya - 1, x - 1), hB = gat(ya - 1, x), hC = gat(ya - 1, x + 1);
#pragma unroll 4
      for (int y = ya; y < yb; ++y) {
        const float2 gA = gat(y, x - 1), gB = gat(y, x), gC = gat(y, x + 1);
        const size_t o = out(y, x);
        const float2 s0 = mix(gB, gA, hB, hA, pre(o)), s1 = mix(gC, gB, hC, hB, pre(o + 1));
        atomicAdd((float4*)(obj + o), make_float4(s0.x, s0.y, s1.x, s1.y));
        hA = gA; hB = gB; hC = gC;
      }
    }
    for (int y = y0 + tid; y < y1; y += T) {
      const int x = odd ? 0 : N;
      const size_t o = out(y, x);
      atomicAdd(obj + o, mix(gat(y, x), gat(y, x - 1), gat(y - 1, x), gat(y - 1, x - 1), pre(o)));
    }
    return;
  }
  for (int q = tid; q < (y1 - y0) * N1; q += T) {
    const int y = y0 + q / N1, x = q % N1;
    const size_t o = out(y, x);
    atomicAdd(obj + o, mix(gat(y, x), gat(y, x - 1), gat(y - 1, x), gat(y - 1, x - 1), pre(o)));
  }
}

// One CTA per band of a position: the solve and the band's update. Every
// band solves the position's system (the same values); band 0 records the steps.
template <int N>
__global__ void __launch_bounds__(UPD_T, 4) k_step_update(Pass2Args a) {
  wait_prior_grid();
  __shared__ double alpha_sh;
  const int slot = blockIdx.x / Bands<N>::NUM, band = blockIdx.x % Bands<N>::NUM;
  if (!a.valid[slot]) return;
  const int e = a.b0 + slot;
  const int j = a.order ? a.order[e] : e;
  if (threadIdx.x == 0) {
    const double* v = a.part + (size_t)slot * 5;
    double aO, aP;
    solve_step(v[0], v[1], v[2], v[3], v[4], a.lam, aO, aP);
    alpha_sh = aO;
    if (band == 0) {
      if (a.alpha_out) {
        a.alpha_out[2 * j] = aO;
        a.alpha_out[2 * j + 1] = aP;
      }
      atomicAdd(&a.sc->sum_alpha_p, aP);
      atomicAdd(&a.sc->count, 1);
    }
  }
  if (!a.update_object) return;
  int ty, tx;
  float fy, fx;
  tile_of(a.pos[2 * j], a.pos[2 * j + 1], N, a.H, a.W, ty, tx, fy, fx);
  const float damp = a.delta_o * __uint_as_float(a.sc->max_illum);
  __syncthreads();
  update_band<N>(band, a.g_s + (size_t)slot * N * N, a.acc, a.obj, a.W, ty, tx, fy, fx, damp, (float)alpha_sh);
}

template <int N, bool OPR>
cudaError_t launch_step(const Pass2Args& a, cudaStream_t s) {
  using S = StepSums<N>;
  const size_t sm = a.update_probe ? (size_t)((OPR ? a.M - 1 + a.K : a.M) * S::T) * sizeof(float4) : 0;
  static unsigned long long done = 0;
  cudaError_t e = smem_optin(k_step_sums<N, OPR>, (size_t)(16 + OPR_KMAX) * S::T * sizeof(float4), &done);
  if (e != cudaSuccess) return e;
  // Positions per CTA: the fewest rounds of positions with 3 CTAs per SM at
  // work (4 more stand for a CTA's start), not a last wave that is nearly empty.
  const long long places = 3 * sm_count();
  int per = STEP_U;
  long long best = -1;
  for (int q = STEP_U; q <= STEP_GROUP; q += STEP_U) {
    const long long ctas = (long long)S::CHUNKS * ((a.nb + q - 1) / q);
    const long long cost = (ctas + places - 1) / places * (q + 4);
    if (best < 0 || cost < best) best = cost, per = q;
  }
  e = launch_pdl(k_step_sums<N, OPR>, dim3(S::CHUNKS * ((a.nb + per - 1) / per)), dim3(S::T), sm, s, a, per);
  if (e != cudaSuccess) return e;
  return launch_pdl(k_step_update<N>, dim3(a.nb * Bands<N>::NUM), dim3(UPD_T), 0, s, a);
}

// The two launches, or one CTA per position at two CTAs per SM? The latter
// costs the time of one position per started wave, the former grow with the
// minibatch. Measured on GB300, one mode, positions: us per CTA each -> two launches
//   window 256: 8: 118 -> 25, 38: 121 -> 44, 64: 131 -> 68, 128: 156 -> 119,
//               192: 193 -> 166, 256: 199 <- 228, 384: 334 -> 312
//   window 192: 8: 74 -> 25, 64: 76 -> 42, 128: 83 -> 77, 192: 121 -> 97, 256: 126 <- 133
//   window 128: 8: 37 -> 21, 64: 39 -> 29, 128: 39 -> 38, 192: 53 -> 52, 256: 55 <- 62, 384: 100 -> 86
//   window  64: 96: 18.5 <- 19, 192: 23.6 -> 20.9, 256: 24.4 <- 26.9, 384: 40 -> 32
//   windows 16 and 32: 10.5 <- 14.6, 12.3 <- 16.5 (the second launch)
// so the line lies where the last wave of CTAs is 0.7 full. A relaxed probe's
// position re-reads K eigenmode directions: from window 128 on the two launches
// always gain (8 eigenmodes, 8 and 256 positions, window 256: 189 -> 26 and
// 289 -> 240, window 192: 94 -> 25 and 146 -> 140, window 128: 55 -> 22 and
// 74 -> 69), at 64 also for the small minibatches (20 -> 17.4).
inline bool use_step(int N, int nb, bool opr) {
  if (N < 64) return false;
  if (opr && N >= 128) return true;
  const int slots = 2 * sm_count(), waves = (nb + slots - 1) / slots;
  if (N == 64 && nb <= sm_count()) return opr;
  return 10LL * nb < 7LL * slots * waves;
}

// variant 0: by the rule above, 1: the two launches, 2 and 3: the cluster form
// at four and three CTAs per SM (64 and 80 registers; windows <= 128, not with
// a relaxed probe)
template <int N>
cudaError_t launch_pass2(const Pass2Args& a, cudaStream_t s, int variant) {
  if (a.nb <= 0) return cudaSuccess;
  const bool opr = a.opr_dU != nullptr;
  if constexpr (N <= 128) {
    if (variant == 2 && !opr) return launch_pdl(k_pass2_cluster<N, 4>, dim3(PASS2C_C * a.nb), dim3(PASS2C_T), 0, s, a);
    if (variant == 3 && !opr) return launch_pdl(k_pass2_cluster<N, 3>, dim3(PASS2C_C * a.nb), dim3(PASS2C_T), 0, s, a);
  }
  if (variant == 1 || use_step(N, a.nb, opr)) return opr ? launch_step<N, true>(a, s) : launch_step<N, false>(a, s);
  if constexpr (N < 128)
    if (opr) return launch_pdl(k_pass2<N, PASS2_T, true>, dim3(a.nb), dim3(PASS2_T), 0, s, a);
  return launch_pdl(k_pass2<N, PASS2_T, false>, dim3(a.nb), dim3(PASS2_T), 0, s, a);
}

}  // namespace ptycho
