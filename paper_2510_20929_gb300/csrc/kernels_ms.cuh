// Multislice forward model, its adjoint and the LSQML tangents (Pty-Chi Sec. 1
// and Sec. 2.1: multislice modelling) on the packed line-pair transforms
// (kernels_pair.cuh's geometries: one CTA per position, or a cluster of CTAs
// with 32 rows each at the windows 192 and 256).
//
// The object has S slices [S, H, W]. For position j and probe mode k the wave
// entering slice 0 is P_k; the wave leaving slice s is (incident_s) o_j^(s)
// with o_j^(s) = S_j(O^(s)); between slices it is carried by the
// angular-spectrum propagator, incident_s = F^-1[H F (leaving_{s-1})]. The
// far field of the last slice's exit wave gives I_j = sum_k |F psi|^2. The
// backward pass carries each mode from the far field back through the slices
// (conj(H)), summing conj(incident_s) g per slice and conj(o^(0)) g per mode.
//
// A wave lives in its threads' registers from the probe to the far field and
// back: a propagation is a forward transform, the product with H and an
// inverse transform with no pass over the tile around them, and the slice
// products take the thread's own pixels. The transforms are the bulk of the
// code, so the modes, slices and directions run through one loop that holds
// one copy of each (a copy per use would run at the speed of instruction
// fetches). Incident waves and far fields are kept in per-thread order (16
// coalesced bytes per access); what other kernels read is in pixel order.
// What bounds it: the transforms, as in kernels_pair.cuh; the incident waves,
// patches and slice gradients stream through L2 between them.
// Measured on GB300 against one line per lane group and passes over the tile
// between the transforms: window 256, 4 slices, 4 modes, 256 positions 7.92 ->
// 6.26 ms; the LSQML pass at window 128 with 3 slices, 2 modes, 128 positions
// 373 -> 289 us.
#pragma once
#include "kernels_ms_line.cuh"
#include "kernels_pair.cuh"
#include "launch.h"

namespace ptycho {

// v *= H / N^2, or conj(H) / N^2, at the thread's far-field pixels. Hf is in
// [ky][kx] order, transposed for a cluster (whose lanes run along ky).
template <class G>
__device__ __forceinline__ void mul_propagator(const G& geo, fp::C2 (&v)[G::NP], const float2* __restrict__ Hf,
                                               bool conj) {
  constexpr int N = G::N, NP = G::NP;
  const float2 sc = fp::splat(1.0f / (float)(N * N));
  const float sg = conj ? -1.f : 1.f;
  ahead<NP, 4>(
      [&](int i) -> float4 {
        const float2* h;
        if constexpr (G::VERT) h = Hf + (G::LR * geo.q + geo.far_x()) * N + geo.far_y(i);
        else h = Hf + geo.far_y(i) * N + geo.far_x(i);
        const float2 a = __ldg(h), b = __ldg(h + N);
        return make_float4(a.x, a.y, b.x, b.y);
      },
      [&](int i, float4 h) {
        v[i] = fp::pscale(fp::pmul(v[i], {make_float2(h.x, h.z), make_float2(sg * h.y, sg * h.w)}), sc);
      });
}

struct Two { float4 a, b; };
struct Three { float4 a, b, c; };

// Start of a multislice kernel's CTA: twiddles and the copy barriers. Joins the block.
template <class G>
__device__ __forceinline__ void ms_begin(float2* tw, uint64_t* bar) {
  if (threadIdx.x == 0) {
    tc::mbar_init(bar, 1);
    tc::mbar_init(bar + 1, 1);
    tc::fence_mbar_init();
  }
  G::fill_twiddles(tw);
  __syncthreads();
}

// One position per CTA (or cluster). LS: the LSQML instantiation (exit-plane
// changes instead of gradients, the slices' illumination, the per-slice
// accumulators). With a.recompute the forward pass keeps no incident waves:
// the backward pass runs each mode through the slices again first and parks
// its waves in the slot's scratch (the same arithmetic, so the same waves).
template <class G, bool LS>
__global__ void __launch_bounds__(G::T, PairCtas<G>::n) k_pass1_ms(MsArgs a) {
  using SM = PairSmem<G>;
  using fp::C2;
  constexpr int N = G::N, T = G::T, NP = G::NP, NN = N * N, LR = G::LR, Q = G::Q, LNN = LR * N, PL = NN / 2;
  extern __shared__ __align__(16) unsigned char smem[];
  double* red = (double*)(smem + SM::red);
  float4* tile = (float4*)(smem + SM::tile);
  float4* rI = (float4*)(smem + SM::rI);
  float2* tw = (float2*)(smem + SM::tw);
  uint64_t* bar = (uint64_t*)(red + 252);

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
  ms_begin<G>(tw, bar);
  // joins the block after a wait for copies; false when a thread's wait gave up (see copy_arrived)
  auto arrived = [&](bool got, uint64_t* b, uint32_t parity) -> bool {
    return copy_arrived(geo, got, b, parity, a.status, a.valid + slot, (a.give_up >> (int)(b - bar)) & 1);
  };

  const int M = a.M, S = a.S, mode = a.mode;
  const bool grad = mode != MODE_FWD;
  const bool rec = grad && a.recompute != 0 && S > 1, keep = grad && !a.recompute;
  const size_t HW = (size_t)a.H * a.W;
  const float invN = 1.0f / (float)N;
  const size_t slotNN = (size_t)slot * NN;
  auto pix = [&](int i) { return (y0 + geo.row(i)) * N + geo.col(i); };   // pixel pair i in a plane
  float2* o_s = a.o_s + slotNN * S;
  // per-thread planes: the far field of mode k, the incident wave of mode k at
  // slice s (the CTA's share of a plane is the memory of its own pixel rows)
  auto psi = [&](int k) { return (float4*)(a.psi_s + slotNN * M + (size_t)k * NN + (size_t)y0 * N) + tid; };
  auto inc = [&](int k, int s) {
    return (float4*)(a.in_s + ms_inc_offset(a.recompute != 0, slotNN, M, S, k, s, NN) + (size_t)y0 * N) + tid;
  };

  bool lost = false;   // a copy of this CTA's never arrived
  // ---- slice patches o^(s) = S_j(O^(s)) -------------------------------------------
#pragma unroll 1
  for (int s = 0; s < S; ++s) {
    const ObjStage<G> stage(tile, bar, a.obj, a.obj + s * HW, a.H, a.W, ty + y0, tx);
    if (tid == 0) stage.expect();
    stage.copy();
    if (!arrived(stage.wait(s & 1), bar, s & 1)) {
      if (Q == 1) return;
      lost = true;
      break;
    }
#pragma unroll 4
    for (int i = 0; i < NP; ++i)
      st_pair<G>(o_s + (size_t)s * NN + pix(i), stage.patch(geo.row(i), geo.col(i), fy, fx));
    tc::fence_async_smem();
    __syncthreads();   // the stage is free
  }

  float2* go_s = a.go_s + slotNN * S;
  float2* h_s = a.h_s + slotNN * M;
  C2 v[NP];
  auto enter = [&](int k) {   // the wave leaving slice 0
    const float2* Pk = a.probe + (size_t)k * NN;
    ahead<NP, NP / 2>([&](int i) { return Two{ldg_pair<G>(Pk + pix(i)), ld_pair<G>(o_s + pix(i))}; },
                      [&](int i, const Two& x) { v[i] = exit_wave(x.a, x.b); });
  };
  auto load_far = [&](int k) {   // the corrected far field of mode k
    get_far<G>(v, psi(k));
    mul_factor<G>(v, rI);
  };
  auto half = [](const C2& c, int h) { return h ? make_float2(c.re.y, c.im.y) : make_float2(c.re.x, c.im.x); };
  // adds conj(w) v to the gradient of a slice at pixel pair i, `p` the sum over
  // the modes so far (they run last to first)
  auto ld_go = [&](int s, int i, int k) {
    return k < M - 1 ? ld_pair<G>(go_s + (size_t)s * NN + pix(i)) : make_float4(0.f, 0.f, 0.f, 0.f);
  };
  auto add_go = [&](int s, int i, float4 w, float4 p) {
    const float2 g0 = cmulc(make_float2(w.x, w.y), half(v[i], 0)), g1 = cmulc(make_float2(w.z, w.w), half(v[i], 1));
    st_pair<G>(go_s + (size_t)s * NN + pix(i), make_float4(g0.x + p.x, g0.y + p.y, g1.x + p.z, g1.y + p.w));
  };

  enum { FWD, REC, BWD };
  int ph = FWD, k = 0, s = 0;
  bool far = false;   // v is a far field already
  enter(0);
#pragma unroll 1
  for (;;) {
    if (!far) {   // v: the wave leaving slice s (backward: reaching its entrance)
      geo.forward(v);
      if (ph == FWD && s == S - 1) {
#pragma unroll
        for (int i = 0; i < NP; ++i) v[i] = fp::pscale(v[i], fp::splat(invN));
        add_intensity<G>(v, rI, k == 0);
        if (grad && (k < M - 1 || rec)) put_far<G>(v, psi(k));
        if (k < M - 1) {
          ++k;
          s = 0;
          enter(k);
          __syncthreads();   // the tile is free
          continue;
        }
        if (!data_term<G, N == 64 || N == 128>(geo, rI, red, bar + 1, a.meas, j, a.ipred, mode, a.eps, a.loss,
                                               a.status, [&](bool got, uint64_t* b) { return arrived(got, b, 0); })) {
          if (Q == 1) return;
          lost = true;
        }
        if (!grad) return;
        settle_lost<G>(a.valid + slot, lost);
        if (rec) {
          ph = REC;
          s = 0;
          enter(k);
          __syncthreads();
          continue;
        }
        ph = BWD;
        mul_factor<G>(v, rI);
      } else {
        mul_propagator(geo, v, a.Hf, ph == BWD);
        if (ph == BWD) --s;
      }
    }
    far = false;
    __syncthreads();   // the tile is free
    geo.inverse(v);
    if (ph != BWD) {   // v: the wave incident on slice s + 1
      ++s;
      if (ph == REC || keep) put_far<G>(v, inc(k, s));
      if (ph == REC && s == S - 1) {   // every incident wave is parked
        ph = BWD;
        load_far(k);
        far = true;
        continue;
      }
      if (LS && ph == FWD) {   // the slice's illumination sum_k |inc_k|^2
        float* w = a.w_s + slotNN * (S - 1) + (size_t)(s - 1) * NN;
        constexpr int DP = G::VERT ? N : 1;
#pragma unroll
        for (int i = 0; i < NP; ++i) {
          float2 w2 = make_float2(cabs2(half(v[i], 0)), cabs2(half(v[i], 1)));
          float* p = w + pix(i);
          if (k > 0) {
            w2.x += p[0];
            w2.y += p[DP];
          }
          p[0] = w2.x;
          p[DP] = w2.y;
        }
      }
      ahead<NP, 4>([&](int i) { return ld_pair<G>(o_s + (size_t)s * NN + pix(i)); },
                   [&](int i, float4 o) {
                     v[i] = pack_pair(cmul(half(v[i], 0), make_float2(o.x, o.y)),
                                      cmul(half(v[i], 1), make_float2(o.z, o.w)));
                   });
    } else if (s > 0) {   // v: the change leaving slice s
      const float4* in = inc(k, s);
      ahead<NP, 3>(
          [&](int i) { return Three{in[i * T], ld_pair<G>(o_s + (size_t)s * NN + pix(i)), ld_go(s, i, k)}; },
          [&](int i, const Three& x) {
            add_go(s, i, make_float4(x.a.x, x.a.z, x.a.y, x.a.w), x.c);   // (the wave's units: re, re, im, im)
            v[i] = pack_pair(cmulc(make_float2(x.b.x, x.b.y), half(v[i], 0)),
                             cmulc(make_float2(x.b.z, x.b.w), half(v[i], 1)));
          });
    } else {   // slice 0: object gradient conj(P_k) g, probe gradient conj(o^(0)) g
      const float2* Pk = a.probe + (size_t)k * NN;
      ahead<NP, 3>(
          [&](int i) { return Three{ldg_pair<G>(Pk + pix(i)), ld_pair<G>(o_s + pix(i)), ld_go(0, i, k)}; },
          [&](int i, const Three& x) {
            add_go(0, i, x.a, x.c);
            const float2 h0 = cmulc(make_float2(x.b.x, x.b.y), half(v[i], 0));
            const float2 h1 = cmulc(make_float2(x.b.z, x.b.w), half(v[i], 1));
            stcs_pair<G>(h_s + (size_t)k * NN + pix(i), make_float4(h0.x, h0.y, h1.x, h1.y));
          });
      if (k == 0) break;
      --k;
      if (rec) {
        ph = REC;
        s = 0;
        enter(k);
      } else {
        s = S - 1;
        load_far(k);
        far = true;
        continue;   // (joined before the inverse)
      }
    }
    __syncthreads();   // the tile is free
  }

  if constexpr (Q > 1)
    if (!__syncthreads_and(*(const volatile int*)(a.valid + slot))) return;   // given up by a CTA of the cluster

  // ---- per slice: scatter S_j^T of its gradient; position gradient over the slices ----
  const float2* gt = (const float2*)tile;
  float* spS = (float*)rI;
  float gyv = 0.f, gxv = 0.f;
#pragma unroll 1
  for (s = 0; s < S; ++s) {
    __syncthreads();   // the tile and the intensity plane are free
#pragma unroll
    for (int i = 0; i < NP; ++i) tile[geo.pixel_unit(i)] = ld_pair<G>(go_s + (size_t)s * NN + pix(i));
    if (LS) {
      const float* w = (s > 0 ? a.w_s + slotNN * (S - 1) + (size_t)(s - 1) * NN : a.Sp) + (size_t)y0 * N;
      for (int p = 4 * tid; p < LNN; p += 4 * T) *(float4*)(spS + p) = *(const float4*)(w + p);
    }
    __syncthreads();
    if (LS) {   // S_j^T of the slice's direction numerator and of its illumination
      float4* acc = a.acc + s * HW;
      bilinear_scatter<N, LR, T>(
          fy, fx,
          [&](int y, int x) {
            const float2 g = gt[G::pixel_slot(y, x)];
            return make_float4(g.x, g.y, spS[y * N + x], 0.f);
          },
          [&](int y, int x, float4 u) {
            atomicAdd(acc + (size_t)(ty + y0 + y) * a.W + (tx + x), make_float4(u.x, u.y, u.z, 0.f));
          });
    } else {
      float2* plane = a.gobj + s * HW;
      bilinear_scatter<N, LR, T>(
          fy, fx,
          [&](int y, int x) {
            const float2 g = gt[G::pixel_slot(y, x)];
            return make_float4(g.x, g.y, 0.f, 0.f);
          },
          [&](int y, int x, float4 u) {
            atomicAdd(plane + (size_t)(ty + y0 + y) * a.W + (tx + x), make_float2(u.x, u.y));
          });
    }
    if (a.gpos) {
      const float2* Os = a.obj + s * HW;
#pragma unroll 4
      for (int p = tid; p < LNN; p += T) {
        const int r = p / N, c = p % N;
        const float2* o = Os + (size_t)(ty + y0 + r) * a.W + (tx + c);
        const float2 O00 = __ldg(o), O01 = __ldg(o + 1), O10 = __ldg(o + a.W), O11 = __ldg(o + a.W + 1);
        const float2 dy = make_float2((1.f - fx) * (O10.x - O00.x) + fx * (O11.x - O01.x),
                                      (1.f - fx) * (O10.y - O00.y) + fx * (O11.y - O01.y));
        const float2 dx = make_float2((1.f - fy) * (O01.x - O00.x) + fy * (O11.x - O10.x),
                                      (1.f - fy) * (O01.y - O00.y) + fy * (O11.y - O10.y));
        const float2 g = gt[G::pixel_slot(r, c)];
        gyv += g.x * dy.x + g.y * dy.y;
        gxv += g.x * dx.x + g.y * dx.y;
      }
    }
  }
  if (a.gpos) {
    double w[2] = {(double)gyv, (double)gxv};
    block_sum<2>(w, red);
    if (tid == 0) {
      atomicAdd(a.gpos + 2 * j, (float)w[0]);
      atomicAdd(a.gpos + 2 * j + 1, (float)w[1]);
    }
  }
}

// Tangents of the multislice forward model for the LSQML step sizes: per mode,
// u starts as P_k d_0 and is carried through the slices as u <- H(u) o_s +
// inc_s d_s, v starts as dP_k o_0 and is carried as v <- H(v) o_s; at the exit
// plane the CTA sums |u|^2, Re(conj(u) v), |v|^2 over its pixels and the modes
// (u of the mode parked in scratch while v runs). With recompute each mode
// first runs through the slices to park its incident waves.
template <class G>
__global__ void __launch_bounds__(G::T, PairCtas<G>::n) k_step_ms(MsStepArgs a) {
  using SM = PairSmem<G>;
  using fp::C2;
  constexpr int N = G::N, T = G::T, NP = G::NP, NN = N * N, LR = G::LR, Q = G::Q;
  extern __shared__ __align__(16) unsigned char smem[];
  double* red = (double*)(smem + SM::red);
  float4* tile = (float4*)(smem + SM::tile);
  float2* tw = (float2*)(smem + SM::tw);
  const int slot = blockIdx.x / Q, tid = threadIdx.x;
  const G geo(tile, tw);
  const int y0 = LR * geo.q;
  double* out = a.part + (size_t)blockIdx.x * 3;
  if (!a.valid[slot]) {   // the same decision in every CTA of a cluster
    if (tid < 3) out[tid] = 0.0;
    return;
  }
  ms_begin<G>(tw, (uint64_t*)(red + 252));
  const int M = a.M, S = a.S;
  const bool rec = a.recompute != 0 && S > 1;
  const size_t slotNN = (size_t)slot * NN;
  auto pix = [&](int i) { return (y0 + geo.row(i)) * N + geo.col(i); };
  const float2* o_s = a.o_s + slotNN * S;
  const float2* d_s = a.d_s + slotNN * S;
  float4* u_s = (float4*)(a.u_s + slotNN + (size_t)y0 * N) + tid;
  auto inc = [&](int k, int s) {
    return (float4*)(a.in_s + ms_inc_offset(a.recompute != 0, slotNN, M, S, k, s, NN) + (size_t)y0 * N) + tid;
  };
  float2 A11 = make_float2(0.f, 0.f), A12 = A11, A22 = A11;
#pragma unroll 1
  for (int k = 0; k < M; ++k) {
#pragma unroll 1
    for (int t = rec ? -1 : 0; t < 2; ++t) {   // the incident waves, the object tangent u, the probe tangent v
      const float2* X = (t == 1 ? a.dP : a.probe) + (size_t)k * NN;
      const float2* Y = t == 0 ? d_s : o_s;
      C2 v[NP];
      ahead<NP, NP / 2>([&](int i) { return Two{ldg_pair<G>(X + pix(i)), ldg_pair<G>(Y + pix(i))}; },
                        [&](int i, const Two& x) { v[i] = exit_wave(x.a, x.b); });
#pragma unroll 1
      for (int s = 1; s < S; ++s) {
        __syncthreads();   // the tile is free
        geo.forward(v);
        mul_propagator(geo, v, a.Hf, false);
        __syncthreads();
        geo.inverse(v);
        if (t < 0) put_far<G>(v, inc(k, s));
        ahead<NP, 4>([&](int i) { return ldg_pair<G>(o_s + (size_t)s * NN + pix(i)); },
                     [&](int i, float4 o) {
                       v[i] = pack_pair(cmul(make_float2(v[i].re.x, v[i].im.x), make_float2(o.x, o.y)),
                                        cmul(make_float2(v[i].re.y, v[i].im.y), make_float2(o.z, o.w)));
                     });
        if (t == 0) {   // the slice's own direction as a source
          const float4* in = inc(k, s);
          ahead<NP, 4>([&](int i) { return Two{in[i * T], ldg_pair<G>(d_s + (size_t)s * NN + pix(i))}; },
                       [&](int i, const Two& x) {   // (the wave's units: re, re, im, im)
                         const float2 y0 = cmul(make_float2(x.a.x, x.a.z), make_float2(x.b.x, x.b.y));
                         const float2 y1 = cmul(make_float2(x.a.y, x.a.w), make_float2(x.b.z, x.b.w));
                         v[i] = {fp::add2(v[i].re, make_float2(y0.x, y1.x)), fp::add2(v[i].im, make_float2(y0.y, y1.y))};
                       });
        }
      }
      if (t == 0) {
#pragma unroll
        for (int i = 0; i < NP; ++i)
          A11 = fp::add2(A11, fp::fma2(v[i].re, v[i].re, fp::mul2(v[i].im, v[i].im)));
        put_far<G>(v, u_s);
      } else if (t == 1) {
#pragma unroll
        for (int i = 0; i < NP; ++i) {
          const float4 u = u_s[i * T];
          A22 = fp::add2(A22, fp::fma2(v[i].re, v[i].re, fp::mul2(v[i].im, v[i].im)));
          A12 = fp::fma2(make_float2(u.x, u.y), v[i].re, fp::fma2(make_float2(u.z, u.w), v[i].im, A12));   // Re(conj(u) v)
        }
      }
    }
  }
  double w[3] = {(double)(A11.x + A11.y), (double)(A12.x + A12.y), (double)(A22.x + A22.y)};
  block_sum<3>(w, red);
  if (tid == 0)
    for (int i = 0; i < 3; ++i) out[i] = w[i];
}

template <class G, class K, class A>
static cudaError_t launch_ms(K kernel, const A& a, cudaStream_t s, unsigned long long* done) {
  constexpr size_t sm = PairSmem<G>::bytes;
  cudaError_t e = smem_optin(kernel, sm, done);
  if (e != cudaSuccess) return e;
  if (a.nb <= 0) return cudaSuccess;
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
  cfg.numAttrs = G::Q > 1 ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, a);
}

// One line of a transform per lane group (kernels_ms_line.cuh), or packed line
// pairs? At 16 and 32 the packed form leaves a position 32 and 64 threads; while
// a launch has few positions per SM, all that counts is how long one takes.
// Measured on GB300, one line <- or -> packed, us per launch (slices x modes):
//   window 16, forward 3x2: 8 positions 9 <- 13, 512: 13 <- 15, 1024: 15 <- 17, 2048: 26 -> 23
//   window 16, gradients 3x2: 8: 18 <- 25, 400: 23 <- 27, 512: 26 <- 29, 1024: 36 -> 33
//   window 16, LSQML (pass and tangents) 3x2: 8: 40 <- 48, 256: 51 <- 56, 400: 60 -> 58
//   window 32, forward 3x2: 8: 15 <- 20, 256: 21 <- 23, 400: 39 -> 29
//   window 32, gradients 3x2: 8: 36 <- 46, 152: 38 <- 46, 200: 51 -> 49
//   window 32, LSQML 3x2: 8: 72 <- 82, 152: 78 <- 86, 200: 114 -> 90; 2x1: 8: 49 -> 48, 152: 60 -> 50
enum class MsUse { FORWARD, GRADIENT, LSQML };
inline bool ms_one_line(int N, int nb, int S, MsUse use) {
  const int sms = sm_count();
  if (N == 16) return nb <= (use == MsUse::FORWARD ? 6 : use == MsUse::GRADIENT ? 4 : 2) * sms;
  if (N == 32) return use == MsUse::LSQML ? S > 2 && nb <= sms : nb <= (use == MsUse::FORWARD ? 2 : 1) * sms;
  return false;
}

template <int N>
cudaError_t launch_pass1_ms(const MsArgs& a, cudaStream_t s) {
  const bool lsqml = a.mode == MODE_LSQML_GAUSS || a.mode == MODE_LSQML_POISSON;
  if constexpr (N <= 32)
    if (ms_one_line(N, a.nb, a.S, a.mode == MODE_FWD ? MsUse::FORWARD : lsqml ? MsUse::LSQML : MsUse::GRADIENT))
      return launch_pass1_ms_line<N>(a, s);
  using G = PairGeo<N>;
  static unsigned long long done[2] = {0, 0};
  return lsqml ? launch_ms<G>(k_pass1_ms<G, true>, a, s, &done[1])
               : launch_ms<G>(k_pass1_ms<G, false>, a, s, &done[0]);
}

template <int N>
cudaError_t launch_step_ms(const MsStepArgs& a, cudaStream_t s) {
  if constexpr (N <= 32)   // (it reads the incident waves in the order the pass left them)
    if (ms_one_line(N, a.nb, a.S, MsUse::LSQML)) return launch_step_ms_line<N>(a, s);
  using G = PairGeo<N>;
  static unsigned long long done = 0;
  return launch_ms<G>(k_step_ms<G>, a, s, &done);
}

}  // namespace ptycho
