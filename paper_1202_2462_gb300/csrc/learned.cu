// Kernels of the learned set-up: a gauge-covariant convolutional network that
// proposes near-kernel test vectors (trained to imitate the bootstrap set-up
// of Sec. 3; the bootstrap stays the fallback).
//
// Layer: out_a(x) = sum_b sum_h W[a][b][h] (T_h in_b)(x), with the parallel
// transports T_0 psi = psi, T_{+mu} psi(x) = U_mu(x) psi(x + mu),
// T_{-mu} psi(x) = U_mu(x - mu)^dagger psi(x - mu) (hop h = 0, 1 + 2 mu,
// 2 + 2 mu) and W[a][b][h] a complex 4 x 4 matrix on the spin index.  Gate
// between layers: psi(x) -> psi(x) / sqrt(1 + |psi(x)|^2) per channel and
// site.  Gradients: G_z = dL/dRe z + i dL/dIm z.
//
// Fields are FP32 complex in the blocked layout, channel c at c * 12V; links
// are the context's FP32 copy.  With few output channels one thread per (site,
// output channel) in the forward pass and per (site, input channel) in the input
// gradient; with more, and for the weight gradient, blocked products over sites
// (the tiled forms below), summed in a fixed order (deterministic).
#include "internal.h"
#include "pair.cuh"

namespace sapmg {

namespace {
using namespace pair;

// T_h psi_b at (blk, loc) into v (4 spins x 3 colours); links in storage type TG
template <class TG = float2>
__device__ __forceinline__ void transport_at(const Geom& g, const TG* __restrict__ U,
                                             const float2* __restrict__ f, int blk, int loc, int h,
                                             Cplx<float> (&v)[12]) {
  if (h == 0) {
    load_spinor<float>(f, blk, loc, v);
    return;
  }
  const int mu = (h - 1) >> 1;
  const int step = ((h - 1) & 1) ? -1 : 1;
  int nb, nl;
  neighbour(g, blk, loc, mu, step, nb, nl);
  Cplx<float> p[12], u[9];
  load_spinor<float>(f, nb, nl, p);
  if (step > 0) {
    load_link<float>(U, blk, mu, loc, u);
#pragma unroll
    for (int s = 0; s < 4; ++s)
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        Cplx<float> acc = u[a * 3] * p[s * 3];
        cfma(acc, u[a * 3 + 1], p[s * 3 + 1]);
        cfma(acc, u[a * 3 + 2], p[s * 3 + 2]);
        v[s * 3 + a] = acc;
      }
  } else {
    load_link<float>(U, nb, mu, nl, u);
#pragma unroll
    for (int s = 0; s < 4; ++s)
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        Cplx<float> acc = cmk(0.f, 0.f);
        cfma_conj(acc, u[a], p[s * 3]);
        cfma_conj(acc, u[3 + a], p[s * 3 + 1]);
        cfma_conj(acc, u[6 + a], p[s * 3 + 2]);
        v[s * 3 + a] = acc;
      }
  }
}

__device__ __forceinline__ int adjoint_hop(int h) { return h == 0 ? 0 : (((h - 1) & 1) ? h - 1 : h + 1); }

}  // namespace

// y_a = sum_b sum_h W[a][b][h] T_h x_b; grid (nblocks, cout), W[a] staged in shared memory.
// TG, TW: storage of the links and of the weights (FP32, or BF16 for inference);
// activations and accumulation in FP32.
template <class TG, class TW>
__global__ void __launch_bounds__(256) gconv_forward_kernel(Geom g, const TG* __restrict__ U,
                                                            const TW* __restrict__ W,
                                                            const float2* __restrict__ x, float2* __restrict__ y,
                                                            int cin) {
  extern __shared__ float2 ws[];                                // [cin][9][16]
  const int blk = MG_CLAMP(kBlock, blockIdx.x, g.nblocks), a = blockIdx.y, loc = threadIdx.x;
  const size_t fs = (size_t)g.V * 12;
  for (int e = loc; e < cin * 9 * 16; e += 256) {
    const Cplx<float> w = Io<float, TW>::ldc(W + (size_t)a * cin * 9 * 16 + e);
    ws[e] = make_float2(w.re, w.im);
  }
  __syncthreads();
  Cplx<float> acc[12];
#pragma unroll
  for (int k = 0; k < 12; ++k) acc[k] = cmk(0.f, 0.f);
  for (int b = 0; b < cin; ++b) {
    for (int h = 0; h < 9; ++h) {
      Cplx<float> v[12];
      transport_at<TG>(g, U, x + (size_t)b * fs, blk, loc, h, v);
      const float2* w = ws + (b * 9 + h) * 16;
#pragma unroll
      for (int s = 0; s < 4; ++s)
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          const Cplx<float> m = cmk(w[s * 4 + t].x, w[s * 4 + t].y);
#pragma unroll
          for (int c = 0; c < 3; ++c) cfma(acc[s * 3 + c], m, v[t * 3 + c]);
        }
    }
  }
  store_spinor<float>(y + (size_t)a * fs, blk, loc, acc);
}

// G_x_b = sum_h T_h^dagger (sum_a W[a][b][h]^dagger G_y_a); T_h^dagger = T_{adjoint hop}.
// grid (nblocks, cin), W[.][b] staged in shared memory.
__global__ void __launch_bounds__(256) gconv_backward_input_kernel(Geom g, const float2* __restrict__ U,
                                                                   const float2* __restrict__ W,
                                                                   const float2* __restrict__ gy,
                                                                   float2* __restrict__ gx, int cin, int cout) {
  extern __shared__ float2 ws[];                                // [cout][9][16] for this b
  const int blk = MG_CLAMP(kBlock, blockIdx.x, g.nblocks), b = blockIdx.y, loc = threadIdx.x;
  const size_t fs = (size_t)g.V * 12;
  for (int e = loc; e < cout * 9 * 16; e += 256) {
    const int a = e / (9 * 16), r = e % (9 * 16);
    ws[e] = W[((size_t)a * cin + b) * 9 * 16 + r];
  }
  __syncthreads();
  Cplx<float> acc[12];
#pragma unroll
  for (int k = 0; k < 12; ++k) acc[k] = cmk(0.f, 0.f);
  for (int h = 0; h < 9; ++h) {
    // q(y) = sum_a W[a][b][h]^dagger G_y_a(y) at y = the site T_{adjoint hop} reads from,
    // then transported: (T_adj q)(x)
    const int ha = adjoint_hop(h);
    int nb = blk, nl = loc;
    if (ha != 0) neighbour(g, blk, loc, (ha - 1) >> 1, ((ha - 1) & 1) ? -1 : 1, nb, nl);
    Cplx<float> q[12];
#pragma unroll
    for (int k = 0; k < 12; ++k) q[k] = cmk(0.f, 0.f);
    for (int a = 0; a < cout; ++a) {
      Cplx<float> p[12];
      load_spinor<float>(gy + (size_t)a * fs, nb, nl, p);
      const float2* w = ws + (a * 9 + h) * 16;
#pragma unroll
      for (int s = 0; s < 4; ++s)
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          const Cplx<float> m = cmk(w[t * 4 + s].x, w[t * 4 + s].y);   // (W^dagger)[s][t] = conj(W[t][s])
#pragma unroll
          for (int c = 0; c < 3; ++c) cfma_conj(q[s * 3 + c], m, p[t * 3 + c]);
        }
    }
    if (ha == 0) {
#pragma unroll
      for (int k = 0; k < 12; ++k) acc[k] = acc[k] + q[k];
    } else {
      const int mu = (ha - 1) >> 1;
      Cplx<float> u[9];
      if (((ha - 1) & 1) == 0) {                                // +mu: U_mu(x) q(x + mu)
        load_link<float>(U, blk, mu, loc, u);
#pragma unroll
        for (int s = 0; s < 4; ++s)
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            cfma(acc[s * 3 + c], u[c * 3], q[s * 3]);
            cfma(acc[s * 3 + c], u[c * 3 + 1], q[s * 3 + 1]);
            cfma(acc[s * 3 + c], u[c * 3 + 2], q[s * 3 + 2]);
          }
      } else {                                                  // -mu: U_mu(x - mu)^dagger q(x - mu)
        load_link<float>(U, nb, mu, nl, u);
#pragma unroll
        for (int s = 0; s < 4; ++s)
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            cfma_conj(acc[s * 3 + c], u[c], q[s * 3]);
            cfma_conj(acc[s * 3 + c], u[3 + c], q[s * 3 + 1]);
            cfma_conj(acc[s * 3 + c], u[6 + c], q[s * 3 + 2]);
          }
      }
    }
  }
  store_spinor<float>(gx + (size_t)b * fs, blk, loc, acc);
}

// ------------------------------------------------------------ tiled forms
// The layer and its input gradient as one blocked product: CTA (32 sites, sixteen
// output channels).  Per chunk of eight (input channel, hop) pairs every thread
// transports one pair's spinor at one site into shared memory, and thread
// (output channel, two sites) accumulates its 4 spins x 2 sites x 3 colours over
// the chunk's 32 input spins, five 16-byte loads for 24 complex products.  The
// kernels above transport every input once per output channel (1.7 times the
// needed flops, at the FP32 peak) or, for the gradient, read every output's
// gradient from L1 once per hop and input channel: 2.17 and 2.40 ms for 16 -> 16
// channels at 16^4, 58 Gflop, against 1.20 and 1.23 ms.  Spin matrices and transports commute, so the input
// gradient is the layer of the adjoint weights, G_x_b = sum_a sum_h
// W[a][b][adj h]^dagger T_h G_y_a (BWD).  FP32-bound.
constexpr int kPairs = 8, kTileSites = 32, kTileCh = 16;
constexpr int kLdW = kTileCh * 4 + 4;              // a row more of 64 bytes: the 16-byte stores of W spread

template <class TG, class TW, bool BWD, bool AL>
__global__ void __launch_bounds__(256, 2) gconv_tile_kernel(Geom g, const TG* __restrict__ U,
                                                            const TW* __restrict__ W, const float2* __restrict__ x,
                                                            float2* __restrict__ y, int cin, int cout) {
  // cin: channels of x; cout: channels of y (BWD: the layer's output and input channels); AL: y starts on 16 bytes
  // [pair, spin][colour][two sites]: (re, re, im, im); [pair, input spin][channel, spin]: (re, re, im, im)
  __shared__ __align__(16) float4 Ts[kPairs * 4][3][kTileSites / 2];
  extern __shared__ __align__(16) float4 Ws[];                        // [kPairs * 4][kLdW]
  const int tid = threadIdx.x, part = blockIdx.x & 7, a0 = blockIdx.y * kTileCh;
  const int blk = MG_CLAMP(kBlock, blockIdx.x >> 3, g.nblocks);
  const size_t fs = (size_t)g.V * 12;
  const int ch = tid >> 4, cg = tid & 15;                             // channel a0 + ch, sites 2 cg and 2 cg + 1
  const bool act = a0 + ch < cout;
  const int npair = cin * 9;
  P2 acc[4][3];                                                       // [spin][colour], the two sites packed
#pragma unroll
  for (int s = 0; s < 4; ++s)
#pragma unroll
    for (int c = 0; c < 3; ++c) acc[s][c].re = acc[s][c].im = f2(0.f);
  for (int p0 = 0; p0 < npair; p0 += kPairs) {
    __syncthreads();
    {
      const int p = tid >> 5, site = tid & 31, q = p0 + p;
      Cplx<float> v[12];
      if (q < npair) {
        transport_at<TG>(g, U, x + (size_t)(q / 9) * fs, blk, part * kTileSites + site, q % 9, v);
      } else {
#pragma unroll
        for (int k = 0; k < 12; ++k) v[k] = cmk(0.f, 0.f);
      }
#pragma unroll
      for (int t = 0; t < 4; ++t)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          float* o = reinterpret_cast<float*>(&Ts[p * 4 + t][c][site >> 1]) + (site & 1);
          o[0] = v[t * 3 + c].re;
          o[2] = v[t * 3 + c].im;
        }
    }
    for (int e = tid; e < kTileCh * kPairs * 16; e += 256) {
      const int a = e / (kPairs * 16), p = (e >> 4) & (kPairs - 1), so = e & 3, ti = (e >> 2) & 3, q = p0 + p;
      Cplx<float> w = cmk(0.f, 0.f);
      if (a0 + a < cout && q < npair) {
        if (BWD)
          w = conj(Io<float, TW>::ldc(W + (((size_t)(q / 9) * cout + a0 + a) * 9 + adjoint_hop(q % 9)) * 16 +
                                      ti * 4 + so));
        else
          w = Io<float, TW>::ldc(W + ((size_t)(a0 + a) * npair + q) * 16 + so * 4 + ti);
      }
      Ws[(p * 4 + ti) * kLdW + a * 4 + so] = make_float4(w.re, w.re, w.im, w.im);
    }
    __syncthreads();
    if (act) {
#pragma unroll 4
      for (int t = 0; t < kPairs * 4; ++t) {
        P2 tv[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          const float4 v = Ts[t][c][cg];
          tv[c].re = make_float2(v.x, v.y);
          tv[c].im = make_float2(v.z, v.w);
        }
#pragma unroll
        for (int s = 0; s < 4; ++s) {
          const float4 w = Ws[t * kLdW + ch * 4 + s];
          B2 u;
          u.r = make_float2(w.x, w.y);
          u.i = make_float2(w.z, w.w);
          u.ni = make_float2(-w.z, -w.w);
#pragma unroll
          for (int c = 0; c < 3; ++c) cmac(acc[s][c], u, tv[c]);
        }
      }
    }
  }
  if (!act) return;
  float2* o = y + (size_t)(a0 + ch) * fs + (size_t)blk * 12 * 256 + part * kTileSites + 2 * cg;
#pragma unroll
  for (int s = 0; s < 4; ++s)
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      float2* d = o + (s * 3 + c) * 256;
      const P2 v = acc[s][c];
      if (AL) {
        *reinterpret_cast<float4*>(d) = make_float4(v.re.x, v.im.x, v.re.y, v.im.y);
      } else {
        d[0] = make_float2(v.re.x, v.im.x);
        d[1] = make_float2(v.re.y, v.im.y);
      }
    }
}

constexpr size_t kTileSmem = sizeof(float4) * kPairs * 4 * kLdW;

// Weight gradient: CTA (sixteen (input channel, hop) pairs, RA output channels,
// slice of the sites).  Per sixteen sites the output gradients and the transported
// inputs (one pair and site a thread) are staged in shared memory and each thread
// accumulates a 4 x 4 tile, (output channel, its 4 spins) x (pair, its 4 spins),
// over the 48 (site, colour) terms; with RA < 16 the 256 / (16 RA) groups of
// threads share the terms.  The slices' sums are added in slice order by a second
// kernel, so the result is deterministic.  One CTA per (a, b, h) over all sites, the
// form below, transports every input once per output channel: 3.4 ms for 16 -> 16
// channels at 16^4, against 1.70 ms.
template <int RA>
__global__ void __launch_bounds__(256, 2) gconv_wgrad_tile_kernel(Geom g, const float2* __restrict__ U,
                                                                  const float2* __restrict__ x,
                                                                  const float2* __restrict__ gy,
                                                                  float2* __restrict__ part, int cin, int cout,
                                                                  int nslice) {
  constexpr int kS = 16, G = 16 / RA, LDT = 33, LDG = RA * 4 + 1;   // odd: the sites' 16-byte stores spread
  extern __shared__ __align__(16) float4 sm[];
  float4* Ts = sm;                                 // [site, colour][two spins][pair]: (re, re, im, im)
  float4* Gs = sm + kS * 3 * LDT;                  // [site, colour][channel, spin]: (re, re, im, im)
  const int tid = threadIdx.x, p0 = blockIdx.x * 16, a0 = blockIdx.y * RA, slice = blockIdx.z;
  const int npair = cin * 9, tile = tid % (16 * RA), grp = tid / (16 * RA), tp = tile & 15, ta = tile >> 4;
  const size_t fs = (size_t)g.V * 12;
  P2 tot[4][2];                                    // [spin of the gradient][two input spins, packed]
#pragma unroll
  for (int s = 0; s < 4; ++s)
#pragma unroll
    for (int t = 0; t < 2; ++t) tot[s][t].re = tot[s][t].im = f2(0.f);
  const int nchunk = g.nblocks * 16;
  for (int ch = slice; ch < nchunk; ch += nslice) {
    const int blk = ch >> 4, l0 = (ch & 15) * kS;
    __syncthreads();
    {
      const int p = tid >> 4, site = tid & 15, q = p0 + p;
      Cplx<float> v[12];
      if (q < npair) {
        transport_at(g, U, x + (size_t)(q / 9) * fs, blk, l0 + site, q % 9, v);
      } else {
#pragma unroll
        for (int k = 0; k < 12; ++k) v[k] = cmk(0.f, 0.f);
      }
#pragma unroll
      for (int t = 0; t < 2; ++t)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          const Cplx<float> a = v[2 * t * 3 + c], b = v[(2 * t + 1) * 3 + c];
          Ts[(site * 3 + c) * LDT + t * 16 + p] = make_float4(a.re, b.re, a.im, b.im);
        }
    }
    for (int e = tid; e < RA * 12 * kS; e += 256) {
      const int site = e & (kS - 1), k = (e / kS) % 12, a = e / (12 * kS);
      const float2 v = a0 + a < cout ? gy[(size_t)(a0 + a) * fs + ((size_t)blk * 12 + k) * 256 + l0 + site]
                                     : make_float2(0.f, 0.f);
      Gs[(site * 3 + k % 3) * LDG + a * 4 + k / 3] = make_float4(v.x, v.x, v.y, v.y);
    }
    __syncthreads();
    P2 acc[4][2];
#pragma unroll
    for (int s = 0; s < 4; ++s)
#pragma unroll
      for (int t = 0; t < 2; ++t) acc[s][t].re = acc[s][t].im = f2(0.f);
#pragma unroll 2
    for (int k = grp; k < kS * 3; k += G) {
      P2 xv[2];
      float2 nxi[2];
#pragma unroll
      for (int t = 0; t < 2; ++t) {
        const float4 v = Ts[k * LDT + t * 16 + tp];
        xv[t].re = make_float2(v.x, v.y);
        xv[t].im = make_float2(v.z, v.w);
        nxi[t] = make_float2(-v.z, -v.w);
      }
#pragma unroll
      for (int s = 0; s < 4; ++s) {
        const float4 w = Gs[k * LDG + ta * 4 + s];
        const float2 gr = make_float2(w.x, w.y), gi = make_float2(w.z, w.w);
#pragma unroll
        for (int t = 0; t < 2; ++t) {              // G_y conj(T x)
          acc[s][t].re = fma2(xv[t].re, gr, acc[s][t].re);
          acc[s][t].re = fma2(xv[t].im, gi, acc[s][t].re);
          acc[s][t].im = fma2(xv[t].re, gi, acc[s][t].im);
          acc[s][t].im = fma2(nxi[t], gr, acc[s][t].im);
        }
      }
    }
#pragma unroll
    for (int s = 0; s < 4; ++s)
#pragma unroll
      for (int t = 0; t < 2; ++t) {
        tot[s][t].re = add2(tot[s][t].re, acc[s][t].re);
        tot[s][t].im = add2(tot[s][t].im, acc[s][t].im);
      }
  }
  // the groups' totals, then W's layout: [slice][a][pair][s][t]
  auto put = [&](float2* o) {
#pragma unroll
    for (int s = 0; s < 4; ++s)
#pragma unroll
      for (int t = 0; t < 2; ++t) {
        o[s * 4 + 2 * t] = make_float2(tot[s][t].re.x, tot[s][t].im.x);
        o[s * 4 + 2 * t + 1] = make_float2(tot[s][t].re.y, tot[s][t].im.y);
      }
  };
  if (G > 1) {
    __syncthreads();
    float2* red = reinterpret_cast<float2*>(sm);                      // [G][16 RA tiles][16]
    put(red + (grp * 16 * RA + tile) * 16);
    __syncthreads();
    for (int e = tid; e < 16 * RA * 16; e += 256) {
      float re = 0.f, im = 0.f;
      for (int q = 0; q < G; ++q) { re += red[q * 256 * RA + e].x; im += red[q * 256 * RA + e].y; }
      const int pr = p0 + ((e >> 4) & 15), a = a0 + (e >> 8);
      if (pr < npair && a < cout)
        part[(((size_t)slice * cout + a) * npair + pr) * 16 + (e & 15)] = make_float2(re, im);
    }
  } else if (p0 + tp < npair && a0 + ta < cout) {
    put(part + (((size_t)slice * cout + a0 + ta) * npair + p0 + tp) * 16);
  }
}

__global__ void __launch_bounds__(256) gconv_wgrad_sum_kernel(const float2* __restrict__ part, size_t n, int nslice,
                                                              float2* __restrict__ gW) {
  const size_t i = (size_t)blockIdx.x * 256 + threadIdx.x;
  if (i >= n) return;
  float re[4] = {0.f, 0.f, 0.f, 0.f}, im[4] = {0.f, 0.f, 0.f, 0.f};   // four chains: loads in flight
  for (int s = 0; s < nslice; s += 4)
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (s + q < nslice) {
        const float2 v = part[(size_t)(s + q) * n + i];
        re[q] += v.x;
        im[q] += v.y;
      }
  gW[i] = make_float2((re[0] + re[1]) + (re[2] + re[3]), (im[0] + im[1]) + (im[2] + im[3]));
}

// The same for few products: CTA (a, b, h), a thread a site of every block.  The
// sums of sixteen blocks (48 products a thread) are added to the totals, those over
// warps and the CTA in a fixed order.
__global__ void __launch_bounds__(256, 2) gconv_wgrad_site_kernel(Geom g, const float2* __restrict__ U,
                                                                  const float2* __restrict__ x,
                                                                  const float2* __restrict__ gy,
                                                                  float2* __restrict__ gW, int cin) {
  const int id = blockIdx.x, h = id % 9, b = (id / 9) % cin, a = id / (9 * cin);
  const size_t fs = (size_t)g.V * 12;
  Cplx<float> tot[16];
#pragma unroll
  for (int k = 0; k < 16; ++k) tot[k] = cmk(0.f, 0.f);
  for (int b0 = 0; b0 < g.nblocks; b0 += 16) {
    Cplx<float> acc[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) acc[k] = cmk(0.f, 0.f);
    for (int blk = b0; blk < min(b0 + 16, g.nblocks); ++blk) {
      Cplx<float> v[12], p[12];
      transport_at(g, U, x + (size_t)b * fs, blk, threadIdx.x, h, v);
      load_spinor<float>(gy + (size_t)a * fs, blk, threadIdx.x, p);
#pragma unroll
      for (int s = 0; s < 4; ++s)
#pragma unroll
        for (int t = 0; t < 4; ++t)
#pragma unroll
          for (int c = 0; c < 3; ++c) cfma_conj(acc[s * 4 + t], v[t * 3 + c], p[s * 3 + c]);
    }
#pragma unroll
    for (int k = 0; k < 16; ++k) tot[k] = tot[k] + acc[k];
  }
  __shared__ float2 red[8][16];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    const float re = warp_sum(tot[k].re), im = warp_sum(tot[k].im);
    if (lane == 0) red[w][k] = make_float2(re, im);
  }
  __syncthreads();
  if (threadIdx.x < 16) {
    float re = 0.f, im = 0.f;
    for (int q = 0; q < 8; ++q) { re += red[q][threadIdx.x].x; im += red[q][threadIdx.x].y; }
    gW[(size_t)id * 16 + threadIdx.x] = make_float2(re, im);
  }
}

// y = x / sqrt(1 + |x(site)|^2) per channel and site
__global__ void gate_forward_kernel(Geom g, const float2* __restrict__ x, float2* __restrict__ y, int channels) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= g.V * channels) return;
  const int ch = (int)(i / g.V);
  const long long site = i % g.V;
  const int blk = (int)(site >> 8), loc = (int)(site & 255);
  const size_t fs = (size_t)g.V * 12;
  Cplx<float> p[12];
  load_spinor<float>(x + (size_t)ch * fs, blk, loc, p);
  float n = 0.f;
#pragma unroll
  for (int k = 0; k < 12; ++k) n += p[k].re * p[k].re + p[k].im * p[k].im;
  const float s = rsqrtf(1.f + n);
#pragma unroll
  for (int k = 0; k < 12; ++k) p[k] = s * p[k];
  store_spinor<float>(y + (size_t)ch * fs, blk, loc, p);
}

// G_x = s G_y - (1 + n)^(-3/2) Re<G_y, x>_site x, s = (1 + n)^(-1/2), n = |x(site)|^2
__global__ void gate_backward_kernel(Geom g, const float2* __restrict__ x, const float2* __restrict__ gy,
                                     float2* __restrict__ gx, int channels) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= g.V * channels) return;
  const int ch = (int)(i / g.V);
  const long long site = i % g.V;
  const int blk = (int)(site >> 8), loc = (int)(site & 255);
  const size_t fs = (size_t)g.V * 12;
  Cplx<float> p[12], q[12];
  load_spinor<float>(x + (size_t)ch * fs, blk, loc, p);
  load_spinor<float>(gy + (size_t)ch * fs, blk, loc, q);
  float n = 0.f, re = 0.f;
#pragma unroll
  for (int k = 0; k < 12; ++k) {
    n += p[k].re * p[k].re + p[k].im * p[k].im;
    re += q[k].re * p[k].re + q[k].im * p[k].im;
  }
  const float s = rsqrtf(1.f + n);
  const float c = re * s * s * s;
#pragma unroll
  for (int k = 0; k < 12; ++k) q[k] = s * q[k] + (-c) * p[k];
  store_spinor<float>(gx + (size_t)ch * fs, blk, loc, q);
}

// Adam on n real parameters (bias-corrected moments; step >= 1).
__global__ void adam_kernel(size_t n, float* __restrict__ p, const float* __restrict__ gr, float* __restrict__ m,
                            float* __restrict__ v, float lr, float b1, float b2, float eps, float c1, float c2) {
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const float gi = gr[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
  }
}

// Output channels (BWD: input channels) from which the tiled form runs: below, most of
// its sixteen channels a CTA would be idle and a thread per site transports little in
// vain.  Thread per site against tiled, 16^4 sites, FP32: layer 4 -> 4 155 and 192 us,
// 5 -> 5 235 and 235, 8 -> 8 572 and 361; input gradient 125 and 194, 185 and 239, 415
// and 371.
constexpr int kTiledFrom = 6, kTiledFromBwd = 8;

// The channels' worth of time that c channels take in tiles of sixteen: nine and more of a
// last tile keep all its warps' sub-partitions as busy as sixteen, up to eight as ten.
static int tile_cost(int c) {
  const int r = c % kTileCh;
  return c - r + (r == 0 ? 0 : r <= 8 ? 10 : kTileCh);
}
// The transports of one or two input channels are cheap to repeat: 16^4, 1 -> 9 92 and 114
// us, 12 118 and 139, 16 152 and 145, 24 225 and 218, 33 305 and 334; 2 -> 9 172 and 180;
// 4 -> 9 330 and 299.
static bool layer_tiled(int cin, int cout) {
  return cout >= kTiledFrom && (cin > 2 || 10 * tile_cost(cout) <= (cin == 1 ? 11 : 15) * cout);
}
// A thread per site reads each output's gradient once per input channel, from L2 while the
// outputs' gradients fit there (8 channels at 16^4: 9 470 and 539 us, 13 about equal, 16 802 and 628,
// 17 848 and 874, 24 1186 and 964), from HBM beyond (16 channels: 8 1224 and 733, 9 1374 and
// 1066, 17 2557 and 1724).
static bool input_gradient_tiled(const Geom& g, int cin, int cout) {
  if (cin < kTiledFromBwd) return false;
  return (size_t)cout * g.V * 96 > (64u << 20) || 10 * tile_cost(cin) <= 13 * cin;
}

template <class TG, class TW, bool BWD, bool AL>
static int gconv_tiled_run(const Geom& g, const void* U, const void* W, const void* x, void* y, int cin, int cout,
                           cudaStream_t s) {
  static bool attr = false;
  if (!attr) {
    SAPMG_CUDA_TRY(cudaFuncSetAttribute(gconv_tile_kernel<TG, TW, BWD, AL>,
                                        cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTileSmem));
    attr = true;
  }
  gconv_tile_kernel<TG, TW, BWD, AL><<<dim3(g.nblocks * 8, (cout + kTileCh - 1) / kTileCh), 256, kTileSmem, s>>>(
      g, (const TG*)U, (const TW*)W, (const float2*)x, (float2*)y, cin, cout);
  count_launches(1);
  SAPMG_CUDA_TRY(cudaGetLastError());
  return MG_OK;
}
template <class TG, class TW, bool BWD>
static int gconv_tiled(const Geom& g, const void* U, const void* W, const void* x, void* y, int cin, int cout,
                       cudaStream_t s) {
  return (reinterpret_cast<uintptr_t>(y) & 15) == 0 ? gconv_tiled_run<TG, TW, BWD, true>(g, U, W, x, y, cin, cout, s)
                                                    : gconv_tiled_run<TG, TW, BWD, false>(g, U, W, x, y, cin, cout, s);
}

template <class TG, class TW>
static int gconv_forward(const Geom& g, const void* U, const void* W, const void* x, void* y, int cin, int cout,
                         cudaStream_t s) {
  const size_t smem = sizeof(float2) * cin * 9 * 16;
  if (smem > 200 * 1024) return MG_ERR_ARG;
  if (layer_tiled(cin, cout)) return gconv_tiled<TG, TW, false>(g, U, W, x, y, cin, cout, s);
  static bool attr = false;
  if (!attr) {
    cudaFuncSetAttribute(gconv_forward_kernel<TG, TW>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    attr = true;
  }
  gconv_forward_kernel<TG, TW><<<dim3(g.nblocks, cout), 256, smem, s>>>(g, (const TG*)U, (const TW*)W,
                                                                         (const float2*)x, (float2*)y, cin);
  count_launches(1);
  SAPMG_CUDA_TRY(cudaGetLastError());
  return MG_OK;
}

int launch_gconv_forward(const Geom& g, const void* U, const void* W, const void* x, void* y, int cin, int cout,
                         cudaStream_t s) {
  return gconv_forward<float2, float2>(g, U, W, x, y, cin, cout, s);
}

int launch_gconv_forward_bf16(const Geom& g, const void* U, const void* W, const void* x, void* y, int cin, int cout,
                              cudaStream_t s) {
  return gconv_forward<__nv_bfloat162, __nv_bfloat162>(g, U, W, x, y, cin, cout, s);
}

// Slices of the sites of the weight gradient: two CTAs an SM over all tiles, no more
// than the sixteen-site chunks, at least four chunks a slice where there are that many.
static int wgrad_slices(const Geom& g, int cin, int cout) {
  const int tiles = (cin * 9 + 15) / 16 * (cout >= 16 ? (cout + 15) / 16 : (cout >= 4 ? (cout + 3) / 4 : cout));
  const int chunks = g.nblocks * 16;
  return std::max(1, std::min(304 / tiles, chunks / 4));       // one wave: a CTA more doubles the time
}
// Whether the tiles beat a CTA per (a, b, h), by the times (us) that describe both within a
// few percent for 1 to 64 channels on 16, 64 and 256 blocks: chunks of a slice, the
// slices' sum and what both kernels cost; waves of CTAs, the first one and a half
// bound by one CTA's own loads.  1 -> 16 channels at 8^4 25 us by sites and 57 by tiles, 1 ->
// 8 25 and 34, 64 -> 3 at 16^4 2630 and 5490; 16 -> 16 at 8^4 216 and 127.
static bool wgrad_tiled(const Geom& g, int cin, int cout) {
  const int ns = wgrad_slices(g, cin, cout);
  const double chunks = (g.nblocks * 16 + ns - 1) / ns, waves = (9 * cin * cout + 151) / 152;
  const double tiles = cout >= 16 ? 13.6 * chunks + 0.3 * ns
                     : cout >= 4 ? 8 + 5.0 * chunks + 0.2 * ns : 10 + 2.5 * chunks + 0.2 * ns;
  return 0.95 * tiles <= 7 + 0.84 * g.nblocks * std::max(1.43, waves);
}

size_t gconv_wgrad_bytes(const Geom& g, int max_channels) {
  size_t most = 0;
  for (int cin = 1; cin <= max_channels; ++cin)
    for (int cout = 1; cout <= max_channels; ++cout) {
      const int ns = wgrad_slices(g, cin, cout);
      if (ns > 1 && wgrad_tiled(g, cin, cout)) most = std::max(most, (size_t)ns * cout * cin * 9 * 16);
    }
  return most * sizeof(float2);
}

template <int RA>
static int wgrad_run(const Geom& g, const void* U, const void* x, const void* gy, float2* part, int cin, int cout,
                     int nslice, cudaStream_t s) {
  constexpr size_t stage = sizeof(float4) * 48 * (33 + RA * 4 + 1);
  constexpr size_t red = RA < 16 ? sizeof(float2) * 256 * 16 : 0;
  constexpr size_t smem = stage > red ? stage : red;
  static bool attr = false;
  if (!attr) {
    SAPMG_CUDA_TRY(cudaFuncSetAttribute(gconv_wgrad_tile_kernel<RA>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        (int)smem));
    attr = true;
  }
  gconv_wgrad_tile_kernel<RA><<<dim3((cin * 9 + 15) / 16, (cout + RA - 1) / RA, nslice), 256, smem, s>>>(
      g, (const float2*)U, (const float2*)x, (const float2*)gy, part, cin, cout, nslice);
  count_launches(1);
  return MG_OK;
}

int launch_gconv_backward(const Geom& g, const void* U, const void* W, const void* x, const void* gy, void* gx,
                          void* gW, void* work, int cin, int cout, cudaStream_t s) {
  const size_t smem = sizeof(float2) * cout * 9 * 16;
  if (smem > 200 * 1024) return MG_ERR_ARG;
  static bool attr = false;
  if (!attr) {
    cudaFuncSetAttribute(gconv_backward_input_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    attr = true;
  }
  if (gx) {
    if (input_gradient_tiled(g, cin, cout)) {
      const int rc = gconv_tiled<float2, float2, true>(g, U, W, gy, gx, cout, cin, s);
      if (rc != MG_OK) return rc;
    } else {
      gconv_backward_input_kernel<<<dim3(g.nblocks, cin), 256, smem, s>>>(
          g, (const float2*)U, (const float2*)W, (const float2*)gy, (float2*)gx, cin, cout);
      count_launches(1);
    }
  }
  if (gW && !wgrad_tiled(g, cin, cout)) {
    gconv_wgrad_site_kernel<<<cout * cin * 9, 256, 0, s>>>(g, (const float2*)U, (const float2*)x, (const float2*)gy,
                                                           (float2*)gW, cin);
    count_launches(1);
  } else if (gW) {
    const size_t n = (size_t)cout * cin * 9 * 16;
    const int nslice = wgrad_slices(g, cin, cout);
    float2* part = nslice > 1 ? (float2*)work : (float2*)gW;         // one slice is gW itself
    const int rc = cout >= 16 ? wgrad_run<16>(g, U, x, gy, part, cin, cout, nslice, s)
                 : cout >= 4  ? wgrad_run<4>(g, U, x, gy, part, cin, cout, nslice, s)
                              : wgrad_run<1>(g, U, x, gy, part, cin, cout, nslice, s);
    if (rc != MG_OK) return rc;
    if (nslice > 1) {
      gconv_wgrad_sum_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(part, n, nslice, (float2*)gW);
      count_launches(1);
    }
  }
  SAPMG_CUDA_TRY(cudaGetLastError());
  return MG_OK;
}

int launch_gate(const Geom& g, const void* x, const void* gy, void* out, int channels, cudaStream_t s) {
  const long long n = g.V * channels;
  const unsigned grid = (unsigned)((n + 255) / 256);
  if (gy) {
    gate_backward_kernel<<<grid, 256, 0, s>>>(g, (const float2*)x, (const float2*)gy, (float2*)out, channels);
  } else {
    gate_forward_kernel<<<grid, 256, 0, s>>>(g, (const float2*)x, (float2*)out, channels);
  }
  count_launches(1);
  SAPMG_CUDA_TRY(cudaGetLastError());
  return MG_OK;
}

int launch_adam(size_t n, float* p, const float* gr, float* m, float* v, double lr, double b1, double b2,
                double eps, int step, cudaStream_t s) {
  if (step < 1) return MG_ERR_ARG;
  const float c1 = (float)(1.0 - std::pow(b1, step)), c2 = (float)(1.0 - std::pow(b2, step));
  const unsigned grid = (unsigned)std::min<size_t>((n + 255) / 256, 152 * 8);
  adam_kernel<<<std::max(1u, grid), 256, 0, s>>>(n, p, gr, m, v, (float)lr, (float)b1, (float)b2, (float)eps, c1,
                                                  c2);
  count_launches(1);
  SAPMG_CUDA_TRY(cudaGetLastError());
  return MG_OK;
}

}  // namespace sapmg
