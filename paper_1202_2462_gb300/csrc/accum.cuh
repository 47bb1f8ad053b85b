// Scalars of the coarse GMRES beyond FP32 without FP64 instructions, one of which takes
// 64 cycles of an SM's sub-partition and made these short serial sums the longest
// part of a kernel on a short vector.
#pragma once
#include "common.cuh"

namespace sapmg {

// A sum across warps and CTAs: FP32 parts as an unevaluated pair of floats with
// error-free additions (Knuth, TAOCP vol. 2, 4.2.2).  The up to 1216 warp sums of a
// dot product, parallel vectors or orthogonal ones, 640 to 829440 elements, come out
// as the FP64 sum of the same parts does, bit for bit: 48 bits hold them.
template <class R> struct Acc;
template <> struct Acc<float> {
  float h, l;
  __device__ __forceinline__ static Acc of(float v) { return Acc{v, 0.f}; }
  __device__ __forceinline__ void add(Acc b) {
    const float s = __fadd_rn(h, b.h), t = __fsub_rn(s, h);
    const float e = __fadd_rn(__fsub_rn(h, __fsub_rn(s, t)), __fsub_rn(b.h, t));
    h = s;
    l = __fadd_rn(__fadd_rn(l, b.l), e);
  }
  __device__ __forceinline__ Acc from(int mask) const {
    return Acc{__shfl_xor_sync(0xffffffffu, h, mask), __shfl_xor_sync(0xffffffffu, l, mask)};
  }
  __device__ __forceinline__ float value() const { return h + l; }
  __device__ __forceinline__ double exact() const { return (double)h + (double)l; }
};
template <> struct Acc<double> {
  double v;
  __device__ __forceinline__ static Acc of(double x) { return Acc{x}; }
  __device__ __forceinline__ void add(Acc b) { v += b.v; }
  __device__ __forceinline__ Acc from(int mask) const { return Acc{__shfl_xor_sync(0xffffffffu, v, mask)}; }
  __device__ __forceinline__ double value() const { return v; }
  __device__ __forceinline__ double exact() const { return v; }
};

// 1 / s^2 of a basis vector with s = ||x|| / beta, and its products with sums: formed
// to 2^-45 and rounded to FP32 once, as a coefficient formed in FP64 is.
template <class R> struct Scale;
template <> struct Scale<float> {
  float h, l;
  __device__ __forceinline__ static Scale one() { return Scale{1.f, 0.f}; }
  __device__ __forceinline__ static Scale of(Acc<float> xx, float invb) {     // ||x||^2, 1 / beta
    const float q = __fmul_rn(invb, invb), ql = fmaf(invb, invb, -q);
    const float s = __fmul_rn(xx.h, q), sl = fmaf(xx.h, q, -s) + (xx.h * ql + xx.l * q);
    if (!(s > 1e-37f)) return Scale{0.f, 0.f};                                // 1 / s would overflow
    const float r = 1.f / s;
    return Scale{r, r * (fmaf(-s, r, 1.f) - sl * r)};
  }
  __device__ __forceinline__ float times(Acc<float> d) const {
    const float p = __fmul_rn(d.h, h);
    return p + (fmaf(d.h, h, -p) + (d.h * l + d.l * h));
  }
};
template <> struct Scale<double> {
  double v;
  __device__ __forceinline__ static Scale one() { return Scale{1.0}; }
  __device__ __forceinline__ static Scale of(Acc<double> xx, double invb) {
    const double s = xx.v * invb * invb;
    return Scale{s > 0.0 ? 1.0 / s : 0.0};
  }
  __device__ __forceinline__ double times(Acc<double> d) const { return d.v * v; }
};
static_assert(sizeof(Scale<float>) == 8 && sizeof(Scale<double>) == 8, "stored in the place of a double");

}  // namespace sapmg
