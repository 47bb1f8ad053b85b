// K8: vector kernels of the Krylov solvers (Sec. 2 and Sec. 4: GMRES on the
// coarse grid, flexible GMRES outside), batched over right-hand sides: one
// launch serves all R systems, each with its own vectors and scalars.
//
// A batched vector is R fields stored back to back (field r at base + r*stride).
// Reductions are deterministic: every CTA writes its partial sums, one CTA per
// right-hand side adds them in a fixed order.  Per-thread and per-warp partial
// sums use the vector's own precision; CTA-level and final sums use FP64.
#include "internal.h"
#include "blas.h"
#include "accum.cuh"
#include "hessenberg.cuh"
#include "pdl.cuh"

#include <type_traits>

namespace sapmg {

template <class T2> struct RealOf;
template <> struct RealOf<double2> { typedef double R; };
template <> struct RealOf<float2> { typedef float R; };

// up to 16 vectors per launch
constexpr int kChunk = 16;
template <class T2> struct Ptrs8 { const T2* p[kChunk]; };

// CTAs per right-hand side of a reduction over n elements, slots double2 of
// partial sums each: 8 elements a thread, R * CTAs within the partial buffer.
// A vector too short to give every SM a CTA that way (152 over all right-hand
// sides) is cut finer, down to one element a thread: there the pass takes the
// latency of one thread's loads and not bandwidth (the 20480-entry coarse
// vectors of 16^3 x 32: a 12-vector dot pass 24.9 us on 5 CTAs).
static int reduce_ctas(size_t n, int R, size_t slots = kChunk) {
  const size_t r = (size_t)std::max(R, 1);
  const size_t per = std::max<size_t>(1, kPartialSums / slots / r);
  const size_t fill = std::min<size_t>((n + 255) / 256, (152 + r - 1) / r);
  return (int)std::max<size_t>(1, std::min<size_t>(std::max((n + 2047) / 2048, fill), per));
}

// Dependent launch (pdl.cuh) below one CTA an SM, where the launch is a large part of a
// kernel: one field's cycle on 512 coarse sites 463 -> 447 us with the coarse product
// (coarse_tma.cu); the chain of 12 fields did not gain.
static bool starts_early(dim3 grid) { return grid.x * grid.y <= 152; }

// Reductions end inside the kernel that forms the partial sums: the CTA of a
// right-hand side that arrives last (a counter per right-hand side behind the
// partial sums; atomicInc wraps it back to 0) adds the CTAs' parts in their
// fixed order, so the result does not depend on which CTA that is.  A separate
// one-CTA kernel for it cost a launch and 7.8 us (12 sums one after the other).
__device__ __forceinline__ bool last_cta(double2* partial, int r) {
  __shared__ int last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0)
    last = atomicInc(reinterpret_cast<unsigned*>(partial + kPartialSums) + r, gridDim.x - 1) == gridDim.x - 1;
  __syncthreads();
  if (last) __threadfence();
  return last != 0;
}

// The calling warp's sum of slot j over the CTAs' partial sums of right-hand side r.
__device__ __forceinline__ double2 sum_slot(const double2* partial, int r, int slots, int j) {
  double a = 0, b = 0;
#pragma unroll 4
  for (int c = threadIdx.x & 31; c < (int)gridDim.x; c += 32) {
    const double2 v = __ldcg(partial + ((size_t)r * gridDim.x + c) * slots + j);
    a += v.x;
    b += v.y;
  }
  return make_double2(warp_sum(a), warp_sum(b));
}

// where the K sums of a dot pass go: out[r*ldo + j] = (mode 1: out +) the sum,
// out2[r*ldo + j] = the sum if out2 != nullptr
struct DotOut {
  double2* out;
  double2* out2;
  int ldo, mode;
};
template <int K>
__device__ __forceinline__ void finish_dots(double2* partial, const DotOut& d) {
  const int r = blockIdx.y;
  if (!last_cta(partial, r)) return;
  for (int j = threadIdx.x >> 5; j < K; j += 8) {
    const double2 t = sum_slot(partial, r, kChunk, j);
    if ((threadIdx.x & 31) == 0) {
      if (d.out) {
        double2* o = d.out + (size_t)r * d.ldo + j;
        if (d.mode == 1) { o->x += t.x; o->y += t.y; }
        else *o = t;
      }
      if (d.out2) d.out2[(size_t)r * d.ldo + j] = t;
    }
  }
}

template <class T2, int K>
__global__ void __launch_bounds__(256) multidot_partial(Ptrs8<T2> v, const T2* __restrict__ w, size_t n,
                                                        size_t vstride, size_t wstride,
                                                        double2* __restrict__ partial, DotOut dout) {
  typedef typename RealOf<T2>::R R;
  const int r = blockIdx.y;
  const T2* wr = w + r * wstride;
  R are[K], aim[K];
#pragma unroll
  for (int j = 0; j < K; ++j) are[j] = aim[j] = 0;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    // issue every load of the element before any arithmetic (memory-level parallelism)
    T2 a[K];
#pragma unroll
    for (int j = 0; j < K; ++j) a[j] = __ldg(&v.p[j][r * vstride + i]);
    const T2 x = __ldg(&wr[i]);
#pragma unroll
    for (int j = 0; j < K; ++j) {
      are[j] = fma(a[j].x, x.x, fma(a[j].y, x.y, are[j]));
      aim[j] = fma(a[j].x, x.y, fma(-a[j].y, x.x, aim[j]));
    }
  }
  __shared__ double red[8][2 * K];
  const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // warp trees in the vector's precision (FP64 arithmetic is scarce), CTA sum in FP64
#pragma unroll
  for (int j = 0; j < K; ++j) {
    const R s = warp_sum(are[j]);
    const R m = warp_sum(aim[j]);
    if (lane == 0) { red[wid][2 * j] = (double)s; red[wid][2 * j + 1] = (double)m; }
  }
  __syncthreads();
  if (threadIdx.x < K) {
    double s = 0, m = 0;
    for (int q = 0; q < 8; ++q) { s += red[q][2 * threadIdx.x]; m += red[q][2 * threadIdx.x + 1]; }
    partial[((size_t)r * gridDim.x + blockIdx.x) * kChunk + threadIdx.x] = make_double2(s, m);
  }
  finish_dots<K>(partial, dout);
}

// FP32 vectors with an even length: two complex numbers per 16-byte load.
template <int K>
__global__ void __launch_bounds__(256) multidot_partial_f4(Ptrs8<float2> v, const float2* __restrict__ w, size_t n,
                                                           size_t vstride, size_t wstride,
                                                           double2* __restrict__ partial, DotOut dout) {
  const int r = blockIdx.y;
  const float4* wr = reinterpret_cast<const float4*>(w + r * wstride);
  const size_t n4 = n / 2;
  float are[K], aim[K];
#pragma unroll
  for (int j = 0; j < K; ++j) are[j] = aim[j] = 0.f;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n4; i += (size_t)gridDim.x * blockDim.x) {
    float4 a[K];
#pragma unroll
    for (int j = 0; j < K; ++j) a[j] = __ldg(reinterpret_cast<const float4*>(v.p[j] + r * vstride) + i);
    const float4 x = __ldg(wr + i);
#pragma unroll
    for (int j = 0; j < K; ++j) {
      are[j] = fmaf(a[j].x, x.x, fmaf(a[j].y, x.y, fmaf(a[j].z, x.z, fmaf(a[j].w, x.w, are[j]))));
      aim[j] = fmaf(a[j].x, x.y, fmaf(-a[j].y, x.x, fmaf(a[j].z, x.w, fmaf(-a[j].w, x.z, aim[j]))));
    }
  }
  __shared__ double red[8][2 * K];
  const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
  for (int j = 0; j < K; ++j) {
    const float s = warp_sum(are[j]);
    const float m = warp_sum(aim[j]);
    if (lane == 0) { red[wid][2 * j] = (double)s; red[wid][2 * j + 1] = (double)m; }
  }
  __syncthreads();
  if (threadIdx.x < K) {
    double s = 0, m = 0;
    for (int q = 0; q < 8; ++q) { s += red[q][2 * threadIdx.x]; m += red[q][2 * threadIdx.x + 1]; }
    partial[((size_t)r * gridDim.x + blockIdx.x) * kChunk + threadIdx.x] = make_double2(s, m);
  }
  finish_dots<K>(partial, dout);
}

template <class T2, int K>
static void md_launch(dim3 grid, const Ptrs8<T2>& p, const T2* w, size_t n, size_t vs, size_t ws, double2* part,
                      const DotOut& d, cudaStream_t s) {
  multidot_partial<T2, K><<<grid, 256, 0, s>>>(p, w, n, vs, ws, part, d); count_launches(1);
}

template <class T2, int K>
static void md_launch_any(bool vec4, dim3 grid, const Ptrs8<T2>& p, const T2* w, size_t n, size_t vs, size_t ws,
                          double2* part, const DotOut& d, cudaStream_t s) {
  if constexpr (std::is_same<T2, float2>::value) {
    if (vec4) {
      multidot_partial_f4<K><<<grid, 256, 0, s>>>(p, w, n, vs, ws, part, d); count_launches(1);
      return;
    }
  }
  md_launch<T2, K>(grid, p, w, n, vs, ws, part, d, s);
}

template <class T2>
static int multidot_t(const BVec& b, const void* const* v, int k, const void* w, double2* out, int ldo, int mode,
                      double2* out2, double2* partial, cudaStream_t s) {
  // two complex numbers per load when every vector is 16-byte aligned and n is even
  bool vec4 = (b.n % 2 == 0) && (b.vstride % 2 == 0) && (b.wstride % 2 == 0) &&
              ((reinterpret_cast<uintptr_t>(w) & 15) == 0);
  for (int j = 0; j < k; ++j) vec4 = vec4 && ((reinterpret_cast<uintptr_t>(v[j]) & 15) == 0);
  const int ncta = reduce_ctas(vec4 ? b.n / 2 : b.n, b.R);
  const dim3 grid(ncta, b.R);
  for (int j0 = 0; j0 < k; j0 += kChunk) {
    const int kk = std::min(kChunk, k - j0);
    Ptrs8<T2> p;
    for (int j = 0; j < kChunk; ++j) p.p[j] = (const T2*)v[j0 + std::min(j, kk - 1)];
    const T2* wp = (const T2*)w;
    const DotOut d{out ? out + j0 : nullptr, out2 ? out2 + j0 : nullptr, ldo, mode};
#define SAPMG_MD(K) case K: md_launch_any<T2, K>(vec4, grid, p, wp, b.n, b.vstride, b.wstride, partial, d, s); break;
    switch (kk) {
      SAPMG_MD(1) SAPMG_MD(2) SAPMG_MD(3) SAPMG_MD(4) SAPMG_MD(5) SAPMG_MD(6) SAPMG_MD(7) SAPMG_MD(8)
      SAPMG_MD(9) SAPMG_MD(10) SAPMG_MD(11) SAPMG_MD(12) SAPMG_MD(13) SAPMG_MD(14) SAPMG_MD(15)
      default: md_launch_any<T2, 16>(vec4, grid, p, wp, b.n, b.vstride, b.wstride, partial, d, s); break;
    }
#undef SAPMG_MD
  }
  SAPMG_CUDA_TRY(cudaGetLastError());
  return MG_OK;
}

int blas_multidot(int type, const BVec& b, const void* const* v, int k, const void* w, double2* out, int ldo,
                  int mode, double2* out2, double2* partial, cudaStream_t s) {
  if (k <= 0 || b.R <= 0) return MG_OK;
  count_bytes((double)(k + (v[k - 1] == w ? 0 : 1)) * b.n * b.R * (type == P64 ? 16 : 8));
  if (type == P64) return multidot_t<double2>(b, v, k, w, out, ldo, mode, out2, partial, s);
  if (type == P32) return multidot_t<float2>(b, v, k, w, out, ldo, mode, out2, partial, s);
  return MG_ERR_ARG;
}

// w[r] += sign * sum_j coeff[r*ldc + j] v_j[r]; with partial != nullptr also
// nrm[r*ldn] = ||w_new||^2.
template <class T2, int K>
__global__ void __launch_bounds__(256) multiaxpy_kernel(T2* __restrict__ w, Ptrs8<T2> v,
                                                        const double2* __restrict__ coeff, int ldc, double sign,
                                                        size_t n, size_t vstride, size_t wstride,
                                                        double2* __restrict__ partial, DotOut dout) {
  typedef typename RealOf<T2>::R R;
  const int r = blockIdx.y;
  R cr[K], ci[K];
#pragma unroll
  for (int j = 0; j < K; ++j) {
    const double2 c = coeff[(size_t)r * ldc + j];
    cr[j] = (R)(sign * c.x);
    ci[j] = (R)(sign * c.y);
  }
  T2* wr = w + r * wstride;
  R nn = 0;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    T2 x = wr[i];
#pragma unroll
    for (int j = 0; j < K; ++j) {
      const T2 a = v.p[j][r * vstride + i];
      x.x = fma(cr[j], a.x, fma(-ci[j], a.y, x.x));
      x.y = fma(cr[j], a.y, fma(ci[j], a.x, x.y));
    }
    wr[i] = x;
    nn = fma(x.x, x.x, fma(x.y, x.y, nn));
  }
  if (partial) {
    __shared__ double red[8];
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const R t = warp_sum(nn);
    if (lane == 0) red[wid] = (double)t;
    __syncthreads();
    if (threadIdx.x == 0) {
      double sum = 0;
      for (int q = 0; q < 8; ++q) sum += red[q];
      partial[((size_t)r * gridDim.x + blockIdx.x) * kChunk] = make_double2(sum, 0.0);
    }
    finish_dots<1>(partial, dout);
  }
}

// Streaming kernels: about 8 CTAs of 256 threads per SM over all right-hand
// sides, 4 elements a thread; a short vector one element a thread until every
// SM has a CTA (as reduce_ctas).
static dim3 stream_grid(size_t n, int R) {
  const size_t r = (size_t)std::max(R, 1);
  const size_t per = std::max<size_t>(16, (size_t)152 * 8 / r);
  const size_t fill = std::min<size_t>((n + 255) / 256, (152 + r - 1) / r);
  return dim3((unsigned)std::max<size_t>(1, std::min<size_t>(std::max((n + 1023) / 1024, fill), per)), R);
}

template <class T2, int K>
static void ma_launch(dim3 g, T2* w, const Ptrs8<T2>& p, const double2* c, int ldc, double sign, const BVec& b,
                      double2* partial, const DotOut& d, cudaStream_t s) {
  multiaxpy_kernel<T2, K><<<g, 256, 0, s>>>(w, p, c, ldc, sign, b.n, b.vstride, b.wstride, partial, d);
  count_launches(1);
}

template <class T2>
static int multiaxpy_t(const BVec& b, void* w, const void* const* v, int k, const double2* coeff, int ldc,
                       double sign, double2* nrm2, int ldn, double2* partial, cudaStream_t s) {
  const dim3 g = nrm2 ? dim3(reduce_ctas(b.n, b.R), b.R) : stream_grid(b.n, b.R);
  for (int j0 = 0; j0 < k; j0 += kChunk) {
    const int kk = std::min(kChunk, k - j0);
    const bool last = j0 + kChunk >= k;
    Ptrs8<T2> p;
    for (int j = 0; j < kChunk; ++j) p.p[j] = (const T2*)v[j0 + std::min(j, kk - 1)];
    const double2* c = coeff + j0;
    double2* part = (last && nrm2) ? partial : nullptr;
    const DotOut d{nrm2, nullptr, ldn, 0};
#define SAPMG_MA(K) case K: ma_launch<T2, K>(g, (T2*)w, p, c, ldc, sign, b, part, d, s); break;
    switch (kk) {
      SAPMG_MA(1) SAPMG_MA(2) SAPMG_MA(3) SAPMG_MA(4) SAPMG_MA(5) SAPMG_MA(6) SAPMG_MA(7) SAPMG_MA(8)
      SAPMG_MA(9) SAPMG_MA(10) SAPMG_MA(11) SAPMG_MA(12) SAPMG_MA(13) SAPMG_MA(14) SAPMG_MA(15)
      default: ma_launch<T2, 16>(g, (T2*)w, p, c, ldc, sign, b, part, d, s); break;
    }
#undef SAPMG_MA
  }
  SAPMG_CUDA_TRY(cudaGetLastError());
  return MG_OK;
}

int blas_multiaxpy(int type, const BVec& b, void* w, const void* const* v, int k, const double2* coeff, int ldc,
                   double sign, cudaStream_t s) {
  if (k <= 0 || b.R <= 0) return MG_OK;
  count_bytes((double)(k + 2) * b.n * b.R * (type == P64 ? 16 : 8));
  if (type == P64) return multiaxpy_t<double2>(b, w, v, k, coeff, ldc, sign, nullptr, 0, nullptr, s);
  if (type == P32) return multiaxpy_t<float2>(b, w, v, k, coeff, ldc, sign, nullptr, 0, nullptr, s);
  return MG_ERR_ARG;
}

int blas_multiaxpy_norm(int type, const BVec& b, void* w, const void* const* v, int k, const double2* coeff, int ldc,
                        double sign, double2* nrm2, int ldn, double2* partial, cudaStream_t s) {
  if (k <= 0 || b.R <= 0) return MG_OK;
  count_bytes((double)(k + 2) * b.n * b.R * (type == P64 ? 16 : 8));
  if (type == P64) return multiaxpy_t<double2>(b, w, v, k, coeff, ldc, sign, nrm2, ldn, partial, s);
  if (type == P32) return multiaxpy_t<float2>(b, w, v, k, coeff, ldc, sign, nrm2, ldn, partial, s);
  return MG_ERR_ARG;
}

// y[r] = a_r x[r] + b_r y[r] with per-RHS scalars passed by value; x and y may
// differ in element type; b_r = 0 means y[r] is not read.
template <class TX, class TY>
__global__ void axpby_kernel(Scal32 a, const TX* __restrict__ x, Scal32 b, TY* __restrict__ y, size_t n,
                             size_t xs, size_t ys) {
  typedef typename RealOf<TY>::R R;
  const int r = blockIdx.y;
  const R ar = (R)a.v[r].x, ai = (R)a.v[r].y, br = (R)b.v[r].x, bi = (R)b.v[r].y;
  const bool yz = (b.v[r].x == 0.0 && b.v[r].y == 0.0);
  // real scalars (every solver update): half the products, which for FP64, where
  // they were the bound, is 1.72 -> 1.11 ms for x64 += s e32 (12 fields of 7.96 M) and
  // 1.32 -> 0.72 ms for r = b - r in FP64
  const bool real = a.v[r].y == 0.0 && b.v[r].y == 0.0;
  const TX* xr = x + r * xs;
  TY* yr = y + r * ys;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const TX u = xr[i];
    const R ux = (R)u.x, uy = (R)u.y;
    TY v;
    v.x = v.y = 0;
    if (!yz) v = yr[i];
    TY o;
    if (real) {
      o.x = ar * ux + br * v.x;
      o.y = ar * uy + br * v.y;
    } else {
      o.x = ar * ux - ai * uy + br * v.x - bi * v.y;
      o.y = ar * uy + ai * ux + br * v.y + bi * v.x;
    }
    yr[i] = o;
  }
}

int blas_axpby2(int tx, const Scal32& a, const void* x, size_t xs, int ty, const Scal32& b, void* y, size_t ys,
                size_t n, int R, cudaStream_t s) {
  if (n == 0 || R == 0) return MG_OK;
  if (R > 32) return MG_ERR_ARG;
  bool yread = false;
  for (int r = 0; r < R; ++r) yread = yread || b.v[r].x != 0.0 || b.v[r].y != 0.0;
  count_bytes((double)n * R * ((tx == P64 ? 16 : 8) + (ty == P64 ? 16 : 8) * (yread ? 2 : 1)));
  const dim3 g = stream_grid(n, R);
  if (tx == P64 && ty == P64) { axpby_kernel<double2, double2><<<g, 256, 0, s>>>(a, (const double2*)x, b, (double2*)y, n, xs, ys); count_launches(1); }
  else if (tx == P32 && ty == P32) { axpby_kernel<float2, float2><<<g, 256, 0, s>>>(a, (const float2*)x, b, (float2*)y, n, xs, ys); count_launches(1); }
  else if (tx == P32 && ty == P64) { axpby_kernel<float2, double2><<<g, 256, 0, s>>>(a, (const float2*)x, b, (double2*)y, n, xs, ys); count_launches(1); }
  else if (tx == P64 && ty == P32) { axpby_kernel<double2, float2><<<g, 256, 0, s>>>(a, (const double2*)x, b, (float2*)y, n, xs, ys); count_launches(1); }
  else return MG_ERR_ARG;
  SAPMG_CUDA_TRY(cudaGetLastError());
  return MG_OK;
}

// out[r] = x[r] / sqrt(nrm2[r*ldn].x); store[r*lds] = (sqrt(...), 0).  A vanishing
// norm gives a zero vector and a zero stored norm (invariant Krylov space).
template <class T2>
__global__ void normalize_kernel(const T2* __restrict__ x, T2* __restrict__ out, const double2* __restrict__ nrm2,
                                 int ldn, double2* __restrict__ store, int lds, size_t n, size_t stride) {
  typedef typename RealOf<T2>::R R;
  const int r = blockIdx.y;
  const double nn = sqrt(fmax(nrm2[(size_t)r * ldn].x, 0.0));
  const R inv = nn > 0.0 ? (R)(1.0 / nn) : (R)0;
  if (blockIdx.x == 0 && threadIdx.x == 0 && store) store[(size_t)r * lds] = make_double2(nn, 0.0);
  const T2* xr = x + r * stride;
  T2* o = out + r * stride;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    T2 u = xr[i];
    u.x *= inv;
    u.y *= inv;
    o[i] = u;
  }
}

int blas_normalize(int type, const BVec& b, const void* x, void* out, const double2* nrm2, int ldn, double2* store,
                   int lds, cudaStream_t s) {
  count_bytes(2.0 * b.n * b.R * (type == P64 ? 16 : 8));
  const dim3 g = stream_grid(b.n, b.R);
  if (type == P64) { normalize_kernel<double2><<<g, 256, 0, s>>>((const double2*)x, (double2*)out, nrm2, ldn, store, lds, b.n, b.wstride); count_launches(1); }
  else if (type == P32) { normalize_kernel<float2><<<g, 256, 0, s>>>((const float2*)x, (float2*)out, nrm2, ldn, store, lds, b.n, b.wstride); count_launches(1); }
  else return MG_ERR_ARG;
  SAPMG_CUDA_TRY(cudaGetLastError());
  return MG_OK;
}

// Least-squares solve of the (m+1) x m Hessenberg system min ||beta e1 - H y||
// of fixed-step GMRES, one warp per right-hand side (hessenberg.cuh).  H for
// RHS r at H + r*ldr, column-major with leading dimension ldh; beta2[r].x =
// ||b_r||^2; y[r*ldy + j].  norms != nullptr: H holds the raw dots of
// blas_arnoldi_step (pairs: as sums of two floats) and norms[r*ldr + j] = (||x||^2,
// 1/beta) of basis vector j >= 1, whose norm is s_j = ||x|| / beta: with the entries
// h_ij / s_i and ||x_{j+1}|| the solution is in the basis vectors as they are.
// Columns after a zero subdiagonal entry are unused.  m <= 32.
// Latency-bound (an FP64 instruction of a warp takes 64 cycles of its
// sub-partition): 12 steps on one vector 73 us with two square roots and
// divisions a step and serial loads, 27 us with one reciprocal square root a
// step and every load and division issued for all columns at once.
__global__ void __launch_bounds__(32) hessenberg_solve_kernel(const double2* __restrict__ Hall, int ldh, int ldr,
                                                              int m, const double2* __restrict__ beta2,
                                                              const double2* __restrict__ norms, int pairs,
                                                              double2* __restrict__ yall, int ldy) {
  __shared__ double hr[33 * 32], hi[33 * 32];
  const int r = blockIdx.x, lane = threadIdx.x;
  const double2* Hin = Hall + (size_t)r * ldr;
  double2* y = yall + (size_t)r * ldy;
  pdl_begin();
  const double beta = sqrt(fmax(__ldcg(beta2 + r).x, 0.0));
  if (beta == 0.0) {
    if (lane < m) y[lane] = make_double2(0, 0);
    return;
  }
  double sub = 1.0, is = 1.0;                            // H_{lane+1,lane}; 1 / s_lane
  if (norms) {
    const double2* nv = norms + (size_t)r * ldr;
    if (lane > 0 && lane < m) {
      const double2 q = __ldcg(nv + lane);
      const double t = sqrt(q.x) * q.y;
      is = t > 0.0 ? 1.0 / t : 0.0;
    }
    if (lane < m) sub = sqrt(__ldcg(nv + lane + 1).x);
  } else if (lane < m) {
    sub = __ldcg(Hin + lane + 1 + lane * ldh).x;
  }
  const unsigned zero = __ballot_sync(0xffffffffu, sub == 0.0);
  const int mm = zero ? __ffs(zero) : m;                 // columns up to the first zero subdiagonal entry
  for (int k = 0; k < mm; ++k) {                         // lane = row
    double2 v = make_double2(0, 0);
    if (lane <= k) {
      v = __ldcg(Hin + lane + k * ldh);
      if (pairs) {
        const float4 f = *reinterpret_cast<const float4*>(&v);
        v = make_double2((double)f.x + (double)f.y, (double)f.z + (double)f.w);
      }
      if (norms) { v.x *= is; v.y *= is; }
    }
    hr[lane + k * 33] = v.x;
    hi[lane + k * 33] = v.y;
    if (lane == 0) hr[32 + k * 33] = hi[32 + k * 33] = 0.0;
  }
  __syncwarp();
  if (lane < mm) {
    hr[lane + 1 + lane * 33] = sub;
    hi[lane + 1 + lane * 33] = 0.0;
  }
  const Cplx<double> v = hessenberg_warp(hr, hi, mm, beta);
  if (lane < m) y[lane] = make_double2(v.re, v.im);
}

// ------------------------------------------------------------ delayed reorthogonalisation
// One Arnoldi step with classical Gram-Schmidt whose second pass is delayed by
// one step (low-synchronisation CGS2, Bielich, Langou, Thomas, Swirydowicz,
// Yamazaki, Boman, Parallel Computing 2022): the previous basis vector u (one
// pass done) is reorthogonalised in the same sweeps that orthogonalise the new
// vector w, so each step reads the basis twice instead of four times.
//   pass 1: A_i = <v_i, u>, B_i = <v_i, w> (i < j), d = <u, u>, c = <u, w>, <w, w>;
//   coefficients: beta = sqrt(d - sum |A_i|^2), v_j = (u - sum A_i v_i) / beta,
//                 h_j = (c - sum conj(A_i) B_i) / beta;
//   pass 2: u <- v_j, w <- w - sum_i B_i v_i - h_j v_j (and both norms).

// A load unit: two FP32 complex numbers (float4) or one FP64 complex (double2).
template <class T2> struct Unit;
template <> struct Unit<float2> { typedef float4 V; typedef float R; static constexpr int C = 2; };
template <> struct Unit<double2> { typedef double2 V; typedef double R; static constexpr int C = 1; };

__device__ __forceinline__ void cdot_acc(const float4& a, const float4& x, float& re, float& im) {
  re = fmaf(a.x, x.x, fmaf(a.y, x.y, fmaf(a.z, x.z, fmaf(a.w, x.w, re))));
  im = fmaf(a.x, x.y, fmaf(-a.y, x.x, fmaf(a.z, x.w, fmaf(-a.w, x.z, im))));
}
__device__ __forceinline__ void cdot_acc(const double2& a, const double2& x, double& re, double& im) {
  re = fma(a.x, x.x, fma(a.y, x.y, re));
  im = fma(a.x, x.y, fma(-a.y, x.x, im));
}
__device__ __forceinline__ void caxpy(float cr, float ci, const float4& a, float4& y) {
  y.x = fmaf(cr, a.x, fmaf(-ci, a.y, y.x));
  y.y = fmaf(cr, a.y, fmaf(ci, a.x, y.y));
  y.z = fmaf(cr, a.z, fmaf(-ci, a.w, y.z));
  y.w = fmaf(cr, a.w, fmaf(ci, a.z, y.w));
}
__device__ __forceinline__ void caxpy(double cr, double ci, const double2& a, double2& y) {
  y.x = fma(cr, a.x, fma(-ci, a.y, y.x));
  y.y = fma(cr, a.y, fma(ci, a.x, y.y));
}
__device__ __forceinline__ float nrm_of(const float4& y) { return y.x * y.x + y.y * y.y + y.z * y.z + y.w * y.w; }
__device__ __forceinline__ double nrm_of(const double2& y) { return y.x * y.x + y.y * y.y; }
template <class V> __device__ __forceinline__ V vzero();
template <> __device__ __forceinline__ float4 vzero<float4>() { return make_float4(0.f, 0.f, 0.f, 0.f); }
template <> __device__ __forceinline__ double2 vzero<double2>() { return make_double2(0.0, 0.0); }

constexpr int kDots2Max = 12;      // basis vectors per pass-1 launch
constexpr int kDots2Slots = 32;    // partial slots per (right-hand side, CTA)
template <class V> struct PtrsV { const V* p[16]; };

// What ends a pass 1: the sums go to A[r*ld + j0 + i], B[r*ld + j0 + i] (i < K)
// and X[r*4 + e]; the pass's last chunk (last) then forms, in one thread,
// beta, h_j and the pass-2 coefficients for the vector list
// [u, w, v_0 .. v_{j-1}]: c1 makes v_j, c2 makes the new w; hcol[0..j] =
// (B_0 .. B_{j-1}, h_j); acol[0..j] = (A_0 .. A_{j-1}, beta).  A vanishing beta
// (u in the span of the basis: a zero or invariant direction) gives zero
// coefficients.
struct Dcgs2Out {
  double2 *A, *B, *X, *c1, *c2, *hcol, *acol;
  int ld, j0, j, last;
};
__device__ inline void dcgs2_coeff(const Dcgs2Out& d, int r) {
  const int j = d.j;
  const double2* a = d.A + (size_t)r * d.ld;
  const double2* b = d.B + (size_t)r * d.ld;
  const double2* x = d.X + (size_t)r * 4;
  double2* o1 = d.c1 + (size_t)r * d.ld;
  double2* o2 = d.c2 + (size_t)r * d.ld;
  double2* hc = d.hcol + (size_t)r * d.ld;
  double2* ac = d.acol + (size_t)r * d.ld;
  double na = 0;
  for (int i = 0; i < j; ++i) na += a[i].x * a[i].x + a[i].y * a[i].y;
  const double dd = x[0].x;
  const double beta2 = dd - na;
  if (!(beta2 > 1e-24 * dd) || !(dd > 0)) {
    for (int i = 0; i < j + 2; ++i) { o1[i] = make_double2(0, 0); o2[i] = make_double2(0, 0); }
    for (int i = 0; i <= j; ++i) { hc[i] = make_double2(0, 0); ac[i] = make_double2(0, 0); }
    return;
  }
  const double beta = sqrt(beta2), ib = 1.0 / beta;
  double sr = x[1].x, si = x[1].y;                          // c - sum conj(a_i) b_i
  for (int i = 0; i < j; ++i) {
    sr -= a[i].x * b[i].x + a[i].y * b[i].y;
    si -= a[i].x * b[i].y - a[i].y * b[i].x;
  }
  const double hr = sr * ib, hi = si * ib;                  // h_j
  const double gr = hr * ib, gi = hi * ib;                  // h_j / beta
  o1[0] = make_double2(ib, 0);
  o1[1] = make_double2(0, 0);
  o2[0] = make_double2(-gr, -gi);
  o2[1] = make_double2(1, 0);
  for (int i = 0; i < j; ++i) {
    o1[2 + i] = make_double2(-a[i].x * ib, -a[i].y * ib);
    // -(b_i - (h_j / beta) a_i)
    o2[2 + i] = make_double2(-(b[i].x - (gr * a[i].x - gi * a[i].y)), -(b[i].y - (gr * a[i].y + gi * a[i].x)));
    hc[i] = b[i];
    ac[i] = a[i];
  }
  hc[j] = make_double2(hr, hi);
  ac[j] = make_double2(beta, 0);
}
template <int K, bool EXTRA>
__device__ __forceinline__ void finish_dots2(double2* partial, const Dcgs2Out& d) {
  const int r = blockIdx.y;
  if (!last_cta(partial, r)) return;
  constexpr int NS = 2 * K + (EXTRA ? 3 : 0);
  for (int q = threadIdx.x >> 5; q < NS; q += 8) {
    const double2 t = sum_slot(partial, r, kDots2Slots, q);
    if ((threadIdx.x & 31) == 0) {
      if (q < K) d.A[(size_t)r * d.ld + d.j0 + q] = t;
      else if (q < 2 * K) d.B[(size_t)r * d.ld + d.j0 + q - K] = t;
      else d.X[(size_t)r * 4 + q - 2 * K] = t;
    }
  }
  if (!d.last) return;
  __syncthreads();
  if (threadIdx.x == 0) dcgs2_coeff(d, r);
}

// slots: [i] = <v_i, u>, [K + i] = <v_i, w>, [2K + 0..2] = <u,u>, <u,w>, <w,w> (EXTRA only)
template <class T2, int K, bool EXTRA>
__global__ void __launch_bounds__(256) dots2_partial(PtrsV<typename Unit<T2>::V> v,
                                                     const typename Unit<T2>::V* __restrict__ u,
                                                     const typename Unit<T2>::V* __restrict__ w, size_t nu,
                                                     size_t stride, double2* __restrict__ partial, Dcgs2Out dout) {
  typedef typename Unit<T2>::V V;
  typedef typename Unit<T2>::R R;
  constexpr int NS = 2 * K + (EXTRA ? 3 : 0);
  const int r = blockIdx.y;
  const V* ur = u + r * stride;
  const V* wr = w + r * stride;
  R re[NS > 0 ? NS : 1], im[NS > 0 ? NS : 1];
#pragma unroll
  for (int q = 0; q < NS; ++q) re[q] = im[q] = 0;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < nu; i += (size_t)gridDim.x * blockDim.x) {
    V a[K > 0 ? K : 1];
#pragma unroll
    for (int q = 0; q < K; ++q) a[q] = __ldg(v.p[q] + r * stride + i);
    const V x = __ldg(ur + i);
    const V y = __ldg(wr + i);
#pragma unroll
    for (int q = 0; q < K; ++q) {
      cdot_acc(a[q], x, re[q], im[q]);
      cdot_acc(a[q], y, re[K + q], im[K + q]);
    }
    if (EXTRA) {
      cdot_acc(x, x, re[2 * K], im[2 * K]);
      cdot_acc(x, y, re[2 * K + 1], im[2 * K + 1]);
      cdot_acc(y, y, re[2 * K + 2], im[2 * K + 2]);
    }
  }
  __shared__ double red[8][2 * kDots2Slots];
  const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
  for (int q = 0; q < NS; ++q) {
    const R s = warp_sum(re[q]);
    const R m = warp_sum(im[q]);
    if (lane == 0) { red[wid][2 * q] = (double)s; red[wid][2 * q + 1] = (double)m; }
  }
  __syncthreads();
  if ((int)threadIdx.x < NS) {
    double s = 0, m = 0;
    for (int q = 0; q < 8; ++q) { s += red[q][2 * threadIdx.x]; m += red[q][2 * threadIdx.x + 1]; }
    partial[((size_t)r * gridDim.x + blockIdx.x) * kDots2Slots + threadIdx.x] = make_double2(s, m);
  }
  finish_dots2<K, EXTRA>(partial, dout);
}

// y1 = (acc ? y1 : 0) + sum c1_q v_q, y2 likewise; y1 and y2 may be v_0, v_1
// (every element is read before it is written, by the same thread).  With
// partial != nullptr the CTA writes its parts of ||y1||^2 and ||y2||^2.
template <class T2, int K>
__global__ void __launch_bounds__(256) axpy2_kernel(PtrsV<typename Unit<T2>::V> v, const double2* __restrict__ c1,
                                                    const double2* __restrict__ c2, int ldc, int j0,
                                                    typename Unit<T2>::V* y1, typename Unit<T2>::V* y2, size_t nu,
                                                    size_t stride, int acc, double2* __restrict__ partial,
                                                    DotOut dout) {
  typedef typename Unit<T2>::V V;
  typedef typename Unit<T2>::R R;
  __shared__ R cf[4][16];
  const int r = blockIdx.y;
  if (threadIdx.x < K) {
    const double2 p = c1[(size_t)r * ldc + j0 + threadIdx.x], q = c2[(size_t)r * ldc + j0 + threadIdx.x];
    cf[0][threadIdx.x] = (R)p.x;
    cf[1][threadIdx.x] = (R)p.y;
    cf[2][threadIdx.x] = (R)q.x;
    cf[3][threadIdx.x] = (R)q.y;
  }
  __syncthreads();
  V* o1 = y1 + r * stride;
  V* o2 = y2 + r * stride;
  R n1 = 0, n2 = 0;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < nu; i += (size_t)gridDim.x * blockDim.x) {
    V a[K];
#pragma unroll
    for (int q = 0; q < K; ++q) a[q] = v.p[q][r * stride + i];
    V s1 = acc ? o1[i] : vzero<V>();
    V s2 = acc ? o2[i] : vzero<V>();
#pragma unroll
    for (int q = 0; q < K; ++q) {
      caxpy(cf[0][q], cf[1][q], a[q], s1);
      caxpy(cf[2][q], cf[3][q], a[q], s2);
    }
    o1[i] = s1;
    o2[i] = s2;
    n1 += nrm_of(s1);
    n2 += nrm_of(s2);
  }
  if (partial) {
    __shared__ double red[8][2];
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const R t1 = warp_sum(n1), t2 = warp_sum(n2);
    if (lane == 0) { red[wid][0] = (double)t1; red[wid][1] = (double)t2; }
    __syncthreads();
    if (threadIdx.x < 2) {
      double sum = 0;
      for (int q = 0; q < 8; ++q) sum += red[q][threadIdx.x];
      partial[((size_t)r * gridDim.x + blockIdx.x) * kChunk + threadIdx.x] = make_double2(sum, 0.0);
    }
    finish_dots<2>(partial, dout);
  }
}

template <class T2>
static int dcgs2_step_t(const BVec& b, const void* const* v, int j, void* u, void* w, const DcgsWork& ws,
                        cudaStream_t s) {
  typedef typename Unit<T2>::V V;
  constexpr int C = Unit<T2>::C;
  const size_t nu = b.n / C, stride = b.vstride / C;
  const int R = b.R;
  // pass 1: dots of u and w with the basis (chunks of kDots2Max) and with each other
  const int ncta1 = reduce_ctas(nu, R, kDots2Slots);
  const dim3 g1(ncta1, R);
  int j0 = 0;
  do {
    const int kk = std::min(kDots2Max, j - j0);
    const bool extra = (j0 == 0);
    const Dcgs2Out d{ws.A, ws.B, ws.X, ws.c1, ws.c2, ws.hcol, ws.acol, ws.ld, j0, j, j0 + kk >= j};
    PtrsV<V> p;
    for (int q = 0; q < 16; ++q) p.p[q] = j > 0 ? (const V*)v[std::max(0, std::min(j0 + q, j - 1))] : (const V*)u;
#define SAPMG_D2(K)                                                                                          \
  case K:                                                                                                    \
    if (extra) { dots2_partial<T2, K, true><<<g1, 256, 0, s>>>(p, (const V*)u, (const V*)w, nu, stride, ws.partial, d); } \
    else { dots2_partial<T2, K, false><<<g1, 256, 0, s>>>(p, (const V*)u, (const V*)w, nu, stride, ws.partial, d); } \
    count_launches(1);                                                                                       \
    break;
    switch (kk) {
      SAPMG_D2(0) SAPMG_D2(1) SAPMG_D2(2) SAPMG_D2(3) SAPMG_D2(4) SAPMG_D2(5) SAPMG_D2(6)
      SAPMG_D2(7) SAPMG_D2(8) SAPMG_D2(9) SAPMG_D2(10) SAPMG_D2(11) SAPMG_D2(12)
      default: return MG_ERR_ARG;
    }
#undef SAPMG_D2
    j0 += kk;
  } while (j0 < j);
  // pass 2 over the list [u, w, v_0 .. v_{j-1}] in chunks of 16
  const dim3 g2(reduce_ctas(nu, R), R);
  const DotOut dn{ws.nrm, nullptr, ws.ld, 0};
  const int total = j + 2;
  for (int q0 = 0; q0 < total; q0 += 16) {
    const int kk = std::min(16, total - q0);
    const bool last = q0 + 16 >= total;
    PtrsV<V> p;
    for (int q = 0; q < 16; ++q) {
      const int t = q0 + std::min(q, kk - 1);
      p.p[q] = (const V*)(t == 0 ? u : (t == 1 ? w : v[t - 2]));
    }
    double2* part = last ? ws.partial : nullptr;
    const int acc = q0 > 0;
#define SAPMG_A2(K)                                                                                            \
  case K:                                                                                                      \
    axpy2_kernel<T2, K><<<g2, 256, 0, s>>>(p, ws.c1, ws.c2, ws.ld, q0, (V*)u, (V*)w, nu, stride, acc, part, dn); \
    count_launches(1);                                                                                         \
    break;
    switch (kk) {
      SAPMG_A2(1) SAPMG_A2(2) SAPMG_A2(3) SAPMG_A2(4) SAPMG_A2(5) SAPMG_A2(6) SAPMG_A2(7) SAPMG_A2(8)
      SAPMG_A2(9) SAPMG_A2(10) SAPMG_A2(11) SAPMG_A2(12) SAPMG_A2(13) SAPMG_A2(14) SAPMG_A2(15) SAPMG_A2(16)
      default: return MG_ERR_ARG;
    }
#undef SAPMG_A2
  }
  SAPMG_CUDA_TRY(cudaGetLastError());
  return MG_OK;
}

int blas_dcgs2_step(int type, const BVec& b, const void* const* v, int j, void* u, void* w, const DcgsWork& ws,
                    cudaStream_t s) {
  if (b.R <= 0) return MG_OK;
  if (j < 0 || j + 2 > ws.ld || b.R > 32) return MG_ERR_ARG;
  // pass 1 reads the j basis vectors, u and w; pass 2 reads them again and writes u and w
  count_bytes((double)(2 * j + 6) * b.n * b.R * (type == P64 ? 16 : 8));
  if (type == P32) {
    bool al = (b.n % 2 == 0) && (b.vstride == b.n) && ((reinterpret_cast<uintptr_t>(u) & 15) == 0) &&
              ((reinterpret_cast<uintptr_t>(w) & 15) == 0);
    for (int q = 0; q < j; ++q) al = al && ((reinterpret_cast<uintptr_t>(v[q]) & 15) == 0);
    if (!al) return MG_ERR_ARG;
    return dcgs2_step_t<float2>(b, v, j, u, w, ws, s);
  }
  if (type == P64) {
    if (b.vstride != b.n) return MG_ERR_ARG;
    return dcgs2_step_t<double2>(b, v, j, u, w, ws, s);
  }
  return MG_ERR_ARG;
}

// ------------------------------------------------------------ FP16 basis
// The finished basis vectors of the mixed form's outer Arnoldi may be kept in
// FP16, scaled by kBasisScale = 2^10 (a unit vector's entries stay below 1, so
// the scaled values stay in FP16's normal range and the scaling is exact).
// Eight bytes = two complex numbers per load unit.

__device__ __forceinline__ float4 h4_to_f4(uint2 u) {
  const float2 a = __half22float2(*reinterpret_cast<const __half2*>(&u.x));
  const float2 b = __half22float2(*reinterpret_cast<const __half2*>(&u.y));
  constexpr float is = 1.f / kBasisScale;
  return make_float4(a.x * is, a.y * is, b.x * is, b.y * is);
}

__device__ __forceinline__ uint2 f4_to_h4(float4 v) {
  const __half2 a = __floats2half2_rn(v.x * kBasisScale, v.y * kBasisScale);
  const __half2 b = __floats2half2_rn(v.z * kBasisScale, v.w * kBasisScale);
  uint2 u;
  u.x = *reinterpret_cast<const unsigned int*>(&a);
  u.y = *reinterpret_cast<const unsigned int*>(&b);
  return u;
}

// pass 1 with an FP16 basis: slots as dots2_partial
// From kRingFrom basis vectors on each thread copies its next element of every vector
// to shared memory while it works on the current one: the compiler spreads that
// many loads between the products, which leaves too few bytes in flight (8 vectors,
// 12 fields of 7.96 M: 1401 us by plain loads, 676 us so, 677 us at the measured HBM
// rate; 6 vectors by plain loads 581 us, 564 us at that rate).
constexpr int kRingFrom = 7;
constexpr size_t dots2h_smem(int K) { return K >= kRingFrom ? (size_t)2 * 256 * (8 * K + 32) : 0; }
__device__ __forceinline__ void cp_async(void* dst, const uint2* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async(void* dst, const float4* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
template <int K, bool EXTRA>
__global__ void __launch_bounds__(256) dots2h_partial(PtrsV<uint2> v, const float4* __restrict__ u,
                                                      const float4* __restrict__ w, size_t nu, size_t stride,
                                                      double2* __restrict__ partial, Dcgs2Out dout) {
  constexpr bool kRing = K >= kRingFrom;
  extern __shared__ __align__(16) float4 ring[];       // per stage [2][256] float4, [K][256] uint2
  constexpr int kStage4 = 256 * (2 + K / 2) + (K % 2) * 128;
  constexpr int NS = 2 * K + (EXTRA ? 3 : 0);
  const int r = blockIdx.y;
  const float4* ur = u + r * stride;
  const float4* wr = w + r * stride;
  float re[NS > 0 ? NS : 1], im[NS > 0 ? NS : 1];
#pragma unroll
  for (int q = 0; q < NS; ++q) re[q] = im[q] = 0.f;
  const size_t i0 = (size_t)blockIdx.x * blockDim.x + threadIdx.x, step = (size_t)gridDim.x * blockDim.x;
  auto fetch = [&](size_t i, int st) {                 // a thread reads back its own copies only
    if (i < nu) {
      float4* d = ring + st * kStage4 + threadIdx.x;
      uint2* e = reinterpret_cast<uint2*>(ring + st * kStage4 + 512) + threadIdx.x;
      cp_async(d, ur + i);
      cp_async(d + 256, wr + i);
#pragma unroll
      for (int q = 0; q < K; ++q) cp_async(e + q * 256, v.p[q] + r * stride + i);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  if (kRing) fetch(i0, 0);
  int st = 0;
  for (size_t i = i0; i < nu; i += step, st ^= 1) {
    uint2 a[K > 0 ? K : 1];
    float4 x, y;
    if (kRing) {
      fetch(i + step, st ^ 1);
      asm volatile("cp.async.wait_group 1;" ::: "memory");
      const float4* d = ring + st * kStage4 + threadIdx.x;
      const uint2* e = reinterpret_cast<const uint2*>(ring + st * kStage4 + 512) + threadIdx.x;
      x = d[0];
      y = d[256];
#pragma unroll
      for (int q = 0; q < K; ++q) a[q] = e[q * 256];
    } else {
#pragma unroll
      for (int q = 0; q < K; ++q) a[q] = __ldg(v.p[q] + r * stride + i);
      x = __ldg(ur + i);
      y = __ldg(wr + i);
    }
#pragma unroll
    for (int q = 0; q < K; ++q) {
      const float4 av = h4_to_f4(a[q]);
      cdot_acc(av, x, re[q], im[q]);
      cdot_acc(av, y, re[K + q], im[K + q]);
    }
    if (EXTRA) {
      cdot_acc(x, x, re[2 * K], im[2 * K]);
      cdot_acc(x, y, re[2 * K + 1], im[2 * K + 1]);
      cdot_acc(y, y, re[2 * K + 2], im[2 * K + 2]);
    }
  }
  __shared__ double red[8][2 * kDots2Slots];
  const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
  for (int q = 0; q < NS; ++q) {
    const float a = warp_sum(re[q]);
    const float b = warp_sum(im[q]);
    if (lane == 0) { red[wid][2 * q] = (double)a; red[wid][2 * q + 1] = (double)b; }
  }
  __syncthreads();
  if ((int)threadIdx.x < NS) {
    double a = 0, b = 0;
    for (int q = 0; q < 8; ++q) { a += red[q][2 * threadIdx.x]; b += red[q][2 * threadIdx.x + 1]; }
    partial[((size_t)r * gridDim.x + blockIdx.x) * kDots2Slots + threadIdx.x] = make_double2(a, b);
  }
  finish_dots2<K, EXTRA>(partial, dout);
}

// pass 2 with an FP16 basis.  Coefficient q of c1/c2 belongs to [u, w, v_0, ...].
// first: y1 = c1_u u + c1_w w + sum, y2 likewise; otherwise y1 += sum (y1 kept
// in u), y2 += sum (in w).  vout != nullptr (last chunk): v_j = y1 is
// written to the FP16 basis and to u only if keep_u; partial: ||y1||^2, ||y2||^2.
template <int K>
__global__ void __launch_bounds__(256) axpy2h_kernel(PtrsV<uint2> v, const double2* __restrict__ c1,
                                                     const double2* __restrict__ c2, int ldc, int q0, float4* u,
                                                     float4* w, uint2* __restrict__ vout, size_t nu, size_t stride,
                                                     int first, double2* __restrict__ partial, DotOut dout) {
  __shared__ float cf[4][18];
  const int r = blockIdx.y;
  if ((int)threadIdx.x < K + 2) {
    const int q = threadIdx.x;                       // 0, 1: u, w (first chunk); 2..: basis entries
    const int ci = q < 2 ? q : 2 + q0 + (q - 2);
    const double2 p = c1[(size_t)r * ldc + ci], t = c2[(size_t)r * ldc + ci];
    cf[0][q] = (float)p.x;
    cf[1][q] = (float)p.y;
    cf[2][q] = (float)t.x;
    cf[3][q] = (float)t.y;
  }
  __syncthreads();
  float4* o1 = u + r * stride;
  float4* o2 = w + r * stride;
  uint2* ov = vout ? vout + r * stride : nullptr;
  float n1 = 0.f, n2 = 0.f;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < nu; i += (size_t)gridDim.x * blockDim.x) {
    uint2 a[K > 0 ? K : 1];
#pragma unroll
    for (int q = 0; q < K; ++q) a[q] = __ldg(v.p[q] + r * stride + i);
    const float4 uu = o1[i], ww = o2[i];
    float4 s1, s2;
    if (first) {
      s1 = vzero<float4>();
      s2 = vzero<float4>();
      caxpy(cf[0][0], cf[1][0], uu, s1);
      caxpy(cf[0][1], cf[1][1], ww, s1);
      caxpy(cf[2][0], cf[3][0], uu, s2);
      caxpy(cf[2][1], cf[3][1], ww, s2);
    } else {
      s1 = uu;
      s2 = ww;
    }
#pragma unroll
    for (int q = 0; q < K; ++q) {
      const float4 av = h4_to_f4(a[q]);
      caxpy(cf[0][2 + q], cf[1][2 + q], av, s1);
      caxpy(cf[2][2 + q], cf[3][2 + q], av, s2);
    }
    if (!ov) o1[i] = s1;
    o2[i] = s2;
    if (ov) ov[i] = f4_to_h4(s1);
    n1 += nrm_of(s1);
    n2 += nrm_of(s2);
  }
  if (partial) {
    __shared__ double red[8][2];
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const float t1 = warp_sum(n1), t2 = warp_sum(n2);
    if (lane == 0) { red[wid][0] = (double)t1; red[wid][1] = (double)t2; }
    __syncthreads();
    if (threadIdx.x < 2) {
      double sum = 0;
      for (int q = 0; q < 8; ++q) sum += red[q][threadIdx.x];
      partial[((size_t)r * gridDim.x + blockIdx.x) * kChunk + threadIdx.x] = make_double2(sum, 0.0);
    }
    finish_dots<2>(partial, dout);
  }
}

template <int K, bool EXTRA>
static cudaError_t dots2h_run(dim3 grid, const PtrsV<uint2>& p, const float4* u, const float4* w, size_t nu,
                              size_t stride, double2* partial, const Dcgs2Out& d, cudaStream_t s) {
  if (dots2h_smem(K) > 0) {
    static bool attr = false;
    if (!attr) {
      const cudaError_t e = cudaFuncSetAttribute(dots2h_partial<K, EXTRA>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                 (int)dots2h_smem(K));
      if (e != cudaSuccess) return e;
      attr = true;
    }
  }
  dots2h_partial<K, EXTRA><<<grid, 256, dots2h_smem(K), s>>>(p, u, w, nu, stride, partial, d);
  count_launches(1);
  return cudaGetLastError();
}

int blas_dcgs2_step_h(const BVec& b, const void* const* vh, int j, void* u, void* w, void* vout, const DcgsWork& ws,
                      cudaStream_t s) {
  if (b.R <= 0) return MG_OK;
  if (j < 0 || j + 2 > ws.ld || b.R > 32 || b.n % 2 != 0 || b.vstride != b.n) return MG_ERR_ARG;
  bool al = ((reinterpret_cast<uintptr_t>(u) & 15) == 0) && ((reinterpret_cast<uintptr_t>(w) & 15) == 0) &&
            ((reinterpret_cast<uintptr_t>(vout) & 7) == 0);
  for (int q = 0; q < j; ++q) al = al && ((reinterpret_cast<uintptr_t>(vh[q]) & 7) == 0);
  if (!al) return MG_ERR_ARG;
  // pass 1: j FP16 basis vectors + u, w; pass 2: the same + w written + v_j in FP16
  // (u is written back only between chunks, when j > 16)
  count_bytes(((double)2 * j * 4 + 5 * 8 + 4) * b.n * b.R);
  const size_t nu = b.n / 2, stride = b.vstride / 2;
  const int R = b.R;
  const int ncta1 = reduce_ctas(nu, R, kDots2Slots);
  const dim3 g1(ncta1, R);
  const float4* uf = (const float4*)u;
  const float4* wf = (const float4*)w;
  int j0 = 0;
  do {
    const int kk = std::min(kDots2Max, j - j0);
    const bool extra = (j0 == 0);
    const Dcgs2Out d{ws.A, ws.B, ws.X, ws.c1, ws.c2, ws.hcol, ws.acol, ws.ld, j0, j, j0 + kk >= j};
    PtrsV<uint2> p;
    for (int q = 0; q < 16; ++q) p.p[q] = j > 0 ? (const uint2*)vh[std::max(0, std::min(j0 + q, j - 1))] : (const uint2*)vout;
#define SAPMG_D2H(K)                                                                                              \
  case K:                                                                                                         \
    if (extra) rc = dots2h_run<K, true>(g1, p, uf, wf, nu, stride, ws.partial, d, s);                              \
    else rc = dots2h_run<K, false>(g1, p, uf, wf, nu, stride, ws.partial, d, s);                                   \
    break;
    cudaError_t rc = cudaSuccess;
    switch (kk) {
      SAPMG_D2H(0) SAPMG_D2H(1) SAPMG_D2H(2) SAPMG_D2H(3) SAPMG_D2H(4) SAPMG_D2H(5) SAPMG_D2H(6)
      SAPMG_D2H(7) SAPMG_D2H(8) SAPMG_D2H(9) SAPMG_D2H(10) SAPMG_D2H(11) SAPMG_D2H(12)
      default: return MG_ERR_ARG;
    }
#undef SAPMG_D2H
    SAPMG_CUDA_TRY(rc);
    j0 += kk;
  } while (j0 < j);
  const dim3 g2(reduce_ctas(nu, R), R);
  const DotOut dn{ws.nrm, nullptr, ws.ld, 0};
  int q0 = 0;
  bool first = true;
  do {
    const int kk = std::min(16, j - q0);
    const bool last = q0 + kk >= j;
    PtrsV<uint2> p;
    for (int q = 0; q < 16; ++q) p.p[q] = j > 0 ? (const uint2*)vh[std::max(0, std::min(q0 + q, j - 1))] : (const uint2*)vout;
    double2* part = last ? ws.partial : nullptr;
    uint2* vo = last ? (uint2*)vout : nullptr;
#define SAPMG_A2H(K)                                                                                                \
  case K:                                                                                                           \
    axpy2h_kernel<K><<<g2, 256, 0, s>>>(p, ws.c1, ws.c2, ws.ld, q0, (float4*)u, (float4*)w, vo, nu, stride, first, \
                                        part, dn);                                                                  \
    count_launches(1);                                                                                              \
    break;
    switch (kk) {
      SAPMG_A2H(0) SAPMG_A2H(1) SAPMG_A2H(2) SAPMG_A2H(3) SAPMG_A2H(4) SAPMG_A2H(5) SAPMG_A2H(6) SAPMG_A2H(7)
      SAPMG_A2H(8) SAPMG_A2H(9) SAPMG_A2H(10) SAPMG_A2H(11) SAPMG_A2H(12) SAPMG_A2H(13) SAPMG_A2H(14)
      SAPMG_A2H(15) SAPMG_A2H(16)
      default: return MG_ERR_ARG;
    }
#undef SAPMG_A2H
    q0 += kk;
    first = false;
  } while (q0 < j);
  SAPMG_CUDA_TRY(cudaGetLastError());
  return MG_OK;
}

__global__ void normalize_h_kernel(const float4* __restrict__ x, uint2* __restrict__ out,
                                   const double2* __restrict__ nrm2, int ldn, double2* __restrict__ store, int lds,
                                   size_t nu, size_t stride) {
  const int r = blockIdx.y;
  const double nn = sqrt(fmax(nrm2[(size_t)r * ldn].x, 0.0));
  const float inv = nn > 0.0 ? (float)(1.0 / nn) : 0.f;
  if (blockIdx.x == 0 && threadIdx.x == 0 && store) store[(size_t)r * lds] = make_double2(nn, 0.0);
  const float4* xr = x + r * stride;
  uint2* o = out + r * stride;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < nu; i += (size_t)gridDim.x * blockDim.x) {
    float4 u = xr[i];
    u.x *= inv;
    u.y *= inv;
    u.z *= inv;
    u.w *= inv;
    o[i] = f4_to_h4(u);
  }
}

int blas_normalize_h(const BVec& b, const void* x, void* out, const double2* nrm2, int ldn, double2* store, int lds,
                     cudaStream_t s) {
  if (b.n % 2 != 0 || b.wstride != b.n) return MG_ERR_ARG;
  count_bytes(12.0 * b.n * b.R);
  const size_t nu = b.n / 2;
  const dim3 g = stream_grid(nu, b.R);
  normalize_h_kernel<<<g, 256, 0, s>>>((const float4*)x, (uint2*)out, nrm2, ldn, store, lds, nu, b.wstride / 2);
  count_launches(1);
  SAPMG_CUDA_TRY(cudaGetLastError());
  return MG_OK;
}

// ------------------------------------------------------------ one Arnoldi step of the coarse levels
// Two kernels a step of fixed-step (flexible) GMRES, w = A v_j given:
//   dots    <v_i, w> (i <= j) and <w, w> in one pass; the last CTA of a
//           right-hand side turns them into column j of H, the update's
//           coefficients and beta^2 = <w, w> - sum |<v_i, w>|^2 / |v_i|^2;
//   update  x = w - sum (<v_i, w> / |v_i|^2) v_i, v_{j+1} = x / beta, and ||x||
//           itself, which is H_{j+1,j}.
// beta (formed before x exists) only has to be near ||x||: v_{j+1} has the norm
// s_{j+1} = ||x|| / beta, which is kept, and H and y are those of the unit
// vectors v_i / s_i, so a beta that cancellation or FP32 has made inexact costs no
// accuracy (the FP32 value that divided x is the one kept); a floor under it
// (kFloor <w, w>) bounds s_{j+1}.  Against a norm pass
// before a separate normalisation this reads and writes w once less and takes
// two launches a step instead of five.  Bound by L2/HBM bandwidth for 12 right-hand
// sides, by latency for one.
struct HalfBasis {          // FP16 basis scaled by kBasisScale, FP32 w
  typedef uint2 V;
  typedef float4 W;
  typedef float R;
  static constexpr int C = 2, CH = 32;
  // 2^10 |v_{j+1}| has to stay below 65504 where the basis has lost its
  // orthogonality and beta^2 comes out too small: beta >= ||w|| / 8
  static constexpr double kFloor = 1.0 / 64;
  static __device__ __forceinline__ W get(V a) { return h4_to_f4(a); }
  static __device__ __forceinline__ V put(W x, R f) { return f4_to_h4(make_float4(x.x * f, x.y * f, x.z * f, x.w * f)); }
};
struct SingleBasis {
  typedef float4 V;
  typedef float4 W;
  typedef float R;
  static constexpr int C = 2, CH = 32;
  static constexpr double kFloor = 1e-6;
  static __device__ __forceinline__ W get(V a) { return a; }
  static __device__ __forceinline__ V put(W x, R f) { return make_float4(x.x * f, x.y * f, x.z * f, x.w * f); }
};
struct DoubleBasis {
  typedef double2 V;
  typedef double2 W;
  typedef double R;
  static constexpr int C = 1, CH = 16;
  static constexpr double kFloor = 1e-14;
  static __device__ __forceinline__ W get(V a) { return a; }
  static __device__ __forceinline__ V put(W x, R f) { return make_double2(x.x * f, x.y * f); }
};
template <class V> struct PtrsK { const V* p[32]; };

// Scalars of a step (per right-hand side, stride ldr): H (33 x 33 column-major)
// takes the raw dots; t[i] a coefficient of the update (Cplx<R>; FP64: the raw dots
// of earlier chunks before), t[40] 1/beta, t[64 + i] = (||x||^2, 1/beta) of basis
// vector i >= 1 and, as Scale<R> from t[100] on, 1 / s_i^2.
struct ArnoldiOut {
  double2 *H, *t;
  int ldr, j, i0, last;    // the step, the chunk's first vector, the chunk that ends the pass
};
template <class R> struct AccC { Acc<R> re, im; };      // sixteen bytes: a slot of the partial sums
static_assert(sizeof(AccC<float>) == 16 && sizeof(AccC<double>) == 16, "a slot holds one complex sum");

// The calling warp's sum of a slot over the CTAs of right-hand side r.
template <class R>
__device__ __forceinline__ AccC<R> sum_slot_acc(const double2* partial, int r, int slots, int j) {
  AccC<R> a;
  a.re = a.im = Acc<R>::of((R)0);
#pragma unroll 4
  for (int c = threadIdx.x & 31; c < (int)gridDim.x; c += 32) {
    const double2 q = __ldcg(partial + ((size_t)r * gridDim.x + c) * slots + j);
    const AccC<R> v = *reinterpret_cast<const AccC<R>*>(&q);
    a.re.add(v.re);
    a.im.add(v.im);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    a.re.add(a.re.from(o));
    a.im.add(a.im.from(o));
  }
  return a;
}

__device__ __forceinline__ float inv_sqrt(float x) { return rsqrtf(x); }
__device__ __forceinline__ double inv_sqrt(double x) { return rsqrt(x); }

// v[0..N) summed over the warp, N a power of two up to 32: halving the values a
// lane holds with every exchange, N - 1 + (5 - log2 N) shuffles instead of 5 N.
// Lane l gets value l / (32 / N).
template <int N, class R>
__device__ __forceinline__ R warp_sums(R (&v)[N]) {
  const int lane = threadIdx.x & 31;
  int mask = 16;
#pragma unroll
  for (int n = N / 2; n >= 1; n /= 2, mask /= 2) {
    const bool up = (lane & mask) != 0;
#pragma unroll
    for (int i = 0; i < n; ++i) {
      const R send = up ? v[i] : v[i + n];
      const R keep = up ? v[i + n] : v[i];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, send, mask);
    }
  }
  for (; mask >= 1; mask /= 2) v[0] += __shfl_xor_sync(0xffffffffu, v[0], mask);
  return v[0];
}

template <class B, int KM>
__global__ void __launch_bounds__(256) arnoldi_dots_kernel(PtrsK<typename B::V> v, int k,
                                                           const typename B::W* __restrict__ w, size_t nu,
                                                           size_t stride, double2* __restrict__ partial,
                                                           ArnoldiOut o) {
  typedef typename B::R R;
  typedef typename B::V V;
  const int r = blockIdx.y, lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const typename B::W* wr = w + r * stride;
  // Sixteen vectors a sweep: with all 32 vectors' sums in registers the compiler spreads
  // the loads between the products, and a step on 20 vectors (12 fields of 103680) took
  // 107 us, against 23 us of one on 16 and 44 us so; w is read again, from L2 mostly.
  constexpr int KS = KM < 16 ? KM : 16, NV = 2 * KS;
  pdl_begin();
  __shared__ R red[8][2 * KM + 1];
  R ww = 0;
#pragma unroll
  for (int h = 0; h < KM; h += KS) {
    R acc[KS][2];
#pragma unroll
    for (int q = 0; q < KS; ++q) acc[q][0] = acc[q][1] = 0;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < nu; i += (size_t)gridDim.x * blockDim.x) {
      const typename B::W x = __ldcg(wr + i);
#pragma unroll
      for (int g = 0; g < KS; g += 8) {                  // up to eight loads in flight
        constexpr int G = KS < 8 ? KS : 8;
        V a[G];
#pragma unroll
        for (int q = 0; q < G; ++q)
          if (h + g + q < k) a[q] = __ldcg(v.p[h + g + q] + r * stride + i);
#pragma unroll
        for (int q = 0; q < G; ++q)
          if (h + g + q < k) cdot_acc(B::get(a[q]), x, acc[g + q][0], acc[g + q][1]);
      }
      if (h == 0) ww += nrm_of(x);
    }
    R u[NV];
#pragma unroll
    for (int q = 0; q < NV; ++q) u[q] = acc[q >> 1][q & 1];
    const R t = warp_sums<NV>(u);
    if (lane % (32 / NV) == 0) red[wid][2 * h + lane / (32 / NV)] = t;
  }
  ww = warp_sum(ww);
  if (lane == 0) red[wid][2 * KM] = ww;
  __syncthreads();
  Acc<R>* part = reinterpret_cast<Acc<R>*>(partial + ((size_t)r * gridDim.x + blockIdx.x) * (KM + 1));
  if ((int)threadIdx.x <= 2 * KM) {
    Acc<R> t = Acc<R>::of(red[0][threadIdx.x]);
#pragma unroll
    for (int q = 1; q < 8; ++q) t.add(Acc<R>::of(red[q][threadIdx.x]));
    part[threadIdx.x] = t;
    if ((int)threadIdx.x == 2 * KM) part[2 * KM + 1] = Acc<R>::of((R)0);
  }
  if (!last_cta(partial, r)) return;
  __shared__ AccC<R> raw[KM + 1];
  for (int q = wid; q <= KM; q += 8) {
    if (q < k || q == KM) {
      const AccC<R> t = sum_slot_acc<R>(partial, r, KM + 1, q);
      if (lane == 0) raw[q] = t;
    }
  }
  __syncthreads();
  if (wid > 0) return;
  double2* t = o.t + (size_t)r * o.ldr;
  AccC<R>* tr = reinterpret_cast<AccC<R>*>(t);
  if (!o.last) {
    if (lane < k) tr[o.i0 + lane] = raw[lane];
    return;
  }
  // lane = basis vector i <= j
  const bool on = lane <= o.j;
  AccC<R> d;
  d.re = d.im = Acc<R>::of((R)0);
  if (on && lane < o.i0) {
    const double2 q = __ldcg(t + lane);
    d = *reinterpret_cast<const AccC<R>*>(&q);
  } else if (on) {
    d = raw[lane - o.i0];
  }
  Scale<R> is2 = Scale<R>::one();
  if (on && lane > 0) {
    const double q = __ldcg(reinterpret_cast<const double*>(t + 100) + lane);
    is2 = *reinterpret_cast<const Scale<R>*>(&q);
  }
  const R cr = is2.times(d.re), ci = is2.times(d.im);
  const R e = warp_sum(d.re.value() * cr + d.im.value() * ci);
  if (on) {
    reinterpret_cast<AccC<R>*>(o.H + (size_t)r * o.ldr)[lane + 33 * o.j] = d;
    reinterpret_cast<Cplx<R>*>(t + lane)[0] = cmk(cr, ci);
  }
  if (lane == 0) {
    const R n2 = raw[KM].re.value(), b2 = max(n2 - e, (R)B::kFloor * n2);
    reinterpret_cast<R*>(t + 40)[0] = b2 > (R)0 ? inv_sqrt(b2) : (R)0;
  }
}

// x = w - sum t_i v_i over the chunk's vectors (written back to w unless the chunk
// ends the pass); last: vnext = x / beta if vnext != nullptr, ||x|| and s_{j+1}.
template <class B, int KM>
__global__ void __launch_bounds__(256) arnoldi_update_kernel(PtrsK<typename B::V> v, int k, typename B::W* w,
                                                             typename B::V* __restrict__ vnext, size_t nu,
                                                             size_t stride, double2* __restrict__ partial,
                                                             ArnoldiOut o) {
  typedef typename B::R R;
  typedef typename B::V V;
  __shared__ R cf[2][KM];
  __shared__ R red[8];
  const int r = blockIdx.y, lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  double2* t = o.t + (size_t)r * o.ldr;
  pdl_begin();
  if ((int)threadIdx.x < k) {
    const double2 q = __ldcg(t + o.i0 + threadIdx.x);
    const Cplx<R> c = reinterpret_cast<const Cplx<R>*>(&q)[0];
    cf[0][threadIdx.x] = -c.re;
    cf[1][threadIdx.x] = -c.im;
  }
  const R invb = __ldcg(reinterpret_cast<const R*>(t + 40));
  __syncthreads();
  typename B::W* wr = w + r * stride;
  R nn = 0;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < nu; i += (size_t)gridDim.x * blockDim.x) {
    typename B::W x = __ldcg(wr + i);
#pragma unroll
    for (int g = 0; g < KM; g += 8) {
      constexpr int G = KM < 8 ? KM : 8;
      V a[G];
#pragma unroll
      for (int q = 0; q < G; ++q)
        if (g + q < k) a[q] = __ldcg(v.p[g + q] + r * stride + i);
#pragma unroll
      for (int q = 0; q < G; ++q)
        if (g + q < k) caxpy(cf[0][g + q], cf[1][g + q], B::get(a[q]), x);
    }
    if (!o.last) wr[i] = x;
    else if (vnext) vnext[r * stride + i] = B::put(x, invb);
    nn += nrm_of(x);
  }
  if (!o.last) return;
  nn = warp_sum(nn);
  if (lane == 0) red[wid] = nn;
  __syncthreads();
  if (threadIdx.x == 0) {
    AccC<R> sum;
    sum.re = Acc<R>::of(red[0]);
    sum.im = Acc<R>::of((R)0);
#pragma unroll
    for (int q = 1; q < 8; ++q) sum.re.add(Acc<R>::of(red[q]));
    reinterpret_cast<AccC<R>*>(partial)[(size_t)r * gridDim.x + blockIdx.x] = sum;
  }
  if (!last_cta(partial, r)) return;
  if (wid > 0) return;
  const Acc<R> sum = sum_slot_acc<R>(partial, r, 1, 0).re;
  if (lane == 0) {
    reinterpret_cast<Scale<R>*>(t + 100)[o.j + 1] = Scale<R>::of(sum, invb);
    t[64 + o.j + 1] = make_double2(fmax(sum.exact(), 0.0), (double)invb);
  }
}

// out = sum y_i v_i (acc: added to what out holds)
template <class B, int KM>
__global__ void __launch_bounds__(256) combine_kernel(PtrsK<typename B::V> v, int k, const double2* __restrict__ y,
                                                      int ldy, typename B::W* __restrict__ out, size_t nu,
                                                      size_t stride, int acc) {
  typedef typename B::R R;
  typedef typename B::V V;
  __shared__ R cf[2][KM];
  const int r = blockIdx.y;
  pdl_begin();
  if ((int)threadIdx.x < k) {
    const double2 c = __ldcg(y + (size_t)r * ldy + threadIdx.x);
    cf[0][threadIdx.x] = (R)c.x;
    cf[1][threadIdx.x] = (R)c.y;
  }
  __syncthreads();
  typename B::W* o = out + r * stride;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < nu; i += (size_t)gridDim.x * blockDim.x) {
    typename B::W x = acc ? __ldcg(o + i) : vzero<typename B::W>();
#pragma unroll
    for (int g = 0; g < KM; g += 8) {
      constexpr int G = KM < 8 ? KM : 8;
      V a[G];
#pragma unroll
      for (int q = 0; q < G; ++q)
        if (g + q < k) a[q] = __ldcg(v.p[g + q] + r * stride + i);
#pragma unroll
      for (int q = 0; q < G; ++q)
        if (g + q < k) caxpy(cf[0][g + q], cf[1][g + q], B::get(a[q]), x);
    }
    o[i] = x;
  }
}

// Vectors per kernel: the smallest of 4, 8, 16, 32 (FP64: 16, longer lists in
// chunks of 16) that holds the list.
#define SAPMG_KM(KERNEL, kk, ...)                                                                          \
  SAPMG_CUDA_TRY((kk) <= 4    ? cudaLaunchKernelEx(&l.cfg, KERNEL<B, 4>, __VA_ARGS__)                      \
                 : (kk) <= 8  ? cudaLaunchKernelEx(&l.cfg, KERNEL<B, 8>, __VA_ARGS__)                      \
                 : (kk) <= 16 ? cudaLaunchKernelEx(&l.cfg, KERNEL<B, 16>, __VA_ARGS__)                     \
                              : cudaLaunchKernelEx(&l.cfg, KERNEL<B, B::CH>, __VA_ARGS__));                \
  count_launches(1);

template <class B>
static PtrsK<typename B::V> ptrs_k(const void* const* v, int i0, int kk) {
  PtrsK<typename B::V> p;
  for (int q = 0; q < 32; ++q) p.p[q] = (const typename B::V*)v[i0 + std::min(q, kk - 1)];
  return p;
}

template <class B>
static int arnoldi_step_t(const BVec& b, const void* const* v, int j, void* w, void* vnext, const ArnoldiWork& a,
                          cudaStream_t s) {
  typedef typename B::V V;
  typedef typename B::W W;
  const size_t nu = b.n / B::C, stride = b.vstride / B::C;
  for (int i0 = 0; i0 <= j; i0 += B::CH) {
    const int kk = std::min(B::CH, j + 1 - i0);
    const ArnoldiOut o{a.H, a.t, a.ldr, j, i0, i0 + kk > j};
    const dim3 grid(reduce_ctas(nu, b.R, 33), b.R);
    const PdlLaunch l(grid, 256, 0, s, starts_early(grid));
    SAPMG_KM(arnoldi_dots_kernel, kk, ptrs_k<B>(v, i0, kk), kk, (const W*)w, nu, stride, a.partial, o)
  }
  for (int i0 = 0; i0 <= j; i0 += B::CH) {
    const int kk = std::min(B::CH, j + 1 - i0);
    const ArnoldiOut o{a.H, a.t, a.ldr, j, i0, i0 + kk > j};
    const dim3 grid(reduce_ctas(nu, b.R), b.R);
    const PdlLaunch l(grid, 256, 0, s, starts_early(grid));
    SAPMG_KM(arnoldi_update_kernel, kk, ptrs_k<B>(v, i0, kk), kk, (W*)w, (V*)vnext, nu, stride, a.partial, o)
  }
  SAPMG_CUDA_TRY(cudaGetLastError());
  return MG_OK;
}

template <class B>
static int combine_t(const BVec& b, const void* const* v, int k, const double2* y, int ldy, void* out,
                     cudaStream_t s) {
  typedef typename B::W W;
  const size_t nu = b.n / B::C, stride = b.vstride / B::C;
  const dim3 grid = stream_grid(nu, b.R);
  for (int i0 = 0; i0 < k; i0 += B::CH) {
    const int kk = std::min(B::CH, k - i0);
    const PdlLaunch l(grid, 256, 0, s, starts_early(grid));
    SAPMG_KM(combine_kernel, kk, ptrs_k<B>(v, i0, kk), kk, y + i0, ldy, (W*)out, nu, stride, i0 > 0)
  }
  SAPMG_CUDA_TRY(cudaGetLastError());
  return MG_OK;
}
#undef SAPMG_KM

// FP32 units are pairs of complex numbers: an even length, 16-byte aligned
// (FP16 basis vectors 8-byte aligned) and contiguous systems.
static bool units_ok(int basis, const BVec& b, const void* const* v, int k, const void* w) {
  if (b.vstride != b.n || b.wstride != b.n) return false;
  if (basis == P64) return true;
  bool al = b.n % 2 == 0 && (reinterpret_cast<uintptr_t>(w) & 15) == 0;
  const uintptr_t m = basis == P16 ? 7 : 15;
  for (int q = 0; q < k; ++q) al = al && (reinterpret_cast<uintptr_t>(v[q]) & m) == 0;
  return al;
}

int blas_arnoldi_step(int basis, const BVec& b, const void* const* v, int j, void* w, void* vnext,
                      const ArnoldiWork& a, cudaStream_t s) {
  if (b.R <= 0) return MG_OK;
  if (j < 0 || j > 31 || b.R > 32 || !units_ok(basis, b, v, j + 1, w)) return MG_ERR_ARG;
  const double vb = basis == P64 ? 16 : (basis == P16 ? 4 : 8), wb = basis == P64 ? 16 : 8;
  // both passes read the basis and w; v_{j+1} written
  count_bytes((2.0 * (j + 1) * vb + 2 * wb + (vnext ? vb : 0)) * b.n * b.R);
  switch (basis) {
    case P16: return arnoldi_step_t<HalfBasis>(b, v, j, w, vnext, a, s);
    case P32: return arnoldi_step_t<SingleBasis>(b, v, j, w, vnext, a, s);
    case P64: return arnoldi_step_t<DoubleBasis>(b, v, j, w, vnext, a, s);
    default: return MG_ERR_ARG;
  }
}

int blas_combine(int basis, const BVec& b, const void* const* v, int k, const double2* y, int ldy, void* out,
                 cudaStream_t s) {
  if (k <= 0 || b.R <= 0) return MG_OK;
  if (b.R > 32 || !units_ok(basis, b, v, k, out)) return MG_ERR_ARG;
  const double vb = basis == P64 ? 16 : (basis == P16 ? 4 : 8), wb = basis == P64 ? 16 : 8;
  count_bytes((k * vb + wb) * b.n * b.R);
  switch (basis) {
    case P16: return combine_t<HalfBasis>(b, v, k, y, ldy, out, s);
    case P32: return combine_t<SingleBasis>(b, v, k, y, ldy, out, s);
    case P64: return combine_t<DoubleBasis>(b, v, k, y, ldy, out, s);
    default: return MG_ERR_ARG;
  }
}

int blas_hessenberg_solve(const double2* H, int ldh, int ldr, int m, const double2* beta2, double2* y, int ldy,
                          int R, cudaStream_t s, const double2* norms, bool pairs) {
  if (m > 32) return MG_ERR_ARG;
  const PdlLaunch l(dim3((unsigned)R), 32, 0, s, starts_early(dim3((unsigned)R)));
  SAPMG_CUDA_TRY(cudaLaunchKernelEx(&l.cfg, hessenberg_solve_kernel, H, ldh, ldr, m, beta2, norms, pairs, y, ldy)); count_launches(1);
  SAPMG_CUDA_TRY(cudaGetLastError());
  return MG_OK;
}

}  // namespace sapmg
