// Global orthonormalisation of the set-up's FP32 test vectors (Sec. 3: "kept
// orthonormal") by Cholesky QR, twice (Yamamoto, Nakatsukasa, Yanagisawa,
// Fukaya, ETNA 44, 2015): G = V^dagger V, G = R^dagger R, V <- V R^{-1}, the
// positive-diagonal QR factor of V as Gram-Schmidt in vector order gives it.
//
// Vector by vector, two classical Gram-Schmidt passes read the earlier vectors
// four times per vector: 760 vector reads for N = 20, 4.3 ms at 16^3 x 32 in
// 190 launches.  Here a pass reads every vector once for G and reads and writes it
// once for the triangular solve, which an element's N values, held in
// registers, go through in place.
//
// G's condition is the square of V's.  A pivot of the first factorisation below
// kPivot of its diagonal entry (a vector within 0.6 degrees of the span of the
// earlier ones, or zero, or not finite) raises a flag, on which the solves leave
// V as it was and the caller orthonormalises vector by vector instead; above it
// the first pass is orthogonal to 1e-2 and the second to rounding.
#include "accum.cuh"
#include "internal.h"
#include "blas.h"

namespace sapmg {
namespace {

constexpr double kPivot = 1e-4;
constexpr int kChunkE = 64;          // elements per staged chunk
constexpr int kRun = 32;             // products in one FP32 sum

__device__ __forceinline__ void cp_async8(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}

// Partial Gram matrices: the upper triangle in 4 x 4 tiles of vectors; thread
// (tile pair, group) takes every G-th element of the staged chunk.  Bound by the FP32
// units (N^2 / 2 complex products an element).  Sums of kRun products go to totals of
// two floats each (accum.cuh) in shared memory: a thread meets 5000 elements at 32^3 x 64.
template <int STAGES>
__global__ void __launch_bounds__(256, 2) gram_kernel(const float2* __restrict__ V, int N, size_t n, int T,
                                                   double2* __restrict__ partial) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int P = T * (T + 1) / 2, G = 256 / P, ld = 4 * T + 2;      // row stride of a staged element
  float2* sx = reinterpret_cast<float2*>(smem);
  float4* tot = reinterpret_cast<float4*>(smem + sizeof(float2) * STAGES * kChunkE * ld);   // [entry][thread]
  const int tid = threadIdx.x, pair = tid % P, grp = tid / P;
  int ti = 0, tj = pair;
  while (tj >= T - ti) { tj -= T - ti; ++ti; }
  tj += ti;
  // vectors N .. 4 T - 1 stay zero in every stage
  for (int e = tid; e < STAGES * kChunkE * ld; e += 256) sx[e] = make_float2(0.f, 0.f);
  for (int k = 0; k < 16; ++k) tot[k * 256 + tid] = make_float4(0.f, 0.f, 0.f, 0.f);
  __syncthreads();
  const size_t nchunk = (n + kChunkE - 1) / kChunkE;
  auto load = [&](size_t ch, int st) {
    if (ch < nchunk) {
      float2* d = sx + st * kChunkE * ld;
      for (int q = tid; q < N * kChunkE; q += 256) {
        const int v = q / kChunkE, e = q % kChunkE;
        const size_t i = ch * kChunkE + e;
        if (i < n) cp_async8(d + e * ld + v, V + (size_t)v * n + i);
        else d[e * ld + v] = make_float2(0.f, 0.f);
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  size_t ch = blockIdx.x;
  for (int s = 0; s < STAGES - 1; ++s) load(ch + (size_t)s * gridDim.x, s);
  Cplx<float> acc[4][4];
  auto flush = [&] {                                               // a thread's own totals: no barrier
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      Cplx<float>& a = acc[k >> 2][k & 3];
      const float4 t = tot[k * 256 + tid];
      Acc<float> re{t.x, t.y}, im{t.z, t.w};
      re.add(Acc<float>::of(a.re));
      im.add(Acc<float>::of(a.im));
      tot[k * 256 + tid] = make_float4(re.h, re.l, im.h, im.l);
      a = cmk(0.f, 0.f);
    }
  };
#pragma unroll
  for (int k = 0; k < 16; ++k) acc[k >> 2][k & 3] = cmk(0.f, 0.f);
  const int run = max(1, kRun * G / kChunkE);                      // chunks a sum
  int left = run;
  for (int st = 0; ch < nchunk; ch += gridDim.x, st = st + 1 == STAGES ? 0 : st + 1) {
    asm volatile("cp.async.wait_group %0;" ::"n"(STAGES - 2) : "memory");
    __syncthreads();
    load(ch + (size_t)(STAGES - 1) * gridDim.x, st == 0 ? STAGES - 1 : st - 1);
    if (grp < G) {
      const float2* x = sx + st * kChunkE * ld;
      for (int e = grp; e < kChunkE; e += G) {
        const float4* xa = reinterpret_cast<const float4*>(x + e * ld + 4 * ti);
        const float4* xb = reinterpret_cast<const float4*>(x + e * ld + 4 * tj);
        const float4 a0 = xa[0], a1 = xa[1], b0 = xb[0], b1 = xb[1];
        const Cplx<float> a[4] = {cmk(a0.x, a0.y), cmk(a0.z, a0.w), cmk(a1.x, a1.y), cmk(a1.z, a1.w)};
        const Cplx<float> b[4] = {cmk(b0.x, b0.y), cmk(b0.z, b0.w), cmk(b1.x, b1.y), cmk(b1.z, b1.w)};
#pragma unroll
        for (int p = 0; p < 4; ++p)
#pragma unroll
          for (int q = 0; q < 4; ++q) cfma_conj(acc[p][q], a[p], b[q]);
      }
    }
    if (--left == 0) {
      flush();
      left = run;
    }
  }
  flush();
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();
  // the groups' totals: entry e of the tiles, its groups shared by as many threads as there are
  const int ne = P * 16, share = max(1, 256 / ne), e0 = tid % ne, part = tid / ne;
  for (int e = e0; e < ne && part < share; e += 256) {
    float4* t = tot + (e & 15) * 256 + (e >> 4);
    Acc<float> re{0.f, 0.f}, im{0.f, 0.f};
    for (int g = part; g < G; g += share) {
      re.add(Acc<float>{t[g * P].x, t[g * P].y});
      im.add(Acc<float>{t[g * P].z, t[g * P].w});
    }
    t[part * P] = make_float4(re.h, re.l, im.h, im.l);
  }
  __syncthreads();
  for (int e = tid; e < ne; e += 256) {
    const float4* t = tot + (e & 15) * 256 + (e >> 4);
    double a = 0, b = 0;
    for (int g = 0; g < share; ++g) {
      a += (double)t[g * P].x + (double)t[g * P].y;
      b += (double)t[g * P].z + (double)t[g * P].w;
    }
    partial[(size_t)blockIdx.x * ne + e] = make_double2(a, b);
  }
}

// CTA per tile pair: Gm[i][j] (leading dimension 32) of its sixteen entries
__global__ void __launch_bounds__(256) gram_sum_kernel(const double2* __restrict__ partial, int ncta, int T,
                                                       double2* __restrict__ Gm) {
  __shared__ double2 red[16][16];
  const int P = T * (T + 1) / 2, pair = blockIdx.x, e = threadIdx.x & 15, part = threadIdx.x >> 4;
  int ti = 0, tj = pair;
  while (tj >= T - ti) { tj -= T - ti; ++ti; }
  tj += ti;
  double a = 0, b = 0;
  for (int c = part; c < ncta; c += 16) {
    const double2 v = partial[((size_t)c * P + pair) * 16 + e];
    a += v.x;
    b += v.y;
  }
  red[part][e] = make_double2(a, b);
  __syncthreads();
  if (part == 0) {
    for (int q = 1; q < 16; ++q) { a += red[q][e].x; b += red[q][e].y; }
    Gm[(4 * ti + (e >> 2)) * 32 + 4 * tj + (e & 3)] = make_double2(a, b);
  }
}

// R of G = R^dagger R (upper triangle of Gm), FP64, one CTA; coef[k][j] = R_jk (j < k) and coef[k][k] = 1 / R_kk
// as floats.  flag is raised by a pivot below kPivot of its diagonal entry.
__global__ void __launch_bounds__(256) gram_chol_kernel(const double2* __restrict__ Gm, int N,
                                                        float2* __restrict__ coef, int* __restrict__ flag) {
  __shared__ double2 a[32][33];
  __shared__ double diag[32];
  const int tid = threadIdx.x;
  for (int e = tid; e < N * N; e += 256)
    if (e / N <= e % N) a[e / N][e % N] = Gm[(e / N) * 32 + e % N];
  __syncthreads();
  if (tid < N) diag[tid] = a[tid][tid].x;
  __syncthreads();
  for (int k = 0; k < N; ++k) {
    const double d = a[k][k].x;
    const bool ok = d > kPivot * diag[k];                           // false for NaN and for a zero vector
    const double inv = ok ? rsqrt(d) : 0.0;
    if (!ok && tid == 0) *flag = 1;
    __syncthreads();
    if (tid > k && tid < N) a[k][tid] = make_double2(a[k][tid].x * inv, a[k][tid].y * inv);
    if (tid == 0) coef[k * 32 + k] = make_float2((float)inv, 0.f);
    __syncthreads();
    const int m = N - 1 - k;
    for (int e = tid; e < m * m; e += 256) {
      const int i = k + 1 + e / m, j = k + 1 + e % m;
      if (j < i) continue;
      const double2 p = a[k][i], q = a[k][j];                       // conj(R_ki) R_kj
      a[i][j] = make_double2(a[i][j].x - (p.x * q.x + p.y * q.y), a[i][j].y - (p.x * q.y - p.y * q.x));
    }
    __syncthreads();
  }
  for (int e = tid; e < N * N; e += 256) {
    const int j = e / N, k = e % N;
    if (j < k) coef[k * 32 + j] = make_float2((float)a[j][k].x, (float)a[j][k].y);
  }
}

// v_k <- (v_k - sum_{j<k} R_jk v_j) / R_kk in place, two elements a thread.  HBM-bound.
template <int NT>
__global__ void __launch_bounds__(256) tri_kernel(float4* __restrict__ V, int N, size_t nu,
                                                  const float2* __restrict__ coef, const int* __restrict__ flag) {
  __shared__ float2 c[NT][NT];
  if (*flag) return;
  for (int e = threadIdx.x; e < NT * NT; e += 256)
    c[e / NT][e % NT] = e / NT < N && e % NT <= e / NT ? coef[(e / NT) * 32 + e % NT] : make_float2(0.f, 0.f);
  __syncthreads();
  const size_t i = (size_t)blockIdx.x * 256 + threadIdx.x;
  if (i >= nu) return;
  float4 v[NT];
#pragma unroll
  for (int k = 0; k < NT; ++k)
    if (k < N) v[k] = V[(size_t)k * nu + i];
#pragma unroll
  for (int k = 0; k < NT; ++k) {
    if (k < N) {
#pragma unroll
      for (int j = 0; j < k; ++j) {
        const float2 r = c[k][j];
        v[k].x = fmaf(-r.x, v[j].x, fmaf(r.y, v[j].y, v[k].x));
        v[k].y = fmaf(-r.x, v[j].y, fmaf(-r.y, v[j].x, v[k].y));
        v[k].z = fmaf(-r.x, v[j].z, fmaf(r.y, v[j].w, v[k].z));
        v[k].w = fmaf(-r.x, v[j].w, fmaf(-r.y, v[j].z, v[k].w));
      }
      const float d = c[k][k].x;
      v[k].x *= d;
      v[k].y *= d;
      v[k].z *= d;
      v[k].w *= d;
      V[(size_t)k * nu + i] = v[k];
    }
  }
}

}  // namespace

int launch_cholqr2(void* V, int N, size_t n, double2* partial, double2* work, int* flag, cudaStream_t s) {
  if (N < 1 || N > 32 || n % 2 != 0 || (reinterpret_cast<uintptr_t>(V) & 15) != 0) return MG_ERR_ARG;
  const int T = (N + 3) / 4, P = T * (T + 1) / 2;
  const int ncta = (int)std::min<size_t>({(size_t)304, (n + kChunkE - 1) / kChunkE, kPartialSums / (size_t)(P * 16)});
  const int stages = T < 8 ? 3 : 2;                                // two CTAs' totals and stages on an SM
  const size_t smem = (size_t)stages * kChunkE * (4 * T + 2) * sizeof(float2) + (size_t)16 * 256 * sizeof(float4);
  double2* Gm = work;                                              // [32][32]
  float2* coef = reinterpret_cast<float2*>(work + 32 * 32);        // [32][32]
  static bool attr = false;
  if (!attr) {
    SAPMG_CUDA_TRY(cudaFuncSetAttribute(gram_kernel<3>, cudaFuncAttributeMaxDynamicSharedMemorySize, 112 * 1024));
    SAPMG_CUDA_TRY(cudaFuncSetAttribute(gram_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, 112 * 1024));
    attr = true;
  }
  SAPMG_CUDA_TRY(cudaMemsetAsync(flag, 0, sizeof(int), s));
  const unsigned tri = (unsigned)((n / 2 + 255) / 256);
  for (int pass = 0; pass < 2; ++pass) {
    if (stages == 3) gram_kernel<3><<<ncta, 256, smem, s>>>((const float2*)V, N, n, T, partial);
    else gram_kernel<2><<<ncta, 256, smem, s>>>((const float2*)V, N, n, T, partial);
    gram_sum_kernel<<<P, 256, 0, s>>>(partial, ncta, T, Gm);
    gram_chol_kernel<<<1, 256, 0, s>>>(Gm, N, coef, flag);
    if (N <= 8) tri_kernel<8><<<tri, 256, 0, s>>>((float4*)V, N, n / 2, coef, flag);
    else if (N <= 16) tri_kernel<16><<<tri, 256, 0, s>>>((float4*)V, N, n / 2, coef, flag);
    else if (N <= 24) tri_kernel<24><<<tri, 256, 0, s>>>((float4*)V, N, n / 2, coef, flag);
    else tri_kernel<32><<<tri, 256, 0, s>>>((float4*)V, N, n / 2, coef, flag);
    count_launches(4);
  }
  SAPMG_CUDA_TRY(cudaGetLastError());
  return MG_OK;
}

}  // namespace sapmg
