// K1: the clover-Wilson operator D over the whole lattice (Sec. 1, Eq. 1.1).
//
// One CTA per 4^4 block, one thread per site, fields in the blocked
// structure-of-arrays layout so that a warp's loads of one component are 256
// contiguous bytes (float2).  Hops are spin-projected (6 complex per
// neighbour instead of 12) and the antiperiodic time boundary, if any, is
// folded into the stored links.
#include "internal.h"
#include "stencil.cuh"
#include "dfloat.cuh"
#include "quad.cuh"

namespace sapmg {

// DAG: apply D^dagger = gamma5 D gamma5 instead (the operator of the normal
// equations).  NORM: also write the CTA's share of ||out||^2 to
// part[blockIdx.x] (CTA index = block * nrhs + right-hand side), reduced in a
// fixed order so that the result does not depend on scheduling.
template <class R, class TS, class TG, bool DAG, bool NORM>
__global__ void __launch_bounds__(256, (sizeof(R) == 4 ? 3 : 1)) dirac_kernel(TS* __restrict__ out, const TS* __restrict__ in,
                                                    const TG* __restrict__ U, const TG* __restrict__ A, Geom g,
                                                    int nrhs, double* __restrict__ part) {
  // right-hand side fastest in the grid: the CTAs of one block run back to
  // back and share its links and clover through L2
  const int blk = MG_CLAMP(kBlock, blockIdx.x / nrhs, g.nblocks);
  const int loc = threadIdx.x;
  const size_t off = (size_t)(blockIdx.x % nrhs) * g.V * 12;
  in += off;
  out += off;
  // acc = A psi - (sum of hops) / 2, the halves exact products of the adding FMAs (FP64,
  // 12 fields, 663552 sites: 16.3 -> 15.7 ms against scaling A psi by -2 and the sum
  // by -1/2, 48 of 1176 instructions of the FP64 units that bound it); double-float
  // arithmetic, where a product costs ten times an addition, keeps the scaling
  constexpr bool kFma = !std::is_same<R, DF>::value;
  constexpr int HOW = kFma ? kHalf : kAdd;
  Cplx<R> acc[12];
  {
    Cplx<R> p[12];
    load_spinor<R>(in, blk, loc, p);
    clover_apply<R>(A, blk, loc, p, acc);
  }
  if constexpr (!kFma) {
#pragma unroll
    for (int c = 0; c < 12; ++c) acc[c] = (R)(-2) * acc[c];
  }
  hops_global_dir<0, R, TS, TG, DAG, HOW>(g, in, U, blk, loc, acc);
  hops_global_dir<1, R, TS, TG, DAG, HOW>(g, in, U, blk, loc, acc);
  hops_global_dir<2, R, TS, TG, DAG, HOW>(g, in, U, blk, loc, acc);
  hops_global_dir<3, R, TS, TG, DAG, HOW>(g, in, U, blk, loc, acc);
  if constexpr (!kFma) {
#pragma unroll
    for (int c = 0; c < 12; ++c) acc[c] = (R)(-0.5) * acc[c];
  }
  store_spinor<R>(out, blk, loc, acc);
  if constexpr (NORM) {
    __shared__ double ws[8];
    R t = 0;
#pragma unroll
    for (int c = 0; c < 12; ++c) t += acc[c].re * acc[c].re + acc[c].im * acc[c].im;
    t = warp_sum(t);
    if ((loc & 31) == 0) ws[loc >> 5] = (double)t;
    __syncthreads();
    if (loc == 0) {
      double sum = 0;
      for (int w = 0; w < 8; ++w) sum += ws[w];
      part[blockIdx.x] = sum;
    }
  }
}

// The same for few blocks: eight CTAs of 32 sites a block, four threads a site (quad.cuh).
template <class R, class TS, class TG, bool DAG>
__global__ void __launch_bounds__(128) dirac_quad_kernel(TS* __restrict__ out, const TS* __restrict__ in,
                                                         const TG* __restrict__ U, const TG* __restrict__ A, Geom g,
                                                         int nrhs) {
  __shared__ __align__(16) unsigned char part_raw[sizeof(Cplx<R>) * 4 * 12 * 32];
  Cplx<R>* part = reinterpret_cast<Cplx<R>*>(part_raw);
  const int id = blockIdx.x >> 3, blk = MG_CLAMP(kBlock, id / nrhs, g.nblocks);
  const int m = threadIdx.x >> 5, lane = threadIdx.x & 31, loc = (blockIdx.x & 7) * 32 + lane;
  const size_t off = (size_t)(id % nrhs) * g.V * 12;
  in += off;
  out += off;
  Cplx<R> o[3];
  switch (m) {
    case 0: quad_dirac<0, R, TS, TG, DAG>(g, in, U, A, blk, loc, lane, part, o); break;
    case 1: quad_dirac<1, R, TS, TG, DAG>(g, in, U, A, blk, loc, lane, part, o); break;
    case 2: quad_dirac<2, R, TS, TG, DAG>(g, in, U, A, blk, loc, lane, part, o); break;
    default: quad_dirac<3, R, TS, TG, DAG>(g, in, U, A, blk, loc, lane, part, o); break;
  }
  TS* q = out + (size_t)blk * 12 * 256 + loc;
#pragma unroll
  for (int k = 0; k < 3; ++k) Io<R, TS>::st(q + (3 * m + k) * 256, o[k]);
}

// Few blocks: FP64 below eight blocks an SM, where the last wave of whole blocks
// leaves a tenth or more of the FP64 units' time unused (16 blocks, 8^4: 87 us
// with a CTA per block on 16 SMs, 46 us with a warp per 32 sites); FP32, which
// needs the warps of a block to hide latency, below one block an SM.  Double-float
// arithmetic runs on the FP32 units, where a block alone on an SM loses little:
// whole blocks 148 us a wave of 152; four threads a site 40 us at 16 blocks, 134 at
// 96, 192 at 128, 268 at 192, 331 at 240, 438 at 320.
template <class R>
static bool few_blocks(const Geom& g, int nrhs) {
  const long long n = (long long)g.nblocks * nrhs;
  if (std::is_same<R, DF>::value) return 20 * idle_sms(n) > 9 * n;
  return n < 152 * (sizeof(R) == 8 ? 8 : 1);
}

template <class R, class TS, class TG, bool DAG, bool NORM>
static void run(const Geom& g, void* out, const void* in, const void* U, const void* A, int nrhs, double* part,
                cudaStream_t s) {
  const unsigned ctas = (unsigned)(g.nblocks * nrhs);
  if constexpr (!NORM) {
    if (few_blocks<R>(g, nrhs)) {
      dirac_quad_kernel<R, TS, TG, DAG><<<ctas * 8, 128, 0, s>>>((TS*)out, (const TS*)in, (const TG*)U, (const TG*)A,
                                                                 g, nrhs);
      count_launches(1);
      return;
    }
  }
  dirac_kernel<R, TS, TG, DAG, NORM><<<ctas, 256, 0, s>>>((TS*)out, (const TS*)in, (const TG*)U, (const TG*)A, g, nrhs,
                                                          part);
  count_launches(1);
}

template <class R, class TS, class TG>
static void run_ex(const Geom& g, void* out, const void* in, const void* U, const void* A, int nrhs, bool dag,
                   double* part, cudaStream_t s) {
  if (dag) {
    if (part) run<R, TS, TG, true, true>(g, out, in, U, A, nrhs, part, s);
    else run<R, TS, TG, true, false>(g, out, in, U, A, nrhs, part, s);
  } else {
    if (part) run<R, TS, TG, false, true>(g, out, in, U, A, nrhs, part, s);
    else run<R, TS, TG, false, false>(g, out, in, U, A, nrhs, part, s);
  }
}

int launch_dirac_ex(int prec, const Geom& g, void* out, const void* in, const void* U, const void* A, int nrhs,
                    bool dag, double* part, cudaStream_t s) {
  switch (prec) {
    case P64: run_ex<double, double2, double2>(g, out, in, U, A, nrhs, dag, part, s); break;
    case P64E:                             // FP64 data, double-float arithmetic (dfloat.cuh)
      if (dag || part) return MG_ERR_ARG;
      run<DF, double2, double2, false, false>(g, out, in, U, A, nrhs, nullptr, s);
      break;
    case P32: run_ex<float, float2, float2>(g, out, in, U, A, nrhs, dag, part, s); break;
    case P16:
      if (dag || part) return MG_ERR_ARG;
      run<float, float2, __half2, false, false>(g, out, in, U, A, nrhs, nullptr, s);
      break;
    case PBF:
      if (dag || part) return MG_ERR_ARG;
      run<float, float2, __nv_bfloat162, false, false>(g, out, in, U, A, nrhs, nullptr, s);
      break;
    default: return MG_ERR_ARG;
  }
  SAPMG_CUDA_TRY(cudaGetLastError());
  return MG_OK;
}

int launch_dirac(int prec, const Geom& g, void* out, const void* in, const void* U, const void* A, int nrhs,
                 cudaStream_t s) {
  return launch_dirac_ex(prec, g, out, in, U, A, nrhs, false, nullptr, s);
}

}  // namespace sapmg
