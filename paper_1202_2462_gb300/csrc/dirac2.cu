// K1, paired form: the clover-Wilson operator D over the whole lattice (Sec. 1,
// Eq. 1.1) for an even number of right-hand sides, two per thread, FP32
// arithmetic on FP32/FP16/BF16 fields.  One CTA per (4^4 block, pair of
// right-hand sides), one thread per site; each link and clover entry is loaded
// and converted once for both right-hand sides of the pair and every add,
// multiply and FMA is the packed two-wide instruction (pair.cuh), with the -1/2
// of the hopping term folded into the reconstruction FMAs.  The pairs of one
// block are adjacent CTAs, so the block's fields are shared through L1/L2.
#include "async.cuh"
#include "internal.h"
#include "pair.cuh"

namespace sapmg {
namespace {
using namespace pair;

// Bound by the latency of the neighbours' spinors (L1 holds a quarter of the
// loads).  So a CTA asks for the spinors and fields of the CTA about one wave later
// to be brought into L2 (12 right-hand sides, FP32, 737280 sites: 783 -> 733 us; the
// same in the one-RHS kernel, with three CTAs an SM, made it slower: 203 -> 267 us),
// and what is used once stays out of L1: clover words by no-allocate loads, the
// results by streaming stores (733 -> 711 us; the links, each used twice, lose
// by it: 735 us; the block's spinors staged in shared memory: 794 us).
// AHEAD: with few pairs a block the blocks of a wave hold more of the lattice, and what
// is fetched ahead pushes the neighbours of t out of L2.  FP32, without and with,
// us: 32^4 two fields 227 and 292, four 403 and 430, six 579 and 577, eight 757 and
// 730; 16^3 x 32 two 31 and 33, four 60 and 61, six 82 and 85, eight 100 and 99, twelve 145 and
// 138; 24^4 six 189 and 186.
constexpr unsigned kAhead = 304;
static bool ahead_wins(const Geom& g, int npairs) { return npairs >= 4 || (npairs == 3 && g.nblocks >= 1024); }

// a clover entry as a broadcast pair, loaded past L1
__device__ __forceinline__ B2 once(const float2* p) {
  float x, y;
  asm volatile("ld.global.nc.L1::no_allocate.v2.f32 {%0, %1}, [%2];" : "=f"(x), "=f"(y) : "l"(p));
  B2 b; b.r = f2(x); b.i = f2(y); b.ni = f2(-y); return b;
}
__device__ __forceinline__ unsigned once_word(const void* p) {
  unsigned w;
  asm volatile("ld.global.nc.L1::no_allocate.b32 %0, [%1];" : "=r"(w) : "l"(p));
  return w;
}
__device__ __forceinline__ B2 once(const __nv_bfloat162* p) {
  const unsigned w = once_word(p);
  const float re = __uint_as_float(w << 16), im = __uint_as_float(w & 0xffff0000u);
  B2 b; b.r = f2(re); b.i = f2(im); b.ni = f2(-im); return b;
}
__device__ __forceinline__ B2 once(const __half2* p) {
  const float2 v = half2_bits_to_float2(once_word(p));
  B2 b; b.r = f2(v.x); b.i = f2(v.y); b.ni = f2(-v.y); return b;
}

template <class TG, bool AHEAD>
__global__ void __launch_bounds__(256, 2)
    dirac_pair_kernel(float2* __restrict__ out, const float2* __restrict__ in, const TG* __restrict__ U,
                      const TG* __restrict__ A, Geom g, int npairs) {
  const int blk = MG_CLAMP(kBlock, blockIdx.x / npairs, g.nblocks);
  const int loc = threadIdx.x;
  const size_t stride = (size_t)g.V * 12;
  const size_t off = (size_t)(blockIdx.x % npairs) * 2 * stride;
  if (AHEAD && threadIdx.x == 0) {
    const unsigned id = blockIdx.x + kAhead;
    if (id < gridDim.x) {
      const size_t b2 = id / npairs;
      const float2* f = in + (id % npairs) * 2 * stride + b2 * 12 * 256;
      bulk_prefetch_l2(f, 12 * 256 * sizeof(float2));
      bulk_prefetch_l2(f + stride, 12 * 256 * sizeof(float2));
      if (id % npairs == 0) {
        bulk_prefetch_l2(U + b2 * 36 * 256, 36 * 256 * sizeof(TG));
        bulk_prefetch_l2(A + b2 * 36 * 256, 36 * 256 * sizeof(TG));
      }
    }
  }
  in += off;
  out += off;
  const size_t site0 = (size_t)blk * 12 * 256 + loc;
  // acc = A psi - 1/2 sum(hops) = D psi
  P2 acc[12];
#pragma unroll
  for (int chi = 0; chi < 2; ++chi) {
    P2 p[6], o[6];
#pragma unroll
    for (int k = 0; k < 6; ++k) p[k] = ldg2(in, stride, site0 + (chi * 6 + k) * 256);
    const TG* a = A + ((size_t)(blk * 36 + chi * 18)) * 256 + loc;
    clover2_chi([&](int q) { return once(a + q * 256); }, p, o);
#pragma unroll
    for (int k = 0; k < 6; ++k) acc[chi * 6 + k] = o[k];
  }
  global_hops2<0>(g, in, stride, U, blk, loc, acc);
  global_hops2<1>(g, in, stride, U, blk, loc, acc);
  global_hops2<2>(g, in, stride, U, blk, loc, acc);
  global_hops2<3>(g, in, stride, U, blk, loc, acc);
#pragma unroll
  for (int c = 0; c < 12; ++c) {
    const size_t i = site0 + c * 256;
    __stcs(out + i, make_float2(acc[c].re.x, acc[c].im.x));
    __stcs(out + i + stride, make_float2(acc[c].re.y, acc[c].im.y));
  }
}

template <class TG>
static int run_pair(const Geom& g, void* out, const void* in, const void* U, const void* A, int nrhs, cudaStream_t s) {
  const int npairs = nrhs / 2;
  const unsigned grid = (unsigned)(g.nblocks * npairs);
  if (ahead_wins(g, npairs))
    dirac_pair_kernel<TG, true><<<grid, 256, 0, s>>>((float2*)out, (const float2*)in, (const TG*)U, (const TG*)A, g,
                                                     npairs);
  else
    dirac_pair_kernel<TG, false><<<grid, 256, 0, s>>>((float2*)out, (const float2*)in, (const TG*)U, (const TG*)A, g,
                                                      npairs);
  count_launches(1);
  SAPMG_CUDA_TRY(cudaGetLastError());
  return MG_OK;
}

}  // namespace

int launch_dirac_pair(int prec, const Geom& g, void* out, const void* in, const void* U, const void* A, int nrhs,
                      cudaStream_t s) {
  if (nrhs < 2 || nrhs % 2 != 0) return MG_ERR_ARG;
  switch (prec) {
    case P32: return run_pair<float2>(g, out, in, U, A, nrhs, s);
    case P16: return run_pair<__half2>(g, out, in, U, A, nrhs, s);
    case PBF: return run_pair<__nv_bfloat162>(g, out, in, U, A, nrhs, s);
    default: return MG_ERR_ARG;
  }
}

}  // namespace sapmg
