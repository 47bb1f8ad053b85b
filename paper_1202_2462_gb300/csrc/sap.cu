// K2: one colour pass of red-black Schwarz (Sec. 2, Algorithm 1).
//
// For every block i of colour c (blocks of one colour never touch, so they
// run as independent CTAs of one launch):
//   r = b - D z on the block's sites (full operator: halo z from the
//       neighbouring blocks of the other colour),
//   e ~ D_i^{-1} r by n_MR minimal-residual steps with the Dirichlet block
//       operator D_i = I^T D I (hops leaving the block dropped),
//   z += e.
// One CTA per block, one thread per site.  The MR iterate rho lives in shared
// memory for the neighbour accesses of D_i, and so does the correction e; the
// block-wide dots are warp shuffles plus one shared-memory exchange.  The two
// colours are two launches in stream order.
#include "cluster.cuh"
#include "internal.h"
#include "quad.cuh"
#include "stencil.cuh"

namespace sapmg {

template <class R>
__device__ __forceinline__ void load_smem_spinor(const Cplx<R>* __restrict__ s, int loc, Cplx<R> (&p)[12]) {
#pragma unroll
  for (int c = 0; c < 12; ++c) p[c] = s[c * 256 + loc];
}

// acc - (hops of D_i at loc) / 2 (neighbours inside the block only, from shared memory).
template <int MU, class R, class TG>
__device__ __forceinline__ void block_hops_dir(const TG* __restrict__ U, const Cplx<R>* __restrict__ rs, int blk,
                                               int loc, Cplx<R> (&acc)[12]) {
  const int ls = 1 << (2 * MU);
  const int c = (loc >> (2 * MU)) & 3;
  Cplx<R> h[6], gg[6], u[9];
  if (c < 3) {
    const Cplx<R>* q = rs + loc + ls;
    spin_project_ld<MU, -1, R>([&](int k) { return q[k * 256]; }, h);
    load_link<R>(U, blk, MU, loc, u);
    su3_mul(u, h, gg);
    spin_reconstruct_add<MU, -1, R, kHalf>(gg, acc);
  }
  if (c > 0) {
    const Cplx<R>* q = rs + loc - ls;
    spin_project_ld<MU, 1, R>([&](int k) { return q[k * 256]; }, h);
    load_link<R>(U, blk, MU, loc - ls, u);
    su3_dag_mul(u, h, gg);
    spin_reconstruct_add<MU, 1, R, kHalf>(gg, acc);
  }
}

template <class R>
__device__ __forceinline__ void block_reduce3(R& a, R& b, R& c, R (*red)[4]) {
  a = warp_sum(a);
  b = warp_sum(b);
  c = warp_sum(c);
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0) { red[w][0] = a; red[w][1] = b; red[w][2] = c; }
  __syncthreads();
  a = b = c = 0;
#pragma unroll
  for (int k = 0; k < 8; ++k) { a += red[k][0]; b += red[k][1]; c += red[k][2]; }
}

// Shared memory per CTA: the MR iterate rho and the block correction e
// (12 x 256 complex each, structure of arrays), and the reduction scratch.
// Registers hold one site's operator image p and the stencil temporaries only,
// so that two CTAs fit on an SM in FP32.
template <class R, class TS, class TG>
__global__ void __launch_bounds__(256, (sizeof(R) == 4 ? 2 : 1))
    sap_colour_kernel(TS* __restrict__ z, const TS* __restrict__ b, const TG* __restrict__ U,
                      const TG* __restrict__ A, Geom g, int colour, int n_mr, int nrhs) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Cplx<R>* rs = reinterpret_cast<Cplx<R>*>(smem_raw);                    // [12][256]
  Cplx<R>* es = rs + 12 * 256;                                            // [12][256]
  R (*red)[4] = reinterpret_cast<R (*)[4]>(smem_raw + sizeof(Cplx<R>) * 24 * 256);
  // right-hand side fastest in the grid (links and clover of a block shared through L2)
  const size_t off = (size_t)(blockIdx.x % nrhs) * g.V * 12;
  z += off;
  if (b) b += off;
  const int blk = colour_block(g, blockIdx.x / nrhs, colour);
  const int loc = threadIdx.x;

  // residual r = b - D z (Algorithm 1: residual update before the colour's block solves);
  // acc = D z = A z - (sum of hops) / 2
  {
    Cplx<R> acc[12];
    {
      Cplx<R> zz[12];
      load_spinor<R>(z, blk, loc, zz);
      clover_apply<R>(A, blk, loc, zz, acc);
    }
    hops_global_dir<0, R, TS, TG, false, kHalf>(g, z, U, blk, loc, acc);
    asm volatile("" ::: "memory");
    hops_global_dir<1, R, TS, TG, false, kHalf>(g, z, U, blk, loc, acc);
    asm volatile("" ::: "memory");
    hops_global_dir<2, R, TS, TG, false, kHalf>(g, z, U, blk, loc, acc);
    asm volatile("" ::: "memory");
    hops_global_dir<3, R, TS, TG, false, kHalf>(g, z, U, blk, loc, acc);
    const size_t bq = (size_t)blk * 12 * 256 + loc;
#pragma unroll
    for (int c = 0; c < 12; ++c)
      rs[c * 256 + loc] = (b ? Io<R, TS>::ldc(b + bq + c * 256) : cmk<R>(0, 0)) - acc[c];
  }
  TS* zq = z + (size_t)blk * 12 * 256 + loc;

  // n_MR minimal-residual steps on D_i e = r, D_i the block operator (hops leaving the block dropped)
  for (int it = 0; it < n_mr; ++it) {
    __syncthreads();                                   // rho of every site written
    Cplx<R> p[12];
    {
      Cplx<R> ro[12];
      load_smem_spinor(rs, loc, ro);
      clover_apply<R>(A, blk, loc, ro, p);
    }
    // the empty asm statements keep the compiler from hoisting the next
    // direction's loads (which would raise register pressure past the limit)
    block_hops_dir<0>(U, rs, blk, loc, p);
    asm volatile("" ::: "memory");
    block_hops_dir<1>(U, rs, blk, loc, p);
    asm volatile("" ::: "memory");
    block_hops_dir<2>(U, rs, blk, loc, p);
    asm volatile("" ::: "memory");
    block_hops_dir<3>(U, rs, blk, loc, p);
    R pr_re = 0, pr_im = 0, pp = 0;
#pragma unroll
    for (int c = 0; c < 12; ++c) {
      const Cplx<R> ro = rs[c * 256 + loc];
      pr_re += p[c].re * ro.re + p[c].im * ro.im;
      pr_im += p[c].re * ro.im - p[c].im * ro.re;
      pp += p[c].re * p[c].re + p[c].im * p[c].im;
    }
    block_reduce3(pr_re, pr_im, pp, red);            // contains the barrier after all neighbour reads
    Cplx<R> alpha = cmk<R>(0, 0);
    if (pp > (R)0) alpha = cmk(pr_re / pp, pr_im / pp);
    // the first step starts e, the last adds it to z (own site only: no barrier needed)
#pragma unroll
    for (int c = 0; c < 12; ++c) {
      const Cplx<R> ro = rs[c * 256 + loc];
      Cplx<R> e = alpha * ro;
      if (it > 0) e = es[c * 256 + loc] + e;
      if (it == n_mr - 1) {
        Io<R, TS>::st(zq + c * 256, Io<R, TS>::ldc(zq + c * 256) + e);
      } else {
        es[c * 256 + loc] = e;
        rs[c * 256 + loc] = ro - alpha * p[c];
      }
    }
  }
}

// The same pass with a block on a cluster of eight CTAs of 32 sites, four threads
// a site (quad.cuh), for few blocks: a block's MR steps then run on eight SMs
// instead of one.  FP64 is bound by the SMs' FP64 units, so the 8 blocks of a
// colour of 8^4 took 514 us a pass on 8 SMs (262 us with one thread a site on
// clusters of eight warps).  rho stays in the shared memory of the CTA that owns
// the site, its neighbours read it through distributed shared memory; e, p and
// the update of a component belong to one thread.
// Rows 3 M .. 3 M + 2 of D_i rho at the warp's sites (rsa: the address of the CTAs' rho, [12][32])
template <int M, class R, class TG>
__device__ __forceinline__ void quad_block(const Geom& g, const TG* __restrict__ U, const TG* __restrict__ A,
                                           const Cplx<R>* rs, uint32_t rsa, int blk, int loc, Cplx<R>* part,
                                           Cplx<R> (&out)[3]) {
  const int ls = 1 << (2 * M), cm = (loc >> (2 * M)) & 3, lane = loc & 31;
  auto at = [&](int l) { return cluster_addr(rsa + (uint32_t)((l & 31) * sizeof(Cplx<R>)), l >> 5); };
  const uint32_t q0 = at(cm < 3 ? loc + ls : loc), q1 = at(cm > 0 ? loc - ls : loc);
  Cplx<R> acc[12];
  quad_hops<M, R, TG, false>(
      g, U, blk, loc,
      [&](int step, int c) { return cluster_ld((step > 0 ? q0 : q1) + (uint32_t)(c * 32 * sizeof(Cplx<R>)), R(0)); },
      [&](int step) { return step > 0 ? cm < 3 : cm > 0; }, acc);
  quad_clover<M, R>(A, blk, loc, [&](int c) { return rs[c * 32 + lane]; }, out);
  quad_swap<M>(part, lane, acc, out);
}

template <class R, class TS, class TG>
__global__ void __launch_bounds__(128) sap_cluster_kernel(TS* __restrict__ z, const TS* __restrict__ b,
                                                          const TG* __restrict__ U, const TG* __restrict__ A, Geom g,
                                                          int colour, int n_mr, int nrhs) {
  __shared__ __align__(16) unsigned char smem_raw[sizeof(Cplx<R>) * 5 * 12 * 32];
  __shared__ R red[2][32][4];                            // two buffers: a step's sums are read while the next arrive
  Cplx<R>* rs = reinterpret_cast<Cplx<R>*>(smem_raw);    // rho of the CTA's sites [12][32]
  Cplx<R>* part = rs + 12 * 32;                          // [4][12][32]
  const uint32_t rsa = smem_u32(rs);
  const int rank = (int)(blockIdx.x & 7), m = threadIdx.x >> 5, lane = threadIdx.x & 31, loc = rank * 32 + lane;
  const int id = blockIdx.x >> 3;
  const size_t off = (size_t)(id % nrhs) * g.V * 12;
  z += off;
  if (b) b += off;
  const int blk = colour_block(g, id / nrhs, colour);
  const size_t own = ((size_t)blk * 12 + 3 * m) * 256 + loc;   // this thread's components 3 m .. 3 m + 2
  Cplx<R> ro[3], e[3], p[3];
  switch (m) {
    case 0: quad_dirac<0, R, TS, TG, false>(g, z, U, A, blk, loc, lane, part, p); break;
    case 1: quad_dirac<1, R, TS, TG, false>(g, z, U, A, blk, loc, lane, part, p); break;
    case 2: quad_dirac<2, R, TS, TG, false>(g, z, U, A, blk, loc, lane, part, p); break;
    default: quad_dirac<3, R, TS, TG, false>(g, z, U, A, blk, loc, lane, part, p); break;
  }
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    ro[k] = (b ? Io<R, TS>::ldc(b + own + k * 256) : cmk<R>(0, 0)) - p[k];
    rs[(3 * m + k) * 32 + lane] = ro[k];
    e[k] = cmk<R>(0, 0);
  }
  for (int it = 0; it < n_mr; ++it) {
    cluster_barrier();                               // rho of every site written, part free again
    switch (m) {
      case 0: quad_block<0, R, TG>(g, U, A, rs, rsa, blk, loc, part, p); break;
      case 1: quad_block<1, R, TG>(g, U, A, rs, rsa, blk, loc, part, p); break;
      case 2: quad_block<2, R, TG>(g, U, A, rs, rsa, blk, loc, part, p); break;
      default: quad_block<3, R, TG>(g, U, A, rs, rsa, blk, loc, part, p); break;
    }
    R v[3] = {0, 0, 0};
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      v[0] += p[k].re * ro[k].re + p[k].im * ro[k].im;
      v[1] += p[k].re * ro[k].im - p[k].im * ro[k].re;
      v[2] += p[k].re * p[k].re + p[k].im * p[k].im;
    }
#pragma unroll
    for (int q = 0; q < 3; ++q) v[q] = warp_sum(v[q]);
    if (lane < 8) {                                      // lane q: this warp's sums to CTA q
      const uint32_t a = cluster_addr(smem_u32(&red[it & 1][rank * 4 + m][0]), lane);
#pragma unroll
      for (int q = 0; q < 3; ++q) cluster_st(a + (uint32_t)(q * sizeof(R)), v[q]);
    }
    cluster_barrier();                               // the sums arrived; every neighbour read of rho done
    // the 32 warps' sums, one a lane
#pragma unroll
    for (int q = 0; q < 3; ++q) v[q] = warp_sum(red[it & 1][lane][q]);
    Cplx<R> alpha = cmk<R>(0, 0);
    if (v[2] > (R)0) alpha = cmk(v[0] / v[2], v[1] / v[2]);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      e[k] = e[k] + alpha * ro[k];
      ro[k] = ro[k] - alpha * p[k];
      rs[(3 * m + k) * 32 + lane] = ro[k];
    }
  }
  cluster_barrier();                                 // n_mr = 0: the residuals' reads of z are over
#pragma unroll
  for (int k = 0; k < 3; ++k) Io<R, TS>::st(z + own + k * 256, Io<R, TS>::ldc(z + own + k * 256) + e[k]);
}

// A cluster per block where whole blocks leave SMs idle.  n blocks of a colour; one
// sweep (two passes, n_MR = 4) by whole blocks and by clusters, us:
// FP32 (whole blocks 50 up to 152): 46 at 72, 50 at 88, 84 at 104, where clusters no
//   longer all fit at once.
// FP64 (bound by the SMs' FP64 units, one block an SM at a time): whole blocks take
//   979 a wave of 152, clusters 7.75 a block and 70; so 104: 979 and 919, 120: 979 and
//   1057, 224: 1962 and 1805, 256: 1962 and 2039, 480: 3916 and 3730, 512: 3916 and 3967.
template <class R>
static bool cluster_wins(const Geom& g, int nrhs) {
  const long long n = (long long)(g.nblocks / 2) * nrhs, idle = idle_sms(n);
  if (sizeof(R) == 4) return n < 96;
  return n < 608 && 5 * idle > n + 55;       // 6.44 (n + idle) > 7.75 n + 70
}

template <class R, class TS, class TG>
static int run_cluster(const Geom& g, void* z, const void* b, const void* U, const void* A, int colour, int n_mr,
                       int nrhs, cudaStream_t s) {
  ClusterLaunch l((unsigned)(g.nblocks / 2 * nrhs * 8), 128, 0, 8, s);
  SAPMG_CUDA_TRY(cudaLaunchKernelEx(&l.cfg, sap_cluster_kernel<R, TS, TG>, (TS*)z, (const TS*)b, (const TG*)U,
                                    (const TG*)A, g, colour, n_mr, nrhs));
  count_launches(1);
  return MG_OK;
}

template <class R, class TS, class TG>
static int run(const Geom& g, void* z, const void* b, const void* U, const void* A, int colour, int n_mr, int nrhs,
               cudaStream_t s) {
  if (cluster_wins<R>(g, nrhs)) return run_cluster<R, TS, TG>(g, z, b, U, A, colour, n_mr, nrhs, s);
  const size_t smem = sizeof(Cplx<R>) * 24 * 256 + sizeof(R) * 8 * 4;
  static bool attr = false;
  if (!attr) {
    SAPMG_CUDA_TRY(cudaFuncSetAttribute(sap_colour_kernel<R, TS, TG>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        (int)smem));
    attr = true;
  }
  sap_colour_kernel<R, TS, TG><<<(unsigned)(g.nblocks / 2 * nrhs), 256, smem, s>>>(
      (TS*)z, (const TS*)b, (const TG*)U, (const TG*)A, g, colour, n_mr, nrhs); count_launches(1);
  SAPMG_CUDA_TRY(cudaGetLastError());
  return MG_OK;
}

int launch_sap_colour(int prec, const Geom& g, void* z, const void* b, const void* U, const void* A, int colour,
                      int n_mr, int nrhs, cudaStream_t s, int pair_shape, int* err) {
  // an even number of FP32-arithmetic right-hand sides goes to the paired
  // kernel (sap2.cu) unless pair_shape < 0
  if (pair_shape >= 0 && prec != P64 && nrhs >= 2 && nrhs % 2 == 0 && n_mr >= 1)
    return launch_sap_colour_pair(prec, g, z, b, U, A, colour, n_mr, nrhs, s, pair_shape, err);
  switch (prec) {
    case P64: return run<double, double2, double2>(g, z, b, U, A, colour, n_mr, nrhs, s);
    case P32: return run<float, float2, float2>(g, z, b, U, A, colour, n_mr, nrhs, s);
    case P16: return run<float, float2, __half2>(g, z, b, U, A, colour, n_mr, nrhs, s);
    case PBF: return run<float, float2, __nv_bfloat162>(g, z, b, U, A, colour, n_mr, nrhs, s);
    default: return MG_ERR_ARG;
  }
}

}  // namespace sapmg
