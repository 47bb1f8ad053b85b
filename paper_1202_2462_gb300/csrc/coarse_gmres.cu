// Fixed-step GMRES on a small coarse lattice (Sec. 4) in one kernel: a cluster of
// sixteen CTAs per right-hand side keeps the operator rows of its sites / 16
// sites, the Krylov basis and every scalar in shared memory for the whole solve.
//
// A lattice of 32 sites (the coarsest level of 16^3 x 32 on three levels) has 1280
// unknowns: its three kernels a step (operator, dots, update) took 27 us of
// launches, L2 round trips and one-warp reductions for about a microsecond of
// work.  Here a step has two exchanges through distributed shared memory, each
// one cluster barrier: the CTAs' partial dots, and the new basis vector with its
// partial norm.  Every CTA adds the sixteen parts in the same order, so all hold
// the same scalars and the result does not depend on scheduling.
//
// Per step, as the two-kernel form of the coarse GMRES (blas.cu): h_i = <v_i, w>,
// beta^2 = <w, w> - sum |h_i|^2 / |v_i|^2 (floored), v_{j+1} = (w - sum h_i v_i /
// |v_i|^2) / beta, whose exact norm s_{j+1} is kept: with rows h_ij / s_i and the
// subdiagonal ||x|| the least squares gives the coefficients of the v_i as they are.
#include "accum.cuh"
#include "cluster.cuh"
#include "coarse.h"
#include "hessenberg.cuh"
#include "internal.h"

namespace sapmg {
namespace {

constexpr int kSolveCluster = 16;

// operator entries: FP16 pairs with FP32 arithmetic, or FP64
struct HalfOp {
  typedef float R;
  typedef uint32_t M;
  static constexpr float kFloor = 1e-6f;
  static __device__ __forceinline__ Cplx<float> get(uint32_t m) {
    const float2 v = half2_bits_to_float2(m);
    return cmk(v.x, v.y);
  }
};
struct DoubleOp {
  typedef double R;
  typedef double2 M;
  static constexpr double kFloor = 1e-14;
  static __device__ __forceinline__ Cplx<double> get(double2 m) { return cmk(m.x, m.y); }
};

// Sum of one value over lanes 0..15 in a fixed order.
template <class R> __device__ __forceinline__ Acc<R> sum16(Acc<R> v) {
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) v.add(v.from(o));
  return v;
}
__device__ __forceinline__ void cluster_st_acc(uint32_t a, Acc<float> v) { cluster_st(a, cmk(v.h, v.l)); }
__device__ __forceinline__ void cluster_st_acc(uint32_t a, Acc<double> v) { cluster_st(a, v.v); }
__device__ __forceinline__ float rsqrt_of(float x) { return rsqrtf(x); }
__device__ __forceinline__ double rsqrt_of(double x) { return rsqrt(x); }

struct Layout {          // byte offsets in shared memory
  int ms, vf, basis, ts, w, pd, pn, hr, hi, coef, dots, sc, tab, flag, bar, total;
};
template <class OP>
__host__ __device__ inline Layout layout(int spc, int nsites, int n2, int k) {
  const int cb = 2 * (int)sizeof(typename OP::R), rows = spc * n2;
  Layout l;
  int o = 0;
  auto take = [&](int bytes) { const int at = o; o += (bytes + 15) & ~15; return at; };
  l.ms = take(spc * 9 * n2 * n2 * (int)sizeof(typename OP::M));
  l.vf = take(2 * nsites * n2 * cb);                       // the current basis vector, two buffers
  l.basis = take(k * rows * cb);                           // the CTA's rows of v_0 .. v_{k-1}
  l.ts = take(spc * 9 * n2 * cb);
  l.w = take(rows * cb);
  l.pd = take(kSolveCluster * 33 * cb);                    // partial dots [rank][33]
  l.pn = take(2 * kSolveCluster * 8);                      // partial norms (Acc), two buffers
  l.hr = take(33 * 32 * 8);
  l.hi = take(33 * 32 * 8);
  l.coef = take(34 * 16);                                  // y (FP64)
  l.dots = take(34 * cb);                                  // <v_i, w> / |v_i|^2
  l.sc = take(34 * 8 * 3);                                 // 1/s_i (FP64), 1/s_i^2 (Scale), |<v_i, w>|^2 / |v_i|^2
  l.tab = take(spc * 9 * 4);
  l.flag = take(kSolveCluster * 4);
  l.bar = take(8);
  l.total = o;
  return l;
}

// N2 > 0: 2N at compile time.  The last warp, beyond those of the products, turns
// sums into H's column and the norms' reciprocals (FP64, 64 cycles an instruction)
// while the others are at the next product.
template <class OP, class TX, int N2>
__global__ void __launch_bounds__(768) coarse_gmres_cluster_kernel(const typename OP::M* __restrict__ M,
                                                                   const TX* __restrict__ b, TX* __restrict__ x,
                                                                   CGeom c, int spc, int k, int* __restrict__ err) {
  typedef typename OP::R R;
  typedef typename OP::M TM;
  typedef Cplx<R> C;
  extern __shared__ __align__(128) unsigned char smem[];
  const int n2 = N2 > 0 ? N2 : c.n2, tile = n2 * n2, rank = cluster_rank(), rows = spc * n2, n = c.nsites * n2;
  const Layout lo = layout<OP>(spc, c.nsites, n2, k);
  TM* Ms = reinterpret_cast<TM*>(smem + lo.ms);
  C* vf = reinterpret_cast<C*>(smem + lo.vf);
  C* basis = reinterpret_cast<C*>(smem + lo.basis);
  C* ts = reinterpret_cast<C*>(smem + lo.ts);
  C* w = reinterpret_cast<C*>(smem + lo.w);
  C* pd = reinterpret_cast<C*>(smem + lo.pd);
  Acc<R>* pn = reinterpret_cast<Acc<R>*>(smem + lo.pn);
  double* hr = reinterpret_cast<double*>(smem + lo.hr);
  double* hi = reinterpret_cast<double*>(smem + lo.hi);
  double2* coef = reinterpret_cast<double2*>(smem + lo.coef);
  double* is = reinterpret_cast<double*>(smem + lo.sc);       // 1 / s_i
  Scale<R>* is2 = reinterpret_cast<Scale<R>*>(is + 34);       // 1 / s_i^2
  R* part2 = reinterpret_cast<R*>(is + 68);                   // what <w, w> loses to v_i
  C* dots = reinterpret_cast<C*>(smem + lo.dots);
  int* tab = reinterpret_cast<int*>(smem + lo.tab);
  int* flag = reinterpret_cast<int*>(smem + lo.flag);
  uint64_t* bar = reinterpret_cast<uint64_t*>(smem + lo.bar);
  const int tid = threadIdx.x, nt = blockDim.x, warp = tid >> 5, lane = tid & 31, nw = nt >> 5;
  const int s0 = rank * spc, ns = max(0, min(spc, c.nsites - s0)), nr = ns * n2;   // this CTA's sites and rows
  const size_t rhs = (size_t)(blockIdx.x / kSolveCluster) * n;
  b += rhs;
  x += rhs;
  if (tid == 0) {
    mbar_init(bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    if (ns > 0) {
      mbar_expect_tx(bar, (uint32_t)(ns * 9 * tile * (int)sizeof(TM)));
      for (int q = 0; q < ns; ++q)
        bulk_copy_g2s(Ms + (size_t)q * 9 * tile, M + (size_t)(s0 + q) * 9 * tile, (uint32_t)(9 * tile * (int)sizeof(TM)),
                      bar);
    }
  }
  for (int q = tid; q < ns * 9; q += nt) {
    const int site = s0 + q / 9, d = q % 9;
    int nb = site;
    if (d > 0) {
      const int mu = (d - 1) >> 1, step = (d & 1) ? 1 : -1;
      int stride = 1, L = 1;
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        if (m < mu) stride *= c.L[m];
        if (m == mu) L = c.L[m];
      }
      const int xc = (site / stride) % L;
      nb = MG_CLAMP(kCoarseNeighbour, site + ((xc + step + L) % L - xc) * stride, c.nsites);
    }
    tab[q] = nb * n2;
  }
  for (int q = tid; q < 33 * k; q += nt) hr[q] = hi[q] = 0.0;
  const int spins = wait_spins(err);
  cluster_barrier();                                         // every CTA of the cluster runs
  // ||b||: the warps' parts are added in warp order, the CTAs' by sum16
  __shared__ R part[24];
  auto all_norm = [&](R v, int buf) {                        // this thread's |.|^2 to every CTA's pn[buf][rank]
    v = warp_sum(v);
    if (lane == 0) part[warp] = v;
    __syncthreads();
    if (tid < kSolveCluster) {
      Acc<R> t = Acc<R>::of((R)0);
      for (int q = 0; q < (nr + 31) / 32 && q < nw; ++q) t.add(Acc<R>::of(part[q]));
      cluster_st_acc(cluster_addr(smem_u32(pn + buf * kSolveCluster + rank), tid), t);
    }
  };
  const uint32_t vf_a = smem_u32(vf), pd_a = smem_u32(pd);
  {
    R v = 0;
    for (int e = tid; e < nr; e += nt) {
      const C t = Io<R, TX>::ldc(b + (size_t)s0 * n2 + e);
      w[e] = t;
      v += t.re * t.re + t.im * t.im;
    }
    all_norm(v, 1);
  }
  const bool waited = ns > 0 ? mbar_wait(bar, 0, spins) : true;
  const int failed = __syncthreads_or(!waited);
  if (tid < kSolveCluster) cluster_st(cluster_addr(smem_u32(flag + rank), tid), failed);
  cluster_barrier();
  {
    int any = 0;
    for (int q = 0; q < kSolveCluster; ++q) any |= flag[q];
    if (any) {                                               // the same decision in all sixteen CTAs
      if (tid == 0) {
        if (failed) {
          atomicExch(err, 1);
          mbar_wait(bar, 0);                                 // let the copies in flight land
        }
      }
      __syncthreads();
      return;
    }
  }
  const double bb = sum16<R>(pn[kSolveCluster + (lane & 15)]).exact();
  const double beta0 = sqrt(fmax(bb, 0.0));
  {
    const R f = beta0 > 0.0 ? (R)(1.0 / beta0) : (R)0;
    for (int e = tid; e < nr; e += nt) {
      const C v = f * w[e];
      basis[e] = v;
      const uint32_t a = vf_a + (uint32_t)((s0 * n2 + e) * sizeof(C));
#pragma unroll
      for (int q = 0; q < kSolveCluster; ++q) cluster_st(cluster_addr(a, q), v);
    }
  }
  if (tid == 0) { is[0] = 1.0; is2[0] = Scale<R>::one(); }
  cluster_barrier();
  for (int j = 0; j < k; ++j) {
    // w = A v_j on the CTA's rows
    const C* vj = vf + (j & 1) * n;
    for (int e = tid; e < ns * 9 * n2; e += nt) {
      const int q = e / n2, row = e - q * n2;
      const TM* m = Ms + (size_t)q * tile + row;
      const C* xv = vj + tab[q];
      C t = cmk<R>(0, 0);
#pragma unroll 8
      for (int i = 0; i < n2; ++i) cfma(t, OP::get(m[i * n2]), xv[i]);
      ts[e] = t;
    }
    __syncthreads();
    for (int e = tid; e < nr; e += nt) {
      const int q = e / n2, row = e - q * n2;
      C t = ts[q * 9 * n2 + row];
#pragma unroll
      for (int d = 1; d < 9; ++d) t = t + ts[(q * 9 + d) * n2 + row];
      w[e] = t;
    }
    __syncthreads();
    // partial dots: value i <= j is <v_i, w>, value j + 1 is <w, w>
    for (int i = warp; i <= j + 1; i += nw) {
      const C* vi = i <= j ? basis + i * rows : w;
      C t = cmk<R>(0, 0);
      for (int e = lane; e < nr; e += 32) cfma_conj(t, vi[e], w[e]);
      t = cmk(warp_sum(t.re), warp_sum(t.im));
      if (lane < kSolveCluster) cluster_st(cluster_addr(pd_a + (uint32_t)((rank * 33 + i) * sizeof(C)), lane), t);
    }
    cluster_barrier();
    for (int i = warp; i <= j + 1; i += nw) {
      const C t = pd[(lane & 15) * 33 + i];
      const Acc<R> a = sum16(Acc<R>::of(t.re)), c2 = sum16(Acc<R>::of(t.im));
      if (lane == 0) {
        if (i <= j) {
          const Scale<R> f = is2[i];
          dots[i] = cmk(f.times(a), f.times(c2));
          part2[i] = dots[i].re * a.value() + dots[i].im * c2.value();
          hr[i + 33 * j] = a.exact();                        // raw; scaled by the last warp
          hi[i + 33 * j] = c2.exact();
        } else {
          part2[i] = a.value();                              // <w, w>
        }
      }
    }
    __syncthreads();
    // x = w - sum h_i v_i / |v_i|^2, v_{j+1} = x / beta
    R invb = 0, nn = 0;
    if (tid < nr || warp == nw - 1) {
      R e2 = 0;
      for (int i = 0; i <= j; ++i) e2 += part2[i];
      const R ww = part2[j + 1];
      const R d2 = max(ww - e2, OP::kFloor * ww);
      invb = d2 > (R)0 ? rsqrt_of(d2) : (R)0;
    }
    for (int e = tid; e < nr; e += nt) {
      C t = w[e];
      for (int i = 0; i <= j; ++i) cfma(t, cmk(-dots[i].re, -dots[i].im), basis[i * rows + e]);
      nn += t.re * t.re + t.im * t.im;
      if (j + 1 < k) {
        const C v = invb * t;
        basis[(j + 1) * rows + e] = v;
        const uint32_t a = vf_a + (uint32_t)((((j + 1) & 1) * n + s0 * n2 + e) * sizeof(C));
#pragma unroll
        for (int q = 0; q < kSolveCluster; ++q) cluster_st(cluster_addr(a, q), v);
      }
    }
    all_norm(nn, j & 1);
    cluster_barrier();
    if (warp == nw - 1) {                                    // while the others start the next product
      const Acc<R> q = sum16<R>(pn[(j & 1) * kSolveCluster + (lane & 15)]);
      if (lane == 0) is2[j + 1] = Scale<R>::of(q, invb);
      const double nrm = sqrt(fmax(q.exact(), 0.0));
      if (lane <= j) {
        hr[lane + 33 * j] *= is[lane];
        hi[lane + 33 * j] *= is[lane];
      }
      __syncwarp();
      if (lane == 0) {
        hr[j + 1 + 33 * j] = nrm;
        const double sc = nrm * (double)invb;
        is[j + 1] = sc > 0.0 ? 1.0 / sc : 0.0;
      }
    }
    // is2[j + 1] is first read after the barriers of the next step's products
  }
  __syncthreads();
  if (warp == 0) {
    const unsigned zero = __ballot_sync(0xffffffffu, lane < k && hr[min(lane, k - 1) + 1 + 33 * min(lane, k - 1)] == 0.0);
    const int mm = zero ? __ffs(zero) : k;                   // columns up to the first zero subdiagonal entry
    const Cplx<double> y = beta0 > 0.0 ? hessenberg_warp(hr, hi, mm, beta0) : cmk(0.0, 0.0);
    if (lane < k) coef[lane] = lane < mm ? make_double2(y.re, y.im) : make_double2(0, 0);
  }
  __syncthreads();
  for (int e = tid; e < nr; e += nt) {
    C t = cmk<R>(0, 0);
    for (int i = 0; i < k; ++i) cfma(t, cmk((R)coef[i].x, (R)coef[i].y), basis[i * rows + e]);
    Io<R, TX>::st(x + (size_t)s0 * n2 + e, t);
  }
}

// Whether the cluster form holds a system of this size on the current device
// (sixteen CTAs are more than the portable cluster; asked once per process).
template <class OP, class TX, int N2>
bool device_takes_cluster() {
  static const bool ok = [] {
    if (cudaFuncSetAttribute(coarse_gmres_cluster_kernel<OP, TX, N2>, cudaFuncAttributeNonPortableClusterSizeAllowed,
                             1) != cudaSuccess ||
        cudaFuncSetAttribute(coarse_gmres_cluster_kernel<OP, TX, N2>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             227 * 1024 - 256) != cudaSuccess) {
      cudaGetLastError();
      return false;
    }
    ClusterLaunch l(kSolveCluster, 768, 220 * 1024, kSolveCluster, nullptr);
    int nclusters = 0;
    if (cudaOccupancyMaxActiveClusters(&nclusters, coarse_gmres_cluster_kernel<OP, TX, N2>, &l.cfg) != cudaSuccess) {
      cudaGetLastError();
      return false;
    }
    return nclusters > 0;
  }();
  return ok;
}

template <class OP>
bool fits(const CGeom& c, int k) {
  const int spc = (c.nsites + kSolveCluster - 1) / kSolveCluster;
  return c.n2 % 2 == 0 && c.n2 <= 64 && spc <= 4 && k <= 32 && layout<OP>(spc, c.nsites, c.n2, k).total <= 220 * 1024;
}

template <class OP, class TX, int N2>
int run(const CGeom& c, const void* M, const void* b, void* x, int k, int R, int* err, cudaStream_t s) {
  const int spc = (c.nsites + kSolveCluster - 1) / kSolveCluster;
  const int threads = std::min(768, std::max(96, (spc * 9 * c.n2 + 31) / 32 * 32) + 32);
  ClusterLaunch l((unsigned)(R * kSolveCluster), (unsigned)threads, (size_t)layout<OP>(spc, c.nsites, c.n2, k).total,
                  kSolveCluster, s);
  SAPMG_CUDA_TRY(cudaLaunchKernelEx(&l.cfg, coarse_gmres_cluster_kernel<OP, TX, N2>, (const typename OP::M*)M,
                                    (const TX*)b, (TX*)x, c, spc, k, err));
  count_launches(1);
  return MG_OK;
}

}  // namespace

bool coarse_gmres_cluster_ok(int store, const CGeom& c, int k) {
  if (store == P16)
    return fits<HalfOp>(c, k) &&
           (c.n2 == 40 ? device_takes_cluster<HalfOp, float2, 40>() : device_takes_cluster<HalfOp, float2, 0>());
  if (store == P64) return fits<DoubleOp>(c, k) && device_takes_cluster<DoubleOp, double2, 0>();
  return false;
}

int launch_coarse_gmres_cluster(int store, const CGeom& c, const void* M, const void* b, void* x, int k, int R,
                                int* err, cudaStream_t s) {
  if (store == P16)
    return c.n2 == 40 ? run<HalfOp, float2, 40>(c, M, b, x, k, R, err, s)
                      : run<HalfOp, float2, 0>(c, M, b, x, k, R, err, s);
  if (store == P64) return run<DoubleOp, double2, 0>(c, M, b, x, k, R, err, s);
  return MG_ERR_ARG;
}

}  // namespace sapmg
