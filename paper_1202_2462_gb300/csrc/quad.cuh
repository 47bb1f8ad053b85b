// D at a site shared by four threads, for lattices with few blocks: warp m of a
// four-warp CTA forms the two hops of direction m at the CTA's 32 sites, the
// partial sums are swapped through shared memory, and each warp ends up with
// three spin-colour components, those whose clover rows it applies.
//
// One SM sub-partition issues an FP64 instruction of a warp every 64 cycles, so
// with a warp per 32 sites the 1130 FP64 instructions of a site take 36 us
// however few warps there are; four warps of 280 each take a quarter of that
// as long as there are sub-partitions for them (608 on the chip).
#pragma once
#include "stencil.cuh"

namespace sapmg {

// The two hops of direction MU at (blk, loc), neighbours through ld(step, component): the sum
// over both of (1 -+ gamma) U psi.  keep(step): whether the hop is inside.
template <int MU, class R, class TG, bool DAG, class LD, class KEEP>
__device__ __forceinline__ void quad_hops(const Geom& g, const TG* __restrict__ U, int blk, int loc, LD ld, KEEP keep,
                                          Cplx<R> (&acc)[12]) {
  constexpr int SF = DAG ? 1 : -1;
  Cplx<R> h[6], gg[6], u[9];
  if (keep(1)) {
    spin_project_ld<MU, SF, R>([&](int c) { return ld(1, c); }, h);
    load_link<R>(U, blk, MU, loc, u);
    su3_mul(u, h, gg);
    spin_reconstruct_add<MU, SF, R, kSet>(gg, acc);
  } else {
#pragma unroll
    for (int c = 0; c < 12; ++c) acc[c] = cmk<R>(0, 0);
  }
  if (keep(-1)) {
    int nb, nl;
    neighbour(g, blk, loc, MU, -1, nb, nl);
    spin_project_ld<MU, -SF, R>([&](int c) { return ld(-1, c); }, h);
    load_link<R>(U, nb, MU, nl, u);
    su3_dag_mul(u, h, gg);
    spin_reconstruct_add<MU, -SF>(gg, acc);
  }
}

// Rows 3 M .. 3 M + 2 of A psi, psi's components of that chirality through ld(component).
template <int M, class R, class TG, class LD>
__device__ __forceinline__ void quad_clover(const TG* __restrict__ A, int blk, int loc, LD ld, Cplx<R> (&out)[3]) {
  constexpr int chi = M >> 1, i0 = 3 * (M & 1);
  const TG* a = A + ((size_t)(blk * 36 + chi * 18)) * 256 + loc;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    constexpr int base = chi * 6;
    const int i = i0 + k;
    const Cplx<R> d = Io<R, TG>::ld(a + (i >> 1) * 256);
    out[k] = ((i & 1) ? d.im : d.re) * ld(base + i);
#pragma unroll
    for (int j = 0; j < 6; ++j) {
      if (j == i) continue;
      const Cplx<R> o = Io<R, TG>::ld(a + (3 + (i < j ? offdiag_index(i, j) : offdiag_index(j, i))) * 256);
      if (i < j) cfma(out[k], o, ld(base + j));
      else cfma_conj(out[k], o, ld(base + j));
    }
  }
}

// out = rows 3 M .. 3 M + 2 of D psi at the warp's sites: part [4][12][32] in
// shared memory takes the warps' hop sums (a CTA barrier inside).
template <int M, class R>
__device__ __forceinline__ void quad_swap(Cplx<R>* part, int lane, const Cplx<R> (&acc)[12], Cplx<R> (&out)[3]) {
#pragma unroll
  for (int c = 0; c < 12; ++c) part[(M * 12 + c) * 32 + lane] = acc[c];
  __syncthreads();
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const Cplx<R>* q = part + (3 * M + k) * 32 + lane;
    const Cplx<R> t = (q[0] + q[12 * 32]) + (q[24 * 32] + q[36 * 32]);
    out[k] = out[k] - (R)0.5 * t;
  }
}

// D psi with neighbours and fields from global memory (psi in storage TS).
template <int M, class R, class TS, class TG, bool DAG>
__device__ __forceinline__ void quad_dirac(const Geom& g, const TS* __restrict__ f, const TG* __restrict__ U,
                                           const TG* __restrict__ A, int blk, int loc, int lane, Cplx<R>* part,
                                           Cplx<R> (&out)[3]) {
  Cplx<R> acc[12];
  int nb[2], nl[2];
  neighbour(g, blk, loc, M, 1, nb[0], nl[0]);
  neighbour(g, blk, loc, M, -1, nb[1], nl[1]);
  const TS* q0 = f + (size_t)nb[0] * 12 * 256 + nl[0];
  const TS* q1 = f + (size_t)nb[1] * 12 * 256 + nl[1];
  quad_hops<M, R, TG, DAG>(g, U, blk, loc, [&](int step, int c) { return Io<R, TS>::ldc((step > 0 ? q0 : q1) + c * 256); },
                           [](int) { return true; }, acc);
  const TS* own = f + (size_t)blk * 12 * 256 + loc;
  quad_clover<M, R>(A, blk, loc, [&](int c) { return Io<R, TS>::ldc(own + c * 256); }, out);
  quad_swap<M>(part, lane, acc, out);
}

}  // namespace sapmg
