// Vector kernels of the Krylov solvers, batched over right-hand sides (internal).
#pragma once
#include "internal.h"

namespace sapmg {

// The buffer of a reduction's partial sums: kPartialSums double2 of sums, then
// one arrival counter (unsigned) per right-hand side, zero between kernels
// (whoever allocates the buffer clears it from kPartialSums on).
constexpr size_t kPartialDouble2 = 65536;
constexpr size_t kPartialSums = kPartialDouble2 - 256;

// Geometry of a batched vector operation: R systems, n elements each; the
// vector v_j of system r is at v_j + r*vstride, w of system r at w + r*wstride.
struct BVec {
  size_t n;
  int R;
  size_t vstride;
  size_t wstride;
};
inline BVec bvec(size_t n, int R, size_t stride) { return BVec{n, R, stride, stride}; }

// Per-system complex scalars passed by value (R <= 32).
struct Scal32 { double2 v[32]; };

// out[r*ldo + j] = <v_j[r], w[r]> = sum conj(v_j) w (out2 too if non-null); mode 1 adds into out.
int blas_multidot(int type, const BVec& b, const void* const* v, int k, const void* w, double2* out, int ldo,
                  int mode, double2* out2, double2* partial, cudaStream_t s);
// w[r] += sign * sum_j coeff[r*ldc + j] v_j[r] with device coefficients.
int blas_multiaxpy(int type, const BVec& b, void* w, const void* const* v, int k, const double2* coeff, int ldc,
                   double sign, cudaStream_t s);
// The same, and nrm2[r*ldn] = ||w_new[r]||^2 computed in the same pass.
int blas_multiaxpy_norm(int type, const BVec& b, void* w, const void* const* v, int k, const double2* coeff, int ldc,
                        double sign, double2* nrm2, int ldn, double2* partial, cudaStream_t s);
// y[r] = a_r x[r] + b_r y[r]; element types tx, ty (P64 / P32); b_r = 0: y not read.
int blas_axpby2(int tx, const Scal32& a, const void* x, size_t xs, int ty, const Scal32& b, void* y, size_t ys,
                size_t n, int R, cudaStream_t s);
// out[r] = x[r] / sqrt(nrm2[r*ldn]); store[r*lds] = sqrt(nrm2[r*ldn]) if store != nullptr.
int blas_normalize(int type, const BVec& b, const void* x, void* out, const double2* nrm2, int ldn, double2* store,
                   int lds, cudaStream_t s);
// Work areas of one delayed-reorthogonalisation Arnoldi step (device, each [R][ld]
// double2 except X = [R][4]): dot products A, B, X, pass-2 coefficients c1, c2,
// and the results hcol (Hessenberg column: <v_i, w> for i < j, h_j), acol
// (<v_i, u> for i < j, beta) and nrm (||v_j||^2, ||w_new||^2).
struct DcgsWork {
  double2 *A, *B, *X, *c1, *c2, *hcol, *acol, *nrm;
  int ld;
  double2* partial;
};
// One Arnoldi step with the second Gram-Schmidt pass delayed by one step: u (the
// last basis vector, one pass done) becomes v_j, w (the operator image of the
// step) becomes w - sum_{i<=j} <v_i, w> v_i; v = the j finished basis vectors.
int blas_dcgs2_step(int type, const BVec& b, const void* const* v, int j, void* u, void* w, const DcgsWork& ws,
                    cudaStream_t s);
// The same step (FP32 u and w) with the finished basis vectors stored in FP16,
// scaled by 2^10: vh = v_0 .. v_{j-1}; the new v_j is written to vout in the
// same format only (u's contents are undefined afterwards); u need not be
// normalised.
int blas_dcgs2_step_h(const BVec& b, const void* const* vh, int j, void* u, void* w, void* vout, const DcgsWork& ws,
                      cudaStream_t s);
// out = x / ||x|| stored as an FP16 basis vector (scaled by 2^10).
int blas_normalize_h(const BVec& b, const void* x, void* out, const double2* nrm2, int ldn, double2* store, int lds,
                     cudaStream_t s);
// Scalars of fixed-step GMRES on a coarse level, per right-hand side at stride
// ldr >= 33 * 33: H (column-major, leading dimension 33) and scratch t (33 * 33),
// for blas_hessenberg_solve with norms = t + 64 and pairs for FP32 w.
struct ArnoldiWork {
  double2 *H, *t;
  int ldr;
  double2* partial;
};
// Step j < 32 of the Arnoldi process on w = A v_j (contents undefined
// afterwards): the dots of column j and, unless vnext is null, v_{j+1}, whose norm is near 1.
// basis: P16 (FP16 vectors as blas_normalize_h stores them, FP32 w), P32 or P64.
int blas_arnoldi_step(int basis, const BVec& b, const void* const* v, int j, void* w, void* vnext,
                      const ArnoldiWork& a, cudaStream_t s);
// out[r] = sum_i y[r*ldy + i] v_i[r] (basis as above; out in the precision of w).
int blas_combine(int basis, const BVec& b, const void* const* v, int k, const double2* y, int ldy, void* out,
                 cudaStream_t s);
// y[r] = argmin || sqrt(beta2[r]) e1 - H_r y || for (m+1) x m Hessenberg H_r (column-major, ldh; H_r at H + r*ldr);
// norms, pairs: H and the basis vectors' norms as blas_arnoldi_step leaves them.
int blas_hessenberg_solve(const double2* H, int ldh, int ldr, int m, const double2* beta2, double2* y, int ldy,
                          int R, cudaStream_t s, const double2* norms = nullptr, bool pairs = false);

}  // namespace sapmg
