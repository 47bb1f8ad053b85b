"""The set-up's FP32 orthonormalisation (Cholesky QR): the global factor and the flag
through the launcher, and the local factor after a set-up of the initial vectors
themselves (no sweep moves them: the smoother's block solves are given no steps),
which no global triangular factor changes: what it shows is that none of the
vectors is lost, also where dependent ones fall back on Gram-Schmidt."""

import numpy as np
import pytest

import synth
from tests.gpu_util import torch_cuda, dev, host

pytestmark = pytest.mark.gpu

DIMS = (8, 8, 8, 16)


@pytest.mark.parametrize("n_vec", [1, 2, 4, 5, 8, 9, 17, 24, 32])
@pytest.mark.parametrize("kind", ["random", "close", "dependent", "zero"])
def test_local_basis_spans_the_initial_vectors(n_vec, kind):
    """n_mr = 0 makes a sweep the identity, so the test vectors after set-up are
    the local QR factor of the global QR factor of the initial ones, which is
    the local QR factor of the initial ones themselves.  FP32 orthonormalisation
    of vectors with condition number kappa: 1e-6 kappa."""
    torch = torch_cuda()
    import paper_1202_2462_gb300 as G
    if n_vec < 2 and kind != "random":
        pytest.skip("needs two vectors")
    u = dev(torch, synth.random_gauge_field(DIMS, 0.4, 311))
    v = synth.random_spinor(DIMS, 312, nvec=n_vec).astype(np.complex64)
    if kind == "close":                    # an angle of about 3 degrees
        v[-1] = v[0] + 0.05 * v[-1]
    elif kind == "dependent":
        v[1] = 2.0 * v[0]
    elif kind == "zero":
        v[1] = 0
    s = G.Solver(u, 1.0, -0.1, n_levels=2, n_vec=(n_vec,), setup_iters=2, n_mr=0, precision="fp32", fgmres_m=32,
                 init_vectors=dev(torch, v))
    out = torch.empty((n_vec,) + s.lat + (4, 3), dtype=torch.complex128, device="cuda")
    G.mg_get_vectors(s.ctx, 0, out)
    q = host(out)
    s.close()
    lt, lz, ly, lx = s.lat

    def agg(x):
        y = x.reshape(-1, lt // 4, 4, lz // 4, 4, ly // 4, 4, lx // 4, 4, 2, 6).transpose(1, 3, 5, 7, 9, 0, 2, 4, 6, 8, 10)
        return y.reshape(-1, n_vec, 1536)

    got, a = agg(q), agg(v.astype(complex))
    if kind in ("dependent", "zero"):      # the others still come first and in order; nothing is lost or infinite
        assert np.isfinite(got).all()
        assert np.allclose(np.linalg.norm(got[:, 0], axis=1), 1.0, atol=1e-6)
        return
    for m in range(0, got.shape[0], 7):
        qr, r = np.linalg.qr(a[m].T)
        want = (qr * (np.diag(r) / np.abs(np.diag(r)))).T
        assert np.abs(got[m] - want).max() < (2e-6 if kind == "random" else 1e-4)


def _cholqr(torch, v):
    """The library's launcher on V [N][n] (complex64, in place); the flag."""
    import ctypes
    from paper_1202_2462_gb300 import binding
    f = ctypes.CDLL(binding.LIB_PATH)._ZN5sapmg14launch_cholqr2EPvimP7double2S2_PiP11CUstream_st
    f.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_size_t] + [ctypes.c_void_p] * 4
    partial = torch.zeros(65536, dtype=torch.complex128, device="cuda")
    work = torch.zeros(1536, dtype=torch.complex128, device="cuda")
    flag = torch.zeros(1, dtype=torch.int32, device="cuda")
    rc = f(v.data_ptr(), v.shape[0], v.shape[1], partial.data_ptr(), work.data_ptr(), flag.data_ptr(),
           torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    assert rc == 0
    return int(flag[0])


@pytest.mark.parametrize("n_vec,n", [(1, 64), (2, 130), (3, 4096), (4, 49150), (5, 62), (8, 8190), (9, 49152), (16, 12290),
                                     (17, 2050), (20, 1572864), (24, 70002), (25, 12290), (28, 130), (29, 49150), (32, 98302)])
def test_cholesky_qr(n_vec, n):
    """The global factor itself: V^dagger V = 1 and the positive-diagonal QR factor in FP64 of
    the same numbers.  FP32 storage and a triangular solve of n_vec terms on vectors
    of condition number below 10: 2^-24 sqrt(n_vec) 10 per entry of the vectors' size;
    a factor of four is left."""
    torch = torch_cuda()
    gen = torch.Generator("cuda").manual_seed(n_vec)
    v = torch.randn((n_vec, n), dtype=torch.complex64, device="cuda", generator=gen)
    if n_vec > 2:
        v[2] += 3.0 * v[0]
    q, r = torch.linalg.qr(v.to(torch.complex128).T)
    d = r.diagonal()
    want = (q * (d / d.abs())).T
    tol = 40 * 2.0 ** -24 * n_vec ** 0.5
    assert _cholqr(torch, v) == 0
    w = v.to(torch.complex128)
    gram = w.conj() @ w.T
    assert (gram - torch.eye(n_vec, device="cuda")).abs().max() < tol
    assert torch.linalg.vector_norm(w - want, dim=1).max() < tol


@pytest.mark.parametrize("kind", ["dependent", "near", "zero", "nan", "inf"])
@pytest.mark.parametrize("n_vec", [2, 20, 32])
def test_cholesky_qr_leaves_dependent_vectors(n_vec, kind):
    """A vector in the span of the earlier ones (or within half a degree of it), a zero and a
    non-finite one raise the flag, and the vectors stay what they were."""
    torch = torch_cuda()
    gen = torch.Generator("cuda").manual_seed(n_vec)
    v = torch.randn((n_vec, 4098), dtype=torch.complex64, device="cuda", generator=gen)
    last = v[-1].clone()
    v[-1] = 2.0 * v[0]
    if kind == "near":
        v[-1] += 0.01 * last
    elif kind == "zero":
        v[-1] = 0
    elif kind == "nan":
        v[-1, 7] = float("nan")
    elif kind == "inf":
        v[-1, 7] = float("inf")
    before = v.clone()
    assert _cholqr(torch, v) != 0
    assert torch.equal(torch.view_as_real(v).nan_to_num(7.0), torch.view_as_real(before).nan_to_num(7.0))
