"""The set-up's FP32 orthonormalisation (Cholesky QR) against the positive-
diagonal QR factor, and its fall-back on dependent vectors: the initial vectors
themselves (no sweep moves them: the smoother's block solves are given no steps)."""

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
