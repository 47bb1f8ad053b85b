"""The launch forms for few blocks (D with four threads a site, a cluster of CTAs
per Schwarz block) against the forms that the same call takes for many: the same
fields once alone and once in a batch that is large enough for the other form;
and the fixed-step coarse GMRES in all its forms against the minimiser."""

import numpy as np
import pytest

import synth
from tests.gpu_util import torch_cuda, dev, host, rel

pytestmark = pytest.mark.gpu

DIMS = (8, 8, 8, 8)      # 16 blocks, 8 of a colour


def _solver(prec, **kw):
    torch = torch_cuda()
    import paper_1202_2462_gb300 as G
    u = dev(torch, synth.random_gauge_field(DIMS, 0.4, 301))
    return torch, G, G.Solver(u, 1.0, -0.1, precision=prec, **kw)


# 1216 / 16 = 76 fields (FP64) and 10 fields (FP32) reach the whole-block form of D; 608 / 8 = 76 and 19 that of
# the Schwarz pass (an odd count: an even one of FP32 fields goes to the paired kernel).  The two forms add the
# same terms in another order: a few roundings of sums of about 100 terms.
@pytest.mark.parametrize("prec,many,tol", [("fp64", 77, 1e-15), ("fp32", 11, 5e-7), ("bf16", 11, 5e-7)])
def test_dirac_four_threads_a_site(prec, many, tol):
    torch, G, s = _solver(prec, n_levels=1, fgmres_m=1)
    dt = torch.complex128 if prec == "fp64" else torch.complex64
    x = torch.randn((many, 16, 12, 256), dtype=dt, device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    for flag in (0, G.MG_DAGGER) if prec != "bf16" else (0,):
        a, one = torch.empty_like(x), torch.empty_like(x[:1])
        G.dirac_apply(s.ctx, x, a, s.prec | G.MG_BLOCKED | flag, many)
        for k in (0, many - 1):
            G.dirac_apply(s.ctx, x[k:k + 1].contiguous(), one, s.prec | G.MG_BLOCKED | flag, 1)
            assert rel(host(a[k]), host(one[0])) < tol
    s.close()


@pytest.mark.parametrize("prec,many,tol", [("fp64", 77, 1e-14), ("fp32", 19, 5e-6), ("bf16", 19, 5e-6)])
@pytest.mark.parametrize("n_mr", [0, 1, 4])
def test_schwarz_cluster(prec, many, tol, n_mr):
    torch, G, s = _solver(prec, n_levels=1, fgmres_m=1, n_mr=n_mr)
    dt = torch.complex128 if prec == "fp64" else torch.complex64
    gen = torch.Generator("cuda").manual_seed(2)
    b = torch.randn((many, 16, 12, 256), dtype=dt, device="cuda", generator=gen)
    z = torch.randn((many, 16, 12, 256), dtype=dt, device="cuda", generator=gen)
    b[1], z[1] = 0, 0                                    # a zero system
    a = z.clone()
    G.sap_smooth(s.ctx, b, a, 2, s.prec | G.MG_BLOCKED, many)
    for k in (0, 1, many - 1):
        one = z[k:k + 1].clone()
        G.sap_smooth(s.ctx, b[k:k + 1].contiguous(), one, 2, s.prec | G.MG_BLOCKED, 1)
        if k == 1:
            assert torch.count_nonzero(one) == 0 and torch.count_nonzero(a[1]) == 0
        else:
            assert rel(host(a[k]), host(one[0])) < tol
    s.close()


@pytest.mark.parametrize("n_vec,nrhs", [(4, 1), (20, 1), (20, 3), (24, 12)])
def test_level1_schwarz_cluster_matches_one_cta_per_box(n_vec, nrhs, monkeypatch):
    """Level-1 boxes of 2^4 sites: the cluster form gives the one-CTA-per-box solve bit for bit."""
    torch = torch_cuda()
    import paper_1202_2462_gb300 as G
    dims = (16, 16, 16, 16)
    u = dev(torch, synth.random_gauge_field(dims, 0.4, 191))
    b = dev(torch, synth.random_spinor(dims, 192, nvec=nrhs))
    out = {}
    for flag in ("0", "1"):
        monkeypatch.setenv("SAPMG_COARSE_SAP_MRHS", flag)
        s = G.Solver(u, 1.0, -0.1, n_levels=3, n_vec=(n_vec, 4), setup_iters=2, precision="bf16", nrhs_max=nrhs,
                     seed=7, coarse_iters=8, fgmres_m=10, inner_iters=3)
        z, info, code = s.solve(b)
        s.close()
        assert code == 0
        out[flag] = (z, info.iterations)
    assert torch.equal(out["0"][0], out["1"][0]) and out["0"][1] == out["1"][1]


# 16 coarse sites: the one-kernel form; 128: a kernel for the dots and one for the
# update a step, with the basis in FP64, FP32 ("fp32") and FP16 ("fp16")
@pytest.mark.parametrize("dims,prec,tol", [
    (DIMS, "fp64", 1e-13), (DIMS, "fp32", 1e-3), (DIMS, "fp16", 1e-3),
    ((16, 8, 16, 16), "fp64", 1e-13), ((16, 8, 16, 16), "fp32", 1e-3), ((16, 8, 16, 16), "fp16", 4e-3)])
@pytest.mark.parametrize("iters", [1, 4, 5, 8, 9, 16, 17, 32])
def test_coarse_gmres_minimises(dims, prec, tol, iters, monkeypatch):
    """The fixed-step coarse solve against the least-squares minimiser over the
    Krylov space, at the step counts where its kernels change size: the norms
    of the two residuals, relative to the source's (the mixed form applies an
    FP16 operator, entries rounded by up to 5e-4, so its residual under the FP64
    operator is off by that much; an FP16 basis adds roundings of 2^-11 of up to
    32 vectors; 1e-13 is FP64 rounding times 256 terms).  On 16 sites the longest
    runs go on after the Krylov space is exhausted."""
    torch = torch_cuda()
    import paper_1202_2462_gb300 as G
    if prec == "fp32":
        monkeypatch.setenv("SAPMG_COARSE_BASIS_FP16", "0")
    u = dev(torch, synth.random_gauge_field(dims, 0.4, 301))
    s = G.Solver(u, 1.0, -0.1, precision=prec, n_levels=2, n_vec=(8,), setup_iters=2, coarse_iters=iters, seed=3)
    lat = [d // 4 for d in dims]
    nb, n2 = int(np.prod(lat)), 16
    m = torch.empty((nb, 9, n2, n2), dtype=torch.complex128, device="cuda")
    G.mg_get_coarse_op(s.ctx, 1, m)
    mh = host(m)
    nbr = np.zeros((nb, 9), dtype=int)
    for a in range(nb):
        x = list(np.unravel_index(a, lat, order="F"))
        nbr[a, 0] = a
        for mu in range(4):
            for step, d in ((1, 1 + 2 * mu), (-1, 2 + 2 * mu)):
                y = list(x)
                y[mu] = (y[mu] + step) % lat[mu]
                nbr[a, d] = np.ravel_multi_index(y, lat, order="F")
    dense = np.zeros((nb * n2, nb * n2), dtype=complex)
    for a in range(nb):
        for d in range(9):
            dense[a * n2:(a + 1) * n2, nbr[a, d] * n2:(nbr[a, d] + 1) * n2] += mh[a, d]
    rng = np.random.default_rng(5)
    b = rng.normal(size=nb * n2) + 1j * rng.normal(size=nb * n2)
    dt = torch.complex128 if prec == "fp64" else torch.complex64
    bd = dev(torch, b, dt)
    x = torch.empty_like(bd)
    G.mg_coarse_solve(s.ctx, 1, bd, x, s.prec)
    q = [b / np.linalg.norm(b)]
    for _ in range(iters - 1):
        w = dense @ q[-1]
        for _ in range(2):
            for v in q:
                w = w - np.vdot(v, w) * v
        q.append(w / np.linalg.norm(w))
    aq = dense @ np.array(q).T
    y = np.linalg.lstsq(aq, b, rcond=None)[0]
    want = np.linalg.norm(b - aq @ y)
    got = np.linalg.norm(b - dense @ host(x).reshape(-1))
    assert abs(got - want) <= tol * np.linalg.norm(b)
    G.mg_coarse_solve(s.ctx, 1, torch.zeros_like(bd), x, s.prec)
    assert torch.count_nonzero(x) == 0
    s.close()
