"""The solver's vector kernels and layout changes at the sizes where they change form."""

import numpy as np
import pytest

import synth
from oracle.aggregation import Aggregation
from tests.gpu_util import dev, emax, host, rel, round_storage, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("dims,nrhs", [((8, 16, 8, 24), 1), ((24, 8, 16, 8), 3), ((32, 16, 16, 32), 3)])
def test_layout_moves_every_number(dims, nrhs, prec):
    """Packing against the blocked order written out, unpacking against its inverse:
    numbers are moved, so the results are the same bits."""
    torch = torch_cuda()
    import paper_1202_2462_gb300 as G
    lx, ly, lz, lt = dims
    v = lx * ly * lz * lt
    s = G.Solver(dev(torch, synth.random_gauge_field(dims, 0.4, 3)), 1.0, 0.1, n_levels=1, precision="fp32", nrhs_max=nrhs)
    rng = np.random.default_rng(4)
    p = rng.normal(size=(nrhs, v, 12)) + 1j * rng.normal(size=(nrhs, v, 12))
    a = dev(torch, p, torch.complex128 if prec == "fp64" else torch.complex64)
    site = np.arange(v)
    x = [site % lx, site // lx % ly, site // (lx * ly) % lz, site // (lx * ly * lz)]
    blk = x[0] // 4 + lx // 4 * (x[1] // 4 + ly // 4 * (x[2] // 4 + lz // 4 * (x[3] // 4)))
    loc = x[0] % 4 + 4 * (x[1] % 4 + 4 * (x[2] % 4 + 4 * (x[3] % 4)))
    want = np.zeros((nrhs, v // 256, 12, 256), dtype=complex)
    want[:, blk, :, loc] = host(a).transpose(1, 0, 2)
    b, c = torch.empty_like(a), torch.empty_like(a)
    code = G.MG_FP64 if prec == "fp64" else G.MG_FP32
    G.mg_pack_spinor(s.ctx, a, b, code, nrhs)
    assert np.array_equal(host(b).reshape(want.shape), want)
    G.mg_unpack_spinor(s.ctx, b, c, code, nrhs)
    assert torch.equal(a, c)
    s.close()


@pytest.mark.parametrize("nrhs", [1, 4])
def test_outer_basis_in_half_precision(monkeypatch, nrhs):
    """Twenty outer steps in one cycle, so dot passes on 0 to 12 vectors and on 1 to 7
    more: the residual estimates with an FP16 basis against those with an FP32 basis.
    Each of the j stored vectors is off by at most 2^-11 of its norm, so the estimate
    after j steps by j 2^-11 of the first residual."""
    torch = torch_cuda()
    import paper_1202_2462_gb300 as G
    u = dev(torch, synth.random_gauge_field((8, 8, 8, 8), 0.4, 3))
    rng = np.random.default_rng(6)
    b = dev(torch, rng.normal(size=(nrhs, 4096, 12)) + 1j * rng.normal(size=(nrhs, 4096, 12)))
    est = []
    for flag in ("1", "0"):
        monkeypatch.setenv("SAPMG_OUTER_FP16", flag)
        s = G.Solver(u, 1.0, -0.2, n_levels=1, precision="fp16", nrhs_max=nrhs, fgmres_m=20, maxiter=20, n_mr=1,
                     tol=1e-12)
        s.solve(b)
        est.append([[e for _, e in s.history()[r]["estimates"]] for r in range(nrhs)])
        s.close()
    for r in range(nrhs):
        n = min(len(est[0][r]), len(est[1][r]))
        assert n >= 14
        for j in range(n):
            assert abs(est[0][r][j] - est[1][r][j]) <= (j + 1) * 2.0 ** -11, (r, j, est[0][r], est[1][r])


@pytest.mark.parametrize("prec", ["fp32", "fp16", "bf16"])
@pytest.mark.parametrize("n_vec", [1, 2, 3, 4, 8, 9, 17, 25])
def test_transfers_of_one_field(prec, n_vec):
    """One field's restriction and prolongation, at the vector counts where a thread per
    site gives way to the wide forms and where a warp has one, two or three vectors, against the oracle with the same rounded vectors: FP32
    sums of 1536 and n_vec products.  The prolongation also to an address that is not
    a multiple of 16 bytes."""
    torch = torch_cuda()
    import paper_1202_2462_gb300 as G
    dims, nb = (8, 8, 8, 8), 16
    u = dev(torch, synth.random_gauge_field(dims, 0.4, 39))
    iv = synth.test_vector_draw(dims, n_vec, 40)
    s = G.Solver(u, 1.0, 0.1, n_levels=2, n_vec=(n_vec,), setup_iters=0, precision=prec, init_vectors=dev(torch, iv))
    agg = Aggregation(dims, (4, 4, 4, 4), (4, 3)).build(iv)
    agg.q = round_storage(agg.q, "fp32" if prec == "fp32" else "fp16")     # BF16 is for links and clover only
    r = synth.random_spinor(dims, 41).astype(np.complex64)
    rc = torch.zeros((nb, 2 * n_vec), dtype=torch.complex64, device="cuda")
    G.mg_restrict(s.ctx, 0, dev(torch, r), rc, s.prec)
    ref = agg.restrict(r.astype(np.complex128)).reshape(nb, 2 * n_vec)
    assert rel(host(rc), ref) < 2e-6 and emax(host(rc), ref) < 6e-6
    z = torch.zeros(dims[::-1] + (4, 3), dtype=torch.complex64, device="cuda")
    G.mg_prolong(s.ctx, 0, rc, z, s.prec)
    back = agg.prolong(host(rc).astype(np.complex128).reshape(-1)).reshape(z.shape)
    assert rel(host(z), back) < 2e-6 and emax(host(z), back) < 6e-6
    odd = torch.zeros(z.numel() + 1, dtype=torch.complex64, device="cuda")[1:]
    G.mg_prolong(s.ctx, 0, rc, odd, s.prec | G.MG_BLOCKED)
    packed = torch.empty_like(odd.clone())
    G.mg_pack_spinor(s.ctx, z, packed, G.MG_FP32, 1)
    assert torch.equal(odd, packed)
    s.close()


@pytest.mark.parametrize("n_vec", [4, 12, 20, 32])
def test_one_coarse_vector(monkeypatch, n_vec):
    """The coarse product of one FP16 basis vector (256 sites, block sizes with full and
    partly idle warps): two GMRES steps with the basis in FP16 against the same with it
    in FP32.  The products and the two basis vectors are rounded by up to 2^-11 each; a
    wrong direction or row would be off by a tenth."""
    torch = torch_cuda()
    import paper_1202_2462_gb300 as G
    u = dev(torch, synth.random_gauge_field((16, 16, 16, 16), 0.4, 3))
    b = torch.randn((256, 2 * n_vec), dtype=torch.complex64, device="cuda",
                    generator=torch.Generator("cuda").manual_seed(3))
    x = []
    for flag in ("1", "0"):
        monkeypatch.setenv("SAPMG_COARSE_BASIS_FP16", flag)
        s = G.Solver(u, 1.0, -0.2, n_levels=2, n_vec=(n_vec,), setup_iters=0, precision="fp16", coarse_iters=2, seed=4)
        out = torch.empty_like(b)
        G.mg_coarse_solve(s.ctx, 1, b, out, s.prec)
        x.append(host(out))
        s.close()
    assert rel(x[0], x[1]) < 4 * 2.0 ** -11
