"""The coarse solves with a second Gram-Schmidt pass (SAPMG_COARSE_REORTH=1)."""

import pytest

import synth
from tests.gpu_util import torch_cuda, dev, host, rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("levels,prec", [(2, "fp64"), (2, "fp32"), (2, "bf16"), (3, "fp64"), (3, "bf16")])
def test_second_pass_changes_rounding_only(levels, prec, monkeypatch):
    """The level-1 solve with the pass against the solve without: the same
    minimiser over the same Krylov space.  2N = 12 keeps the basis in the vector
    precision on every level, so the two differ by its rounding (2^-24 or 2^-53
    of a vector's norm per step and level) times the condition of the small
    least squares, which a thousandfold margin covers."""
    torch = torch_cuda()
    import paper_1202_2462_gb300 as G
    dims = (16, 8, 8, 16)
    kw = dict(n_levels=levels, n_vec=(6, 6), setup_iters=2, precision=prec, seed=7, coarse_iters=12)
    if levels == 3:
        kw.update(sap_block2=(2, 1, 1, 2), inner_iters=3)
    u = dev(torch, synth.random_gauge_field(dims, 0.4, 331))
    b = dev(torch, synth.random_spinor((4, 2, 2, 4), 332).reshape(64, 12),
            torch.complex128 if prec == "fp64" else torch.complex64)
    x = []
    for flag in ("1", "0"):
        monkeypatch.setenv("SAPMG_COARSE_REORTH", flag)
        s = G.Solver(u, 1.0, -0.1, **kw)
        out = torch.empty_like(b)
        G.mg_coarse_solve(s.ctx, 1, b, out, s.prec)
        x.append(host(out))
        s.close()
    assert rel(x[0], x[1]) < 1000 * (2.0 ** -53 if prec == "fp64" else 2.0 ** -24)
