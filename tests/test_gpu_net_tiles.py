"""The set-up network's layer kernels at channel counts around their tile sizes (4
and 16 output channels, 16 (input channel, hop) pairs) and around the lines
between tiles and threads or CTAs of single channels, against the FP64 oracle;
fields at odd elements; a captured weight gradient."""

import numpy as np
import pytest

import synth
from oracle import learned as L
from tests.gpu_util import torch_cuda, dev, host, rel, round_storage

pytestmark = pytest.mark.gpu

DIMS = (8, 8, 8, 16)


def _blocked(torch, s, x):
    from paper_1202_2462_gb300.learned import GaugeNet
    return torch.cat([GaugeNet.blocked(s, dev(torch, x[c], torch.complex64)) for c in range(x.shape[0])])


def _canonical(torch, s, y, c):
    from paper_1202_2462_gb300.learned import GaugeNet
    fs = y.numel() // c
    return np.stack([host(GaugeNet.canonical(s, y[k * fs:(k + 1) * fs].contiguous()))[0] for k in range(c)])


# FP32 sums of 36 cin products (forward), of 36 cout (input gradient) and of 3 V
# (weights): 2e-6 as in the layer's own parity test
@pytest.mark.parametrize("cin,cout", [(1, 1), (1, 4), (4, 3), (3, 5), (2, 16), (16, 2), (5, 17), (7, 5), (8, 6), (13, 9), (2, 9),
                                      (1, 16)])
def test_layer_tiles(cin, cout):
    torch = torch_cuda()
    import paper_1202_2462_gb300 as G
    u = synth.random_gauge_field(DIMS, 0.4, 321)
    s = G.Solver(dev(torch, u), 1.0, -0.1, n_levels=1, precision="bf16", fgmres_m=1, antiperiodic_t=0)
    w = L.init_weights([(cout, cin)], 1)[0] * 3.0
    x = synth.random_spinor(DIMS, 322, nvec=cin)
    gy = synth.random_spinor(DIMS, 323, nvec=cout)
    wd, xd, gyd = dev(torch, w, torch.complex64), _blocked(torch, s, x), _blocked(torch, s, gy)
    yd = torch.empty(cout * xd.numel() // cin, dtype=torch.complex64, device="cuda")
    G.mg_net_layer_forward(s.ctx, cin, cout, wd, xd, yd)
    assert rel(_canonical(torch, s, yd, cout), L.layer(u, w, x)) < 2e-6
    gxd, gwd = torch.empty_like(xd), torch.empty_like(wd)
    G.mg_net_layer_backward(s.ctx, cin, cout, wd, xd, gyd, gxd, gwd)
    gx, gw = L.layer_backward(u, w, x, gy)
    assert rel(_canonical(torch, s, gxd, cin), gx) < 2e-6
    assert rel(host(gwd), gw) < 2e-6
    again = torch.empty_like(wd)
    G.mg_net_layer_backward(s.ctx, cin, cout, wd, xd, gyd, None, again)
    assert torch.equal(again, gwd)
    wb = torch.view_as_real(wd).to(torch.bfloat16).contiguous()
    G.mg_net_layer_forward_bf16(s.ctx, cin, cout, wb, xd, yd)
    ref = L.layer(round_storage(u, "bf16"), round_storage(w, "bf16"), x)
    assert rel(_canonical(torch, s, yd, cout), ref) < 2e-6
    s.close()


@pytest.mark.parametrize("cin,cout", [(4, 4), (8, 16), (16, 6)])
def test_layer_fields_at_odd_elements(cin, cout):
    """Fields that start on 8 bytes but not on 16 give the aligned fields' results bit for bit."""
    torch = torch_cuda()
    import paper_1202_2462_gb300 as G
    s = G.Solver(dev(torch, synth.random_gauge_field(DIMS, 0.4, 324)), 1.0, -0.1, n_levels=1, precision="bf16", fgmres_m=1)
    fs = int(np.prod(DIMS)) * 12
    gen = torch.Generator("cuda").manual_seed(5)

    def rnd(n):
        return torch.randn(n, dtype=torch.complex64, device="cuda", generator=gen)

    def odd(t):
        return torch.cat([t[:1], t])[1:]

    w, x, gy = rnd(cout * cin * 144), rnd(cin * fs), rnd(cout * fs)
    wb = torch.view_as_real(w).to(torch.bfloat16).contiguous()
    out = []
    for f in (lambda t: t, odd):
        xx, yy, yb, gg, gx, gw = f(x), f(torch.zeros_like(gy)), f(torch.zeros_like(gy)), f(gy), f(torch.zeros_like(x)), f(torch.zeros_like(w))
        assert all(t.data_ptr() % 16 == (0 if f is not odd else 8) for t in (xx, yy, yb, gg, gx, gw))
        G.mg_net_layer_forward(s.ctx, cin, cout, f(w), xx, yy)
        G.mg_net_layer_forward_bf16(s.ctx, cin, cout, wb, xx, yb)
        G.mg_net_layer_backward(s.ctx, cin, cout, f(w), xx, gg, gx, gw)
        out.append((yy, yb, gx, gw))
    assert all(torch.equal(a, b) for a, b in zip(*out))
    s.close()


def test_captured_weight_gradient():
    """A weight gradient captured as the first call of its context and replayed after a
    wider layer's: the eager call's result bit for bit, each time."""
    torch = torch_cuda()
    import paper_1202_2462_gb300 as G
    stream = torch.cuda.Stream()
    u = dev(torch, synth.random_gauge_field(DIMS, 0.4, 325))
    fs = int(np.prod(DIMS)) * 12
    gen = torch.Generator("cuda").manual_seed(6)

    def layer(cin, cout):
        def rnd(n):
            return torch.randn(n, dtype=torch.complex64, device="cuda", generator=gen)
        return cin, cout, rnd(cout * cin * 144), rnd(cin * fs), rnd(cout * fs)

    narrow, wide = layer(6, 6), layer(24, 16)
    gw = torch.empty_like(narrow[2])
    gwide = torch.empty_like(wide[2])
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        s = G.Solver(u, 1.0, -0.1, n_levels=1, precision="fp32", fgmres_m=1)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        G.mg_net_layer_backward(s.ctx, *narrow, None, gw)
    got = []
    for _ in range(2):
        gw.zero_()
        torch.cuda.synchronize()
        graph.replay()
        torch.cuda.synchronize()
        got.append(gw.clone())
        G.mg_net_layer_backward(s.ctx, *wide, None, gwide)
        torch.cuda.synchronize()
    G.mg_net_layer_backward(s.ctx, *narrow, None, gw)
    torch.cuda.synchronize()
    assert torch.equal(got[0], gw) and torch.equal(got[1], gw)
    s.close()
