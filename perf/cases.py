"""What the library's speed is measured on: the calls a program makes through the
public entry points, with seeded inputs, over the sizes, precisions and options
this repository's own workloads, tests and benchmark use.

Kinds of case:

* dirac   one application of D (or D^dagger) to a batch of fields;
* smooth  red-black Schwarz sweeps on D z = b;
* coarse  the coarse-grid pieces of a cycle for a batch: P^dagger v, D_c of it,
          and P of it;
* cycle   one application of the two-level cycle as a preconditioner;
* solve   mg_solve to 1e-10, two or three levels, one or many sources;
* setup   building a hierarchy from a gauge field (bootstrap, P, D_c);
* net     one training step of the set-up network, or its BF16 inference.

Gauge links are exp(i eps H), H traceless Hermitian with Gaussian entries, the
recipe of the repository's synthetic workloads, drawn on the GPU.  The lattices
have extents that are multiples of 8 (what the library accepts), cubic and
elongated.  exact() restates every path in FP64 torch, from the definitions.
"""

import math

import torch

import paper_1202_2462_gb300 as G
from paper_1202_2462_gb300 import binding as B
from paper_1202_2462_gb300.learned import GaugeNet

C_SW = 1.0
EPS = 0.5
M0 = -0.40          # the physical side of the critical mass (about -0.50 at eps 0.5)
DIMS = ("lx", "ly", "lz", "lt")


def _case(kind, dims, **kw):
    c = {"kind": kind}
    c.update(zip(DIMS, dims))
    c.update(kw)
    return c


def listed():
    return [
        # the smallest call: an FP64 application on the test lattice, canonical layout, where launches count
        dict(_case("dirac", (8, 8, 8, 8), prec="fp64", nrhs=1, blocked=False, dagger=False, anti=False),
             name="dirac-fp64-small"),
        # the benchmark's HBM figure: one field at the largest lattice, BF16 links
        dict(_case("dirac", (32, 32, 32, 64), prec="bf16", nrhs=1, blocked=True, dagger=False, anti=False),
             name="dirac-bf16-large"),
        # the Krylov operator of the 12-source solve: FP32 links, 12 fields, an elongated lattice
        dict(_case("dirac", (24, 16, 40, 48), prec="fp32", nrhs=12, blocked=True, dagger=False, anti=True),
             name="dirac-fp32-batch"),
        # the smoother of the 12-source solve with the production parameters
        dict(_case("smooth", (32, 32, 32, 32), prec="bf16", nrhs=12, blocked=True, n_mr=5, sweeps=1, tuned=True),
             name="smooth-bf16-batch"),
        # a caller's own five fields in the canonical layout: an odd count, FP16 links
        dict(_case("smooth", (16, 24, 8, 40), prec="fp16", nrhs=5, blocked=False, n_mr=4, sweeps=2, tuned=False),
             name="smooth-fp16-odd"),
        # the coarse side of the 12-source solve at the largest lattice
        dict(_case("coarse", (32, 32, 32, 64), prec="bf16", nrhs=12, n_vec=20), name="coarse-bf16-batch"),
        # the cycle as a preconditioner of a caller's own Krylov method, one field
        dict(_case("cycle", (16, 16, 16, 32), prec="fp16", n_vec=20, n_mr=4, nu_post=2, coarse_iters=12,
                   setup_iters=3), name="cycle-fp16-single"),
        # the 12 point sources of a propagator with the production parameters
        dict(_case("solve", (24, 24, 24, 48), prec="bf16", nrhs=12, levels=2, n_vec=20, n_mr=5, nu_post=1,
                   coarse_iters=20, inner_iters=8, setup_iters=20, fgmres_m=14), name="solve-bf16-batch"),
        # one source on three levels (the three-level workload's parameters)
        dict(_case("solve", (16, 16, 16, 32), prec="fp16", nrhs=1, levels=3, n_vec=20, n_mr=4, nu_post=2,
                   coarse_iters=12, inner_iters=8, setup_iters=3, fgmres_m=20), name="solve-fp16-three-level"),
        # the plain FP64 method on the test lattice: many short launches and host round trips
        dict(_case("solve", (8, 8, 8, 8), prec="fp64", nrhs=1, levels=2, n_vec=8, n_mr=4, nu_post=2,
                   coarse_iters=12, inner_iters=8, setup_iters=3, fgmres_m=20), name="solve-fp64-small"),
        # a new gauge field: the whole set-up, as every field of an ensemble pays it once
        dict(_case("setup", (16, 16, 16, 32), prec="bf16", nrhs=12, n_vec=20, n_mr=5, setup_iters=20),
             name="setup-bf16"),
        # one training step of the set-up network on its training lattice
        dict(_case("net", (16, 16, 16, 16), prec="fp32", mode="train", channels=16, layers=3), name="net-train"),
    ]


def _draw_dims(rng, most):
    """Extents from 8 to 64 whose volume is spread over its logarithm up to `most` sites."""
    want = math.exp(rng.uniform(math.log(4096), math.log(most * 1.001)))
    for _ in range(1000):
        d = [rng.choice((8, 16, 24, 32, 40, 48, 56, 64)) for _ in range(4)]
        v = d[0] * d[1] * d[2] * d[3]
        if want / 1.5 <= v <= min(most, want * 1.5):
            return d
    return [8, 8, 8, 8]


def draw(rng):
    kind = rng.choice(("dirac", "dirac", "smooth", "smooth", "coarse", "cycle", "solve", "solve", "setup", "net"))
    if kind == "dirac":
        prec = rng.choice(("fp64", "fp32", "fp16", "bf16"))
        nrhs = rng.randint(1, 12)
        dims = _draw_dims(rng, 2097152 // (nrhs if prec == "fp64" else max(1, nrhs // 3)))
        return _case("dirac", dims, prec=prec, nrhs=nrhs, blocked=rng.random() < 0.5,
                     dagger=prec in ("fp64", "fp32") and rng.random() < 0.3, anti=rng.random() < 0.5)
    if kind == "smooth":
        prec = rng.choice(("fp64", "fp32", "fp16", "bf16", "bf16"))
        nrhs = rng.randint(1, 2) if prec == "fp64" else rng.randint(1, 12)
        return _case("smooth", _draw_dims(rng, 65536 if prec == "fp64" else 4194304 // max(4, nrhs)), prec=prec,
                     nrhs=nrhs, blocked=rng.random() < 0.5, n_mr=rng.randint(2, 6), sweeps=rng.randint(1, 3),
                     tuned=prec != "fp64" and rng.random() < 0.5)
    if kind == "coarse":
        return _case("coarse", _draw_dims(rng, 1048576), prec=rng.choice(("fp32", "fp16", "bf16")),
                     nrhs=rng.randint(1, 12), n_vec=rng.choice((8, 12, 15, 16, 20, 24)))
    if kind == "cycle":
        return _case("cycle", _draw_dims(rng, 262144), prec=rng.choice(("fp32", "fp16", "bf16")),
                     n_vec=rng.choice((8, 12, 16, 20, 24)), n_mr=rng.randint(3, 5), nu_post=rng.randint(1, 2),
                     coarse_iters=rng.randint(8, 20), setup_iters=rng.randint(1, 3))
    if kind == "solve":
        levels = rng.choice((2, 2, 3))
        prec = rng.choice(("fp16", "bf16", "bf16"))
        if levels == 3:                     # the level-1 boxes of 2^4 need extents that are multiples of 16
            dims = [rng.choice((16, 16, 32)) for _ in range(4)]
        else:
            dims = _draw_dims(rng, 300000)
        return _case("solve", dims, prec=prec, nrhs=rng.choice((1, 2, 3, 4, 6, 12)) if levels == 2 else 1,
                     levels=levels, n_vec=20, n_mr=rng.randint(4, 5), nu_post=rng.randint(1, 2),
                     coarse_iters=rng.randint(12, 20), inner_iters=rng.randint(2, 8), setup_iters=rng.randint(4, 12),
                     fgmres_m=rng.randint(12, 20))
    if kind == "setup":
        return _case("setup", _draw_dims(rng, 200000), prec=rng.choice(("fp32", "fp16", "bf16")),
                     nrhs=rng.choice((2, 12)), n_vec=rng.choice((8, 12, 16, 20, 24)), n_mr=rng.randint(4, 5),
                     setup_iters=rng.randint(3, 12))
    mode = rng.choice(("train", "infer"))
    return _case("net", _draw_dims(rng, 65536), prec="fp32" if mode == "train" else "bf16", mode=mode,
                 channels=rng.choice((8, 12, 16)), layers=rng.randint(2, 3))


# ---------------------------------------------------------------- seeded inputs

def _lat(case):
    return tuple(case[d] for d in reversed(DIMS))       # (Lt, Lz, Ly, Lx)


def _volume(case):
    return case["lx"] * case["ly"] * case["lz"] * case["lt"]


def _gen(seed, stream):
    return torch.Generator(device="cuda").manual_seed(1000 * int(seed) + stream)


def _mm(a, b):
    """3x3 products over the leading axes."""
    return a[..., :, 0:1] * b[..., 0:1, :] + a[..., :, 1:2] * b[..., 1:2, :] + a[..., :, 2:3] * b[..., 2:3, :]


def _dag(a):
    return a.transpose(-1, -2).conj()


def _gauge(case, seed):
    """exp(i EPS H): a Taylor series of the exponential (||EPS H|| is below 4: 30 terms reach rounding)."""
    lat = _lat(case)
    out = torch.empty(lat + (4, 3, 3), dtype=torch.complex128, device="cuda")
    gen = _gen(seed, 1)
    eye = torch.eye(3, dtype=torch.complex128, device="cuda")
    for t in range(lat[0]):
        m = torch.randn(lat[1:] + (4, 3, 3), dtype=torch.complex128, device="cuda", generator=gen)
        h = 0.5 * (m + _dag(m))
        h = 1j * EPS * (h - eye * (h.diagonal(dim1=-2, dim2=-1).sum(-1) / 3.0)[..., None, None])
        acc = eye + h / 30.0
        for k in range(29, 0, -1):
            acc = eye + _mm(h, acc) / k
        out[t] = acc
    return out


def _fields(case, seed, stream, n, dtype):
    return torch.randn((n,) + _lat(case) + (4, 3), dtype=dtype, device="cuda", generator=_gen(seed, stream))


def _sources(case, seed, n):
    """The first n of the 12 spin-colour point sources at a seeded origin."""
    lat = _lat(case)
    at = torch.randint(0, 1 << 30, (4,), generator=torch.Generator().manual_seed(int(seed) + 7)).tolist()
    b = torch.zeros((n,) + lat + (4, 3), dtype=torch.complex128, device="cuda")
    for k in range(n):
        b[(k,) + tuple(a % l for a, l in zip(at, lat)) + (k // 3, k % 3)] = 1.0
    return b


def _to_blocked(x):
    """(R, Lt, Lz, Ly, Lx, 4, 3) -> (R, blocks, 12, 256), the library's blocked layout."""
    r, lt, lz, ly, lx = x.shape[:5]
    y = x.reshape(r, lt // 4, 4, lz // 4, 4, ly // 4, 4, lx // 4, 4, 12)
    return y.permute(0, 1, 3, 5, 7, 9, 2, 4, 6, 8).reshape(r, lt * lz * ly * lx // 256, 12, 256).contiguous()


def _net_weights(case, seed):
    ch = case["channels"]
    shapes = [(ch, 1)] + [(ch, ch)] * (case["layers"] - 2) + [(1, ch)]
    gen = _gen(seed, 5)
    return [torch.randn((co, ci, 9, 4, 4), dtype=torch.complex64, device="cuda", generator=gen) *
            (1.0 / math.sqrt(ci * 36)) for co, ci in shapes]


def _solver(case, u, **kw):
    return G.Solver(u, C_SW, M0, precision=case["prec"], **kw)


class State:
    pass


def prepare(case, seed):
    s = State()
    s.case = dict(case)
    kind, n = case["kind"], case.get("nrhs", 1)
    vt = torch.complex128 if case["prec"] == "fp64" else torch.complex64
    u = _gauge(case, seed)
    if kind == "dirac":
        s.solver = _solver(case, u, n_levels=1, nrhs_max=n, fgmres_m=1, antiperiodic_t=int(case["anti"]))
        s.prec = s.solver.prec | (B.MG_BLOCKED if case["blocked"] else 0) | (B.MG_DAGGER if case["dagger"] else 0)
        x = _fields(case, seed, 2, n, vt)
        s.x = _to_blocked(x) if case["blocked"] else x
    elif kind == "smooth":
        kw = dict(n_levels=2, n_vec=(8,), setup_iters=0, autotune=1, seed=seed + 1) if case["tuned"] else dict(n_levels=1)
        s.solver = _solver(case, u, nrhs_max=n, fgmres_m=8, n_mr=case["n_mr"], **kw)
        b, z = _fields(case, seed, 2, n, vt), _fields(case, seed, 3, n, vt)
        s.b, s.z = (_to_blocked(b), _to_blocked(z)) if case["blocked"] else (b, z)
    elif kind == "coarse":
        init = _fields(case, seed, 4, case["n_vec"], torch.complex64)
        s.solver = _solver(case, u, n_levels=2, nrhs_max=n, n_vec=(case["n_vec"],), setup_iters=0,
                           fgmres_m=-(-case["n_vec"] // n), autotune=1, init_vectors=init)
        del init
        s.v = _to_blocked(_fields(case, seed, 2, n, vt))
    elif kind == "cycle":
        init = _fields(case, seed, 4, case["n_vec"], torch.complex64)
        s.solver = _solver(case, u, n_levels=2, n_vec=(case["n_vec"],), setup_iters=case["setup_iters"],
                           n_mr=case["n_mr"], nu_post=case["nu_post"], coarse_iters=case["coarse_iters"],
                           fgmres_m=case["n_vec"], init_vectors=init)
        s.v = _fields(case, seed, 2, 1, vt)[0]
    elif kind == "solve":
        s.solver = _solver(case, u, n_levels=case["levels"], nrhs_max=n, n_vec=(case["n_vec"], case["n_vec"]),
                           setup_iters=case["setup_iters"], n_mr=case["n_mr"], nu_post=case["nu_post"],
                           coarse_iters=case["coarse_iters"], inner_iters=case["inner_iters"],
                           fgmres_m=case["fgmres_m"], seed=seed + 1, autotune=int(case["prec"] != "fp64"))
        s.b = _sources(case, seed, n)
    elif kind == "setup":
        s.u = u
        s.init = _fields(case, seed, 4, case["n_vec"], torch.complex64)
    elif kind == "net":
        s.solver = _solver(case, u, n_levels=1, fgmres_m=2)
        s.net = GaugeNet(channels=case["channels"], layers=case["layers"])
        for w, w0 in zip(s.net.weights, _net_weights(case, seed)):
            w.copy_(w0)
        x, t = _fields(case, seed, 2, 1, torch.complex64), _fields(case, seed, 3, 1, torch.complex64)
        # the target of training is a smoothed field of the input's size: here the input and half as much noise
        s.x, s.t = _to_blocked(x).reshape(-1), _to_blocked(0.8 * x + 0.4 * t).reshape(-1)
    else:
        raise ValueError(kind)
    return s


def run(s):
    case = s.case
    kind, n = case["kind"], case.get("nrhs", 1)
    if kind == "dirac":
        return s.solver.dirac(s.x, s.prec)
    if kind == "smooth":
        if not case["blocked"]:
            return s.solver.smooth(s.b, s.z, case["sweeps"])
        B.sap_smooth(s.solver.ctx, s.b, s.z, case["sweeps"], s.solver.prec | B.MG_BLOCKED, n)
        return s.z
    if kind == "coarse":
        ctx, prec = s.solver.ctx, s.solver.prec
        vc = torch.empty((n, _volume(case) // 256, 2 * case["n_vec"]), dtype=s.v.dtype, device="cuda")
        y, z = torch.empty_like(vc), torch.empty_like(s.v)
        B.mg_restrict_batch(ctx, 0, s.v, vc, prec | B.MG_BLOCKED, n)
        B.mg_coarse_apply_batch(ctx, 1, vc, y, prec, n)
        B.mg_prolong_batch(ctx, 0, vc, z, prec | B.MG_BLOCKED, n)
        return [vc, y, z]
    if kind == "cycle":
        z = torch.empty_like(s.v)
        B.mg_precondition(s.solver.ctx, s.v, z, B.MG_FP32)
        return z
    if kind == "solve":
        z, info, code = s.solver.solve(s.b)
        if code != B.MG_OK:
            raise RuntimeError("the solve did not converge: %g after %d iterations" % (info.relres, info.iterations))
        return list(z)
    if kind == "setup":
        solver = _solver(case, s.u, n_levels=2, nrhs_max=n, n_vec=(case["n_vec"],), n_mr=case["n_mr"],
                         setup_iters=case["setup_iters"], fgmres_m=14, init_vectors=s.init)
        v = torch.empty((case["n_vec"],) + solver.lat + (4, 3), dtype=torch.complex128, device="cuda")
        n2 = 2 * case["n_vec"]
        m = torch.empty((_volume(case) // 256, 9, n2, n2), dtype=torch.complex128, device="cuda")
        B.mg_get_vectors(solver.ctx, 0, v)
        B.mg_get_coarse_op(solver.ctx, 1, m)
        solver.close()
        return [v, m]
    if case["mode"] == "infer":
        return s.net.forward_bf16(s.solver, s.x)
    out, cache = s.net.forward(s.solver, s.x)
    loss, grads = s.net.backward(s.solver, out, cache, s.t)
    s.net.adam(s.solver, grads)
    return {"out": out, "loss": loss, "grads": grads, "weights": s.net.weights}


# ---------------------------------------------------------------- the work of one pass

_EB = {"fp64": 16, "fp32": 8, "fp16": 8, "bf16": 8}       # bytes of a vector entry
_SB = {"fp64": 16, "fp32": 8, "fp16": 4, "bf16": 4}       # bytes of a stored field entry
_DIRAC = 1848.0                                            # flops of D a site and field
_ITERATIONS = 32.0                                         # outer iterations of a solve at M0, about


def _smooth_flops(v, n, n_mr):
    return v * n * (1896.0 + 1854.0 * n_mr)


def _net_layers(case):
    ch = case["channels"]
    return [(ch, 1)] + [(ch, ch)] * (case["layers"] - 2) + [(1, ch)]


def work(case):
    kind, n, v = case["kind"], case.get("nrhs", 1), float(_volume(case))
    eb, sb = _EB[case["prec"]], _SB[case["prec"]]
    if kind == "dirac":
        return {"bytes": v * (24 * eb * n + 72 * sb), "flops": _DIRAC * v * n}
    if kind == "smooth":
        return {"bytes": v * (36 * eb * n + 72 * sb), "flops": case["sweeps"] * _smooth_flops(v, n, case["n_mr"])}
    nv = case.get("n_vec", 0)
    sites, n2 = v / 256, 2.0 * nv
    transfer = v * 12 * nv * 8.0
    if kind == "coarse":
        return {"bytes": v * (12 * nv * min(sb, 8) + 24 * 8 * n) + sites * (9 * n2 * n2 * 4 + 4 * n2 * 8 * n),
                "flops": n * (2 * transfer + sites * 9 * n2 * n2 * 8)}
    if kind in ("cycle", "solve"):
        cycle = 2 * transfer + case["coarse_iters"] * sites * 9 * n2 * n2 * 8 + \
            case["nu_post"] * _smooth_flops(v, 1, case["n_mr"])
        if kind == "cycle":
            return {"bytes": v * (24 * eb + 72 * sb + 12 * nv * min(sb, 8)) + sites * 9 * n2 * n2 * 4, "flops": cycle}
        return {"bytes": v * (24 * 16 * n + 72 * 16 + 12 * nv * min(sb, 8)) + sites * 9 * n2 * n2 * 4,
                "flops": n * _ITERATIONS * (cycle + _DIRAC * v)}
    if kind == "setup":
        return {"bytes": v * (36 * 16 + 12 * nv * (8 + 16)) + sites * 9 * n2 * n2 * 16,
                "flops": nv * case["setup_iters"] * (_smooth_flops(v, 1, case["n_mr"]) + 2 * nv * 12 * 8 * v) +
                n2 * v * (_DIRAC + 3 * 12 * nv * 8.0)}
    layers = sum(co * ci for co, ci in _net_layers(case)) * 9 * 16 * 3 * 8.0 * v
    fields = sum(co + ci for co, ci in _net_layers(case)) * 12 * 8.0 * v
    train = case["mode"] == "train"
    return {"bytes": (3 if train else 1) * fields + 36 * sb * v, "flops": (3 if train else 1) * layers}


def tolerance(case):
    """About four times what the path differs from exact() by at the listed and drawn sizes."""
    kind, prec = case["kind"], case["prec"]
    if kind == "dirac":                 # 2e-16 and 1e-7 seen
        return {"rel": 1e-15, "max": 1e-13} if prec == "fp64" else {"rel": 5e-7, "max": 2e-5}
    if kind == "smooth":                # 4e-16 and 5e-7
        return {"rel": 4e-15, "max": 4e-13} if prec == "fp64" else {"rel": 2e-6, "max": 1e-4}
    if kind == "coarse":                # TF32 transfers, FP16 operator and P: 4e-4
        return {"rel": 2e-3, "max": 2e-2}
    if kind == "cycle":                 # a fixed number of coarse GMRES steps, FP16 operator and P: 1e-4
        return {"rel": 5e-4, "max": 2e-2}
    if kind == "solve":                 # both stop at 1e-10 of the source, times ||D|| / sigma_min: 1e-9
        return {"rel": 1e-8, "max": 1e-6}
    if kind == "setup":                 # FP32 sweeps from the same initial vectors: 1.3e-6
        return {"rel": 1e-5, "max": 1e-3}
    return {"rel": 1e-5, "max": 1e-3}   # the updated weights: 2e-6


# ---------------------------------------------------------------- the same in FP64 torch

def _rounded(x, prec):
    """x in the storage precision, back in complex128."""
    t = {"fp64": torch.float64, "fp32": torch.float32, "fp16": torch.float16, "bf16": torch.bfloat16}[prec]
    return torch.view_as_complex(torch.view_as_real(x).to(t).to(torch.float64))


def _clover(u):
    """A(x) - (4 + m0) as two 6x6 chiral blocks (..., 2, 6, 6) in the chiral basis."""
    def sh(f, mu, k):
        return torch.roll(f, -k, 3 - mu)

    def gmat(mu, nu):                    # c_sw (i/2) Fhat, Fhat = (Q - Q^dagger) / 8, Q the four leaves
        a, b = u[..., mu, :, :], u[..., nu, :, :]
        am, bm = sh(a, mu, -1), sh(b, mu, -1)
        an, bn = sh(a, nu, -1), sh(b, nu, -1)
        q = _mm(_mm(a, sh(b, mu, 1)), _mm(_dag(sh(a, nu, 1)), _dag(b)))
        q = q + _mm(_mm(b, _dag(sh(am, nu, 1))), _mm(_dag(bm), am))
        q = q + _mm(_mm(_dag(am), _dag(sh(bm, nu, -1))), _mm(sh(am, nu, -1), bn))
        q = q + _mm(_mm(_dag(bn), an), _mm(sh(bn, mu, 1), _dag(a)))
        return (0.5j * C_SW / 8.0) * (q - _dag(q))

    gxy, gxz, gyz, gxt, gyt, gzt = (gmat(*p) for p in ((0, 1), (0, 2), (1, 2), (0, 3), (1, 3), (2, 3)))
    out = torch.empty(u.shape[:4] + (2, 6, 6), dtype=u.dtype, device=u.device)
    for chi, sg in ((0, 1.0), (1, -1.0)):
        # sigma_xy = -s3, sigma_xz = s2, sigma_yz = -s1, sigma_kt = +-s_k on the two chiralities
        b1, b2, b3 = sg * gxt - gyz, gxz + sg * gyt, sg * gzt - gxy
        out[..., chi, :3, :3], out[..., chi, 3:, 3:] = b3, -b3
        out[..., chi, :3, 3:], out[..., chi, 3:, :3] = b1 - 1j * b2, b1 + 1j * b2
    return out


class Ref:
    """D of Eq. 1.1 with its links and clover term rounded to a storage precision."""

    X = [[[0, -1j], [-1j, 0]], [[0, -1], [1, 0]], [[-1j, 0], [0, 1j]], [[1, 0], [0, 1]]]   # -i s_k and 1

    def __init__(self, case, u, prec):
        self.lat = _lat(case)
        a = _clover(u)
        a += (4.0 + M0) * torch.eye(6, dtype=u.dtype, device=u.device)
        self.a = _rounded(a, prec)
        v = u.clone() if case.get("anti") else u
        if case.get("anti"):
            v[-1, ..., 3, :, :] *= -1.0
        v = _rounded(v, prec)
        self.uf = [v[..., mu, :, :].contiguous() for mu in range(4)]
        self.ub = [_dag(torch.roll(self.uf[mu], 1, 3 - mu)).resolve_conj().contiguous() for mu in range(4)]
        self.x = [torch.tensor(x, dtype=torch.complex128, device=u.device) for x in self.X]
        c = torch.meshgrid(*[torch.arange(l, device=u.device) for l in self.lat], indexing="ij")     # t, z, y, x
        self.coord = [c[3 - mu] for mu in range(4)]
        self.colour = sum(q // 4 for q in self.coord) % 2

    def local(self, p):
        return torch.einsum("...ij,...j->...i", self.a, p.reshape(self.lat + (2, 6))).reshape(self.lat + (4, 3))

    def hop(self, p, mu, step):
        """-1/2 (1 -+ gamma_mu) U psi(x +- mu)."""
        sg, w = (-1.0, self.uf[mu]) if step > 0 else (1.0, self.ub[mu])
        n = torch.roll(p, -step, 3 - mu)
        h = n[..., :2, :] + sg * torch.einsum("st,...tc->...sc", self.x[mu], n[..., 2:, :])
        g = -0.5 * (w[..., None, :, :] * h[..., None, :]).sum(-1)
        low = sg * torch.einsum("ts,...tc->...sc", self.x[mu].conj(), g)
        return torch.cat((g, low), -2)

    def crossing(self, mu, step):
        """1 at the sites whose hop leaves the 4^4 block."""
        return (self.coord[mu] % 4 == (3 if step > 0 else 0)).to(torch.float64)[..., None, None]

    def apply(self, p, inside=False):
        out = self.local(p)
        for mu in range(4):
            for step in (1, -1):
                h = self.hop(p, mu, step)
                out += h * (1.0 - self.crossing(mu, step)) if inside else h
        return out

    def dagger(self, p):
        f = p.clone()
        f[..., 2:, :] *= -1.0
        f = self.apply(f)
        f[..., 2:, :] *= -1.0
        return f

    def block_sum(self, f):
        lt, lz, ly, lx = self.lat
        s = f.reshape(lt // 4, 4, lz // 4, 4, ly // 4, 4, lx // 4, 4).sum((1, 3, 5, 7), keepdim=True)
        return s.expand(lt // 4, 4, lz // 4, 4, ly // 4, 4, lx // 4, 4).reshape(self.lat)

    def sweeps(self, b, z, n, n_mr):
        """Algorithm 1 with n_mr minimal-residual steps a block; b may be None (zero)."""
        for _ in range(n):
            for col in (0, 1):
                m = (self.colour == col).to(torch.float64)[..., None, None]
                d = self.apply(z)
                r = m * (-d if b is None else b - d)
                e = torch.zeros_like(z)
                for _ in range(n_mr):
                    p = self.apply(r, inside=True)
                    pr = self.block_sum((p.conj() * r).sum((-1, -2)))
                    pp = self.block_sum((p.conj() * p).real.sum((-1, -2)))
                    al = torch.where(pp > 0, pr / torch.where(pp > 0, pp, 1.0), 0.0)[..., None, None]
                    e = e + al * r
                    r = r - al * p
                z = z + e
        return z

    # aggregates: the 4^4 blocks, split by chirality; (..., blocks, 2, 1536)
    def agg(self, p):
        lt, lz, ly, lx = self.lat
        y = p.reshape(lt // 4, 4, lz // 4, 4, ly // 4, 4, lx // 4, 4, 2, 6).permute(0, 2, 4, 6, 8, 9, 1, 3, 5, 7)
        return y.reshape(-1, 2, 1536)

    def unagg(self, y):
        lt, lz, ly, lx = self.lat
        y = y.reshape(lt // 4, lz // 4, ly // 4, lx // 4, 2, 6, 4, 4, 4, 4).permute(0, 6, 1, 7, 2, 8, 3, 9, 4, 5)
        return y.reshape(self.lat + (4, 3))

    def local_basis(self, vectors):
        """The positive-diagonal QR factor of the vectors on every aggregate: (blocks, 2, N, 1536)."""
        q = torch.stack([self.agg(x) for x in vectors], 2)
        for _ in range(2):                               # Cholesky QR twice
            gr = q @ q.conj().transpose(-1, -2)          # gr[i, j] = sum q_i conj(q_j)
            q = torch.linalg.solve_triangular(torch.linalg.cholesky(gr), q, upper=False)
        return q

    def restrict(self, q, p):
        return (q.conj() @ self.agg(p)[..., None])[..., 0].reshape(q.shape[0], -1)

    def prolong(self, q, e):
        return self.unagg((e.reshape(q.shape[0], 2, 1, -1) @ q)[..., 0, :])

    def bootstrap(self, init, sweeps, n_mr):
        v = [x.to(torch.complex128) for x in init]
        for _ in range(sweeps):
            for k in range(len(v)):
                v[k] = self.sweeps(None, v[k], 1, n_mr)
                for _ in range(2):
                    for j in range(k):
                        v[k] = v[k] - (v[j].conj() * v[k]).sum() * v[j]
                v[k] = v[k] / torch.linalg.vector_norm(v[k])
        return v


def _gmres(apply, b, k):
    """k steps of GMRES from zero."""
    beta = torch.linalg.vector_norm(b)
    v, h = [b / beta], torch.zeros((k + 1, k), dtype=b.dtype, device=b.device)
    for j in range(k):
        w = apply(v[j])
        for _ in range(2):
            for i in range(j + 1):
                c = (v[i].conj() * w).sum()
                h[i, j] += c
                w = w - c * v[i]
        h[j + 1, j] = torch.linalg.vector_norm(w)
        v.append(w / h[j + 1, j])
    e = torch.zeros((k + 1, 1), dtype=b.dtype, device=b.device)
    e[0, 0] = beta
    hh = h.conj().T
    y = torch.linalg.solve(hh @ h, hh @ e)[:, 0]
    return sum(y[j] * v[j] for j in range(k))


def _cgn(ref, b):
    """D^{-1} b by CG on the normal equations to rounding."""
    x, r = torch.zeros_like(b), b.clone()
    s = ref.dagger(r)
    p, g = s.clone(), (s.conj() * s).real.sum()
    bb = float((b.conj() * b).real.sum())
    for k in range(4000):
        q = ref.apply(p)
        al = g / (q.conj() * q).real.sum()
        x, r = x + al * p, r - al * q
        s = ref.dagger(r)
        g2 = (s.conj() * s).real.sum()
        p, g = s + (g2 / g) * p, g2
        if k % 20 == 19 and float((r.conj() * r).real.sum()) < 1e-25 * bb:
            break
    return x


def _exact_net(case, u, seed):
    train = case["mode"] == "train"
    v = _rounded(u, "fp32" if train else "bf16")
    uf = [v[..., mu, :, :] for mu in range(4)]
    ub = [_dag(torch.roll(uf[mu], 1, 3 - mu)) for mu in range(4)]

    def transport(x, h):
        if h == 0:
            return x
        mu, step = (h - 1) // 2, 1 if h % 2 else -1
        w = uf[mu] if step > 0 else ub[mu]
        n = torch.roll(x, -step, 4 - mu)
        return sum(w[..., None, :, k] * n[..., :, k:k + 1] for k in range(3))

    def layer(w, x):
        return sum(torch.einsum("abst,b...tc->a...sc", w[:, :, h], transport(x, h)) for h in range(9))

    weights = [w.to(torch.complex128) if train else _rounded(w.to(torch.complex128), "bf16")
               for w in _net_weights(case, seed)]
    x0, t = (_fields(case, seed, k, 1, torch.complex64) for k in (2, 3))
    t = (0.8 * x0 + 0.4 * t).to(torch.complex128)
    x = x0.to(torch.complex128)
    for w in weights:
        w.requires_grad_(train)
    for k, w in enumerate(weights):
        x = layer(w, x)
        if k + 1 < len(weights):
            x = x / torch.sqrt(1.0 + (x.conj() * x).real.sum((-1, -2), keepdim=True))
    out = _to_blocked(x.detach()).reshape(-1)
    if not train:
        return out
    loss = ((x - t).conj() * (x - t)).real.sum() / (t.conj() * t).real.sum()
    loss.backward()
    grads = [w.grad for w in weights]
    new = []
    for w, g in zip(weights, grads):                     # Adam's first step on real and imaginary parts
        r = torch.view_as_real(g)
        new.append(w.detach() - torch.view_as_complex(1e-2 * r / (r.abs() + 1e-8)))
    return {"out": out, "loss": float(loss.detach()), "grads": grads, "weights": new}


def exact(case, seed):
    kind, n, prec = case["kind"], case.get("nrhs", 1), case["prec"]
    vt = torch.complex128 if prec == "fp64" else torch.complex64
    if kind == "solve" and _volume(case) > 140000:
        return None
    u = _gauge(case, seed)
    if kind == "net":
        return _exact_net(case, u, seed)
    if kind == "solve":
        ref = Ref(case, u, "fp64")
        return [_cgn(ref, b) if k == 0 else None for k, b in enumerate(_sources(case, seed, n))]
    ref = Ref(case, u, "fp32" if kind == "coarse" else prec)
    if kind == "dirac":
        x = _fields(case, seed, 2, n, vt)
        out = torch.empty(x.shape, dtype=torch.complex128, device="cuda")
        for k in range(n):
            p = x[k].to(torch.complex128)
            out[k] = ref.dagger(p) if case["dagger"] else ref.apply(p)
        return _to_blocked(out) if case["blocked"] else out
    if kind == "smooth":
        b, z = _fields(case, seed, 2, n, vt), _fields(case, seed, 3, n, vt)
        out = torch.empty(b.shape, dtype=torch.complex128, device="cuda")
        for k in range(n):
            out[k] = ref.sweeps(b[k].to(torch.complex128), z[k].to(torch.complex128), case["sweeps"], case["n_mr"])
        return _to_blocked(out) if case["blocked"] else out
    init = _fields(case, seed, 4, case["n_vec"], torch.complex64)
    if kind == "coarse":
        q = ref.local_basis([x.to(torch.complex128) for x in init])
        del init
        vs = _fields(case, seed, 2, n, vt)
        nb = q.shape[0]
        vc, y = (torch.empty((n, nb, 2 * case["n_vec"]), dtype=torch.complex128, device="cuda") for _ in range(2))
        z = torch.empty((n, nb, 12, 256), dtype=torch.complex64, device="cuda")
        for k in range(n):
            vc[k] = ref.restrict(q, vs[k].to(torch.complex128))
            p = ref.prolong(q, vc[k])
            y[k] = ref.restrict(q, ref.apply(p))
            z[k] = _to_blocked(p[None])[0]
        return [vc, y, z]
    basis = ref.bootstrap(init, case["setup_iters"], case["n_mr"])
    q = ref.local_basis(basis)
    fine = Ref(case, u, "fp32")                          # D_c is built from FP32 links
    if kind == "cycle":
        v = _fields(case, seed, 2, 1, vt)[0].to(torch.complex128)
        e = _gmres(lambda x: fine.restrict(q, fine.apply(fine.prolong(q, x))), fine.restrict(q, v),
                   case["coarse_iters"])
        return ref.sweeps(v, fine.prolong(q, e), case["nu_post"], case["n_mr"])
    nb, nv = q.shape[0], case["n_vec"]
    m = torch.empty((nb, 9, 2 * nv, 2 * nv), dtype=torch.complex128, device="cuda")
    for j in range(2 * nv):
        col = torch.zeros((nb, 2, 1536), dtype=torch.complex128, device="cuda")
        col[:, j // nv] = q[:, j // nv, j % nv]
        p = fine.unagg(col)
        m[:, 0, :, j] = fine.restrict(q, fine.apply(p, inside=True))
        for mu in range(4):
            for d, step in ((1 + 2 * mu, 1), (2 + 2 * mu, -1)):
                m[:, d, :, j] = fine.restrict(q, fine.hop(p, mu, step) * fine.crossing(mu, step))
    v = torch.stack([fine.unagg(q[:, :, k]) for k in range(nv)])
    return [v, m]
