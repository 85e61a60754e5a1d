"""The work that users of this framework have it do, as cases that can be timed.

Every case is one call (or the short sequence of calls) that a program makes
through the public Python entry points, on inputs made from a seed:

  poisson      a constant-coefficient Poisson problem solved with a cascade
               that the program keeps (many right-hand sides, one operator)
  step         one problem from scratch: hierarchy, cascade and solve
  variable     a variable-coefficient problem solved with a kept cascade
  batch        many uneven 2D problems with several right-hand sides each,
               solved together through a kept plan
  rhs          one cascade step of a block smoother on many right-hand sides
               (a building block of a caller's own cycle)
  label        exact block setup of a bilinear finite-element mesh and its
               blocks as training targets (the learned setup's data)
  general      an unstructured sparse operator (CSR) solved with a kept cascade
  gradients    loss and gradients of the learned setup's network on a minibatch
  predict      the network's forward pass over the blocks of a mesh
  gemm         the tensor-core product C = A B^T

``listed`` holds the sizes of the repository's own benchmark and tests (64^2,
256^3, 1024^2, 511^2, 8192^3, the network of 3x3 blocks) and odd, ragged ones
beside them; ``draw`` draws from the same ranges.  ``exact`` restates each
result in FP64 with plain torch.
"""
import math

import torch

import paper_2606_12577_gb300 as cmg
import problems

DEV = "cuda" if torch.cuda.is_available() else "cpu"
F64, F32 = torch.float64, torch.float32

# V-cycles (or Krylov steps) that `work` charges to one solve: what the
# listed cases take, roughly; the count of a drawn case depends on its field
CYCLES = {"poisson": 9, "step": 7, "variable": 14, "batch": 60, "general": 20}


def listed():
    return [
        # the smallest solve: a 2D model problem on a grid that fits any cache, FP64 throughout; all
        # latency and launches (a user's inner solve inside a larger program)
        {"name": "poisson2d_64_fp64", "family": "poisson", "dim": 2, "nx": 64, "ny": 64, "nz": 1, "kind": "additive",
         "nu": 3, "mu": 1, "method": "stationary", "precision": "fp64"},
        # an ordinary 3D model problem on an odd side, FP64 throughout, red-black cascade
        {"name": "poisson3d_127_redblack_fp64", "family": "poisson", "dim": 3, "nx": 127, "ny": 127, "nz": 127,
         "kind": "multiplicative", "nu": 2, "mu": 1, "method": "stationary", "precision": "fp64"},
        # the benchmark's workload, time to solution from the operator and the right-hand side alone
        {"name": "step3d_256", "family": "step", "dim": 3, "nx": 256, "ny": 256, "nz": 256, "kind": "additive",
         "nu": 3, "mu": 2, "method": "refine", "precision": "fp32"},
        # a heterogeneous 3D medium on a ragged grid, FP32 cycles in FP64 refinement
        {"name": "variable3d_ragged_refine", "family": "variable", "dim": 3, "nx": 230, "ny": 201, "nz": 177,
         "kind": "additive", "nu": 3, "mu": 2, "method": "refine", "precision": "fp32", "contrast": 1.0},
        # a heterogeneous 2D medium, Krylov solve around FP32 cycles
        {"name": "variable2d_1023_gmres", "family": "variable", "dim": 2, "nx": 1023, "ny": 1023, "nz": 1,
         "kind": "multiplicative", "nu": 3, "mu": 1, "method": "gmres_right", "precision": "fp32", "contrast": 1.0},
        # many uneven 2D problems, 1..8 right-hand sides each (parameter studies)
        {"name": "batch_16_gmres", "family": "batch", "problems": 16, "nmin": 33, "nmax": 257, "mmax": 8, "nu": 3,
         "method": "gmres_right", "contrast": 2.0},
        # 32 right-hand sides of the elliptic interface problem, one 2x2-block step in FP32
        {"name": "rhs32_interface_1024", "family": "rhs", "n": 1024, "nrhs": 32, "count": 200},
        # one training mesh of the learned setup: 3x3 blocks, depth 3
        {"name": "label_q1_511", "family": "label", "n": 511, "bs": 3, "nu": 3},
        # an unstructured mesh in CSR form, FP64
        {"name": "general_q1_255_gmres", "family": "general", "n": 255, "kind": "additive", "nu": 2, "blocks": False},
        # a training minibatch of the 3x3-block network, and its inference over a 511^2 mesh's blocks
        {"name": "gradients_4096", "family": "gradients", "batch": 4096, "nin": 225, "nhid": 256, "nout": 243},
        {"name": "predict_29241", "family": "predict", "batch": 29241, "nin": 225, "nhid": 256, "nout": 243},
        # a large dense product on the tensor cores
        {"name": "gemm_8192", "family": "gemm", "m": 8192, "n": 8192, "k": 8192},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    family = rng.choice(["poisson", "poisson", "step", "variable", "variable", "batch", "rhs", "label", "general",
                         "gradients", "predict", "gemm"])
    if family in ("poisson", "step", "variable"):
        dim = 3 if family == "step" else rng.choice([2, 3])
        base = _log(rng, 33, 1023) if dim == 2 else _log(rng, 33, 256 if family == "step" else 200)
        n = [max(24, int(base * rng.uniform(0.75, 1.0))) for _ in range(dim)] + [1] * (3 - dim)
        kind = "additive" if family == "step" else rng.choice(["additive", "multiplicative"])
        method = rng.choice(["stationary", "gmres_right"]) if family == "poisson" else "refine"
        precision = "fp64" if family == "poisson" else "fp32"
        if family == "variable":
            method = rng.choice(["refine", "gmres_right"])
        case = {"family": family, "dim": dim, "nx": n[0], "ny": n[1], "nz": n[2], "kind": kind,
                "nu": rng.randint(1, 2) if kind == "multiplicative" else rng.randint(2, 3), "mu": rng.randint(1, 2),
                "method": method, "precision": precision}
        if family == "variable":
            case["contrast"] = rng.choice([0.5, 1.0])
        return case
    if family == "batch":
        return {"family": family, "problems": rng.randint(4, 16), "nmin": 33, "nmax": rng.randint(65, 257),
                "mmax": rng.randint(1, 8), "nu": rng.randint(2, 3), "method": rng.choice(["gmres", "gmres_right"]),
                "contrast": rng.choice([1.0, 2.0])}
    if family == "rhs":
        return {"family": family, "n": _log(rng, 100, 1024), "nrhs": rng.randint(1, 32), "count": 200}
    if family == "label":
        return {"family": family, "n": _log(rng, 63, 511), "bs": rng.choice([2, 3]), "nu": rng.randint(2, 3)}
    if family == "general":
        return {"family": family, "n": _log(rng, 63, 255), "kind": rng.choice(["additive", "multiplicative"]),
                "nu": rng.randint(1, 2), "blocks": rng.choice([False, True])}
    if family in ("gradients", "predict"):
        top = 4096 if family == "gradients" else 32768
        return {"family": family, "batch": _log(rng, 257, top), "nin": 225, "nhid": rng.choice([128, 256]),
                "nout": 243}
    return {"family": "gemm", "m": _log(rng, 100, 8192), "n": _log(rng, 100, 8192), "k": 8 * _log(rng, 16, 1024)}


# ------------------------------------------------------------------- inputs
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _uniform(g, *shape, dtype=F64):
    return torch.rand(*shape, generator=g, device=DEV, dtype=dtype) * 2 - 1


def _star(dim):
    offs = [(0, 0, 0)]
    for d in range(dim):
        for s in (-1, 1):
            offs.append(tuple(s if k == d else 0 for k in range(3)))
    return offs


def _shift(a, axis, k):
    """a moved by k along an axis with zeros shifted in: out[i] = a[i + k]."""
    out = torch.zeros_like(a)
    m = a.shape[axis]
    if k > 0:
        out.narrow(axis, 0, m - k).copy_(a.narrow(axis, k, m - k))
    elif k < 0:
        out.narrow(axis, -k, m + k).copy_(a.narrow(axis, 0, m + k))
    else:
        out.copy_(a)
    return out


def _poisson(shape):
    """Coefficients [2 d + 1, nz, ny, nx] of the finite-difference Laplacian; shape (nz, ny, nx)."""
    dim = 2 if shape[0] == 1 else 3
    w = float(max(shape) + 1) ** 2
    c = torch.full((2 * dim + 1,) + shape, -w, dtype=F64, device=DEV)
    c[0] = 2 * dim * w
    for d in range(dim):
        axis = 2 - d
        c[1 + 2 * d].select(axis, 0).zero_()
        c[2 + 2 * d].select(axis, shape[axis] - 1).zero_()
    return c


def _finite_volume(mu, dim):
    """Coefficients of -div(mu grad u) on the interior nodes; mu on the cells, (nz + 1, ny + 1, nx + 1) or, in
    2D, (ny + 1, nx + 1): an edge takes the mean of the cells that share it."""
    m = mu if dim == 3 else mu[None]
    n = [m.shape[k] - 1 if (dim == 3 or k > 0) else 1 for k in range(3)]
    c = torch.zeros((2 * dim + 1, n[0], n[1], n[2]), dtype=F64, device=DEV)
    h2 = float(max(m.shape)) ** 2
    for d in range(dim):
        axis = 2 - d
        e = m
        for other in range(3):
            if other != axis and (dim == 3 or other > 0):
                k = e.shape[other] - 1
                e = 0.5 * (e.narrow(other, 0, k) + e.narrow(other, 1, k))
        k = e.shape[axis] - 1
        lo, hi = e.narrow(axis, 0, k) * h2, e.narrow(axis, 1, k) * h2
        c[0] += lo + hi
        c[1 + 2 * d] = -lo
        c[2 + 2 * d] = -hi
        c[1 + 2 * d].select(axis, 0).zero_()
        c[2 + 2 * d].select(axis, n[axis] - 1).zero_()
    return c


def _log_uniform_field(g, ny, nx, corr, contrast):
    """Correlated 2D cell coefficients with a log-uniform marginal on [10^-contrast, 10^contrast]."""
    py, px = ny + int(6 * corr), nx + int(6 * corr)
    w = torch.randn(py, px, generator=g, device=DEV, dtype=F64)
    ky = 2 * math.pi * torch.fft.fftfreq(py, device=DEV, dtype=F64)
    kx = 2 * math.pi * torch.fft.fftfreq(px, device=DEV, dtype=F64)
    f = torch.fft.ifft2(torch.fft.fft2(w) * torch.exp(-0.25 * corr * corr * (ky[:, None] ** 2 + kx[None] ** 2))).real
    f = f[:ny, :nx]
    f = (f - f.mean()) / f.std()
    return 10.0 ** (contrast * (2 * torch.special.ndtr(f) - 1))


def _inclusions(g, n, count):
    """The interface problem's cells: background 1, circular inclusions of 10^U[-4, 4]."""
    u = torch.rand(count, 4, generator=g, device=DEV, dtype=F64).cpu()
    x = (torch.arange(n + 1, device=DEV, dtype=F64) + 0.5) / (n + 1)
    mu = torch.ones(n + 1, n + 1, dtype=F64, device=DEV)
    for cx, cy, r, p in u.tolist():
        rad = (8 + 56 * r) / (n + 1)
        mu[(x[None] - cx) ** 2 + (x[:, None] - cy) ** 2 <= rad * rad] = 10.0 ** (8 * p - 4)
    return mu


def _shape(case):
    return (case["nz"], case["ny"], case["nx"])


def _operator(case, g):
    """(coefficients [nst, nz, ny, nx], offsets) of a poisson, step or variable case."""
    shape = _shape(case)
    if case["family"] != "variable":
        return _poisson(shape), _star(case["dim"])
    if case["dim"] == 3:
        mu = 10.0 ** (case["contrast"] * _uniform(g, *[m + 1 for m in shape]))
    else:
        mu = _log_uniform_field(g, shape[1] + 1, shape[2] + 1, 8.0, case["contrast"])
    return _finite_volume(mu, case["dim"]), _star(case["dim"])


def _hierarchy(c, offs, **kw):
    dim = 2 if len(offs) in (5, 9) else 3
    nz, ny, nx = c.shape[1:]
    return cmg.setup_hierarchy(dim, (nx, ny, nz), offs, c.reshape(len(offs), -1), **kw)


def _batch_inputs(case, seed):
    """[(coefficients, nrhs, b)] of the batch's problems: sides and right-hand-side counts are the case's own, the
    fields and right-hand sides the seed's."""
    P = case["problems"]
    u = problems.uniform01(97, 2 * P).reshape(P, 2)
    out = []
    for k in range(P):
        n = case["nmin"] + int(u[k, 0] * (case["nmax"] - case["nmin"] + 1))
        m = 1 + int(u[k, 1] * case["mmax"])
        g = _gen(1000 * seed + k)
        c = _finite_volume(_log_uniform_field(g, n + 1, n + 1, 8.0, case["contrast"]), 2)
        out.append((c, m, _uniform(g, n * n * m)))
    return out


def _rhs_inputs(case, seed):
    g = _gen(seed)
    n, m = case["n"], case["nrhs"]
    c = _finite_volume(_inclusions(g, n, case["count"]), 2)
    return c, _uniform(g, n * n, m, dtype=F32), _uniform(g, n * n, m, dtype=F32)


def _network(case, g):
    """He-uniform weights [W1, b1, W2, b2, W3, b3] (FP32), small biases."""
    i, h, o = case["nin"], case["nhid"], case["nout"]
    out = []
    for r, c in ((h, i), (h, h), (o, h)):
        out += [_uniform(g, r, c, dtype=F32) * math.sqrt(6.0 / c), 0.05 * _uniform(g, r, dtype=F32)]
    return out


def _network_inputs(case, seed):
    """Weights, features and targets: rows of a prescaled operator (a unit diagonal, small couplings) and blocks of
    the size of its inverse's."""
    g = _gen(seed)
    p = _network(case, g)
    X = 0.3 * _uniform(g, case["batch"], case["nin"], dtype=F32)
    X = torch.where(torch.rand(X.shape, generator=g, device=DEV) < 0.7, torch.zeros_like(X), X)
    T = 0.5 * _uniform(g, case["batch"], case["nout"], dtype=F32)
    return p, X, T


def _gemm_inputs(case, seed):
    g = _gen(seed)
    return (_uniform(g, case["m"], case["k"], dtype=F32).bfloat16(),
            _uniform(g, case["n"], case["k"], dtype=F32).bfloat16())


def _general(case, seed):
    u = problems.unstructured_q1(case["n"], 100 + seed % 100000)
    return u, _uniform(_gen(seed), u["A"].shape[0])


# ------------------------------------------------------------ prepare and run
def prepare(case, seed):
    f = case["family"]
    s = {"case": case}
    if f in ("poisson", "step", "variable"):
        g = _gen(seed)
        c, offs = _operator(case, g)
        s["b"] = _uniform(g, c[0].numel())
        if f == "step":
            s["coeff"], s["offs"] = c, offs
        else:
            s["h"] = _hierarchy(c, offs)
            s["c"] = cmg.setup_cascade(s["h"], case["kind"], nu=case["nu"], lowp=case["precision"] == "fp32")
    elif f == "batch":
        P = _batch_inputs(case, seed)
        s["m"], s["b"] = [m for _, m, _ in P], [b for _, _, b in P]
        s["h"] = [_hierarchy(c, _star(2)) for c, _, _ in P]
        s["c"] = [cmg.setup_cascade(h, "multiplicative", nu=case["nu"], lowp=True) for h in s["h"]]
        s["plan"] = cmg.Batch(s["h"], s["c"], s["m"], precision="fp32", method=case["method"])
    elif f == "rhs":
        c, s["b"], s["x"] = _rhs_inputs(case, seed)
        s["h"] = _hierarchy(c, _star(2), block=2)
        s["c"] = cmg.setup_cascade(s["h"], "additive", nu=1, lowp=True)
        s["out"] = torch.empty_like(s["x"])
    elif f == "label":
        A = problems.q1_jittered(case["n"], 5000 + seed % 100000)
        s["coeff"] = torch.tensor(A.coeff, device=DEV).reshape(9, 1, case["n"], case["n"])
        s["offs"] = A.offsets
    elif f == "general":
        u, s["b"] = _general(case, seed)
        s["h"] = cmg.gsetup_hierarchy(u["A"], u["Ps"], rscale=0.25, blocks=u["blocks"] if case["blocks"] else None,
                                      seed=3)
        s["c"] = cmg.gsetup_cascade(s["h"], case["kind"], nu=case["nu"])
    elif f in ("gradients", "predict"):
        p, s["X"], s["T"] = _network_inputs(case, seed)
        s["net"] = cmg.MLP(case["nin"], case["nhid"], case["nout"], max_batch=32768 if f == "predict" else 4096)
        s["net"].set_params(torch.cat([t.reshape(-1) for t in p]).cpu().numpy())
    else:
        s["A"], s["B"] = _gemm_inputs(case, seed)
    return s


def run(s):
    case = s["case"]
    f = case["family"]
    if f in ("poisson", "step", "variable"):
        if f == "step":
            h = _hierarchy(s["coeff"], s["offs"])
            c = cmg.setup_cascade(h, case["kind"], nu=case["nu"], lowp=True, setup_precision="fp32")
        else:
            h, c = s["h"], s["c"]
        x = torch.zeros_like(s["b"])
        cmg.solve(h, c, s["b"], x, method=case["method"], precision=case["precision"], tol=1e-10, maxit=200,
                  mu_pre=case["mu"], mu_post=case["mu"], order="RF")
        return x
    if f == "batch":
        xs = [torch.zeros_like(b) for b in s["b"]]
        s["plan"].solve(s["b"], xs, tol=1e-10, maxit=400)
        return xs
    if f == "rhs":
        cmg.sweep_rhs(s["h"], s["c"], 0, 0, s["b"], s["x"], s["out"], case["nrhs"])
        return s["out"]
    if f == "label":
        h = _hierarchy(s["coeff"], s["offs"], block=case["bs"], max_levels=1)
        c = cmg.setup_cascade(h, "additive", nu=case["nu"])
        return cmg.block_features(h, 0), cmg.block_targets(c, 0)
    if f == "general":
        x = torch.zeros_like(s["b"])
        cmg.gsolve(s["h"], s["c"], s["b"], x, method="gmres_right", tol=1e-10, maxit=200)
        return x
    if f == "gradients":
        return s["net"].gradients(s["X"], s["T"])
    if f == "predict":
        return s["net"].forward(s["X"])
    return cmg.tc_gemm_bf16(s["A"], s["B"])


def work(case):
    """The bytes of the inputs and outputs of one pass, each once, and its arithmetic: a solve is charged the
    sweeps of CYCLES cycles over all levels, a setup the products of its least squares."""
    f = case["family"]
    if f in ("poisson", "step", "variable"):
        N, dim = case["nx"] * case["ny"] * case["nz"], case["dim"]
        w = 4 if case["precision"] == "fp32" else 8
        nst = 2 * dim + 1
        sweeps = 2 * case["mu"] * case["nu"] * CYCLES[f] * (1 + 1 / (2 ** dim - 1))
        op = 8 * nst if f == "step" else (w * (nst + case["nu"]))
        return {"bytes": N * (op + 16.0), "flops": N * sweeps * (2.0 * nst + 3)}
    if f == "batch":
        u = problems.uniform01(97, 2 * case["problems"]).reshape(-1, 2)
        got = {"bytes": 0.0, "flops": 0.0}
        for a, c in u:
            n = case["nmin"] + int(a * (case["nmax"] - case["nmin"] + 1))
            m = 1 + int(c * case["mmax"])
            got["bytes"] += n * n * (4.0 * (5 + case["nu"]) + 16.0 * m)
            got["flops"] += n * n * m * CYCLES[f] * 4 / 3 * 2 * case["nu"] * 13.0
        return got
    if f == "rhs":
        N, m = case["n"] ** 2, case["nrhs"]
        return {"bytes": N * 4.0 * (5 + 4 + 3 * m), "flops": N * m * 2.0 * (5 + 4)}
    if f == "label":
        N, q = case["n"] ** 2, case["bs"] ** 2
        b = 4.0 * N * ((case["bs"] + 2) ** 2 + case["nu"] * q)
        cols = [(case["bs"] * (2 * k + 1) + 2) ** 2 for k in range(case["nu"])]
        return {"bytes": 72.0 * N + b, "flops": sum(N * 2.0 * c * (9 + 2.5 * q) for c in cols)}
    if f == "general":
        N = case["n"] ** 2
        lam = 9 * N if case["blocks"] else N
        return {"bytes": N * (9 * 12.0 + 16) + 8.0 * case["nu"] * lam,
                "flops": N * CYCLES[f] * 4 / 3 * 2 * case["nu"] * (18.0 + 2 * lam / N)}
    if f in ("gradients", "predict"):
        i, h, o, B = case["nin"], case["nhid"], case["nout"], case["batch"]
        w = i * h + h * h + h * o
        if f == "predict":
            return {"bytes": 4.0 * B * (i + o) + 2.0 * w, "flops": 2.0 * B * w}
        return {"bytes": 4.0 * B * (i + o) + 6.0 * w, "flops": 2.0 * B * (3.0 * w - i * h)}
    m, n, k = case["m"], case["n"], case["k"]
    return {"bytes": 2.0 * (m + n) * k + 4.0 * m * n, "flops": 2.0 * m * n * k}


# -------------------------------------------------------------------- exact
def _cg(apply, diag, b):
    """Jacobi-preconditioned conjugate gradients in FP64, restarted from the true residual until ||b - A x|| no
    longer falls."""
    x, nb, last = torch.zeros_like(b), float(b.norm()), math.inf
    for _ in range(6):
        r = b - apply(x)
        rn = float(r.norm())
        if rn <= 2e-15 * nb or rn > 0.5 * last:
            break
        last = rn
        z = r / diag
        p, rz = z.clone(), torch.dot(r.flatten(), z.flatten())
        for k in range(20000):
            q = apply(p)
            a = rz / torch.dot(p.flatten(), q.flatten())
            x += a * p
            r -= a * q
            if k % 20 == 19 and float(r.norm()) <= max(1e-15 * nb, 1e-7 * rn):
                break
            z = r / diag
            new = torch.dot(r.flatten(), z.flatten())
            p = z + (new / rz) * p
            rz = new
    return x


def _stencil_apply(c, offs):
    def apply(x):
        y = c[0] * x
        for s, (dx, dy, dz) in enumerate(offs):
            if s:
                axis, k = (2, dx) if dx else (1, dy) if dy else (0, dz)
                m = x.shape[axis] - 1
                to, of = (0, 1) if k > 0 else (1, 0)
                y.narrow(axis, to, m).addcmul_(c[s].narrow(axis, to, m), x.narrow(axis, of, m))
        return y
    return apply


def _solve(c, offs, b):
    return _cg(_stencil_apply(c, offs), c[0], b.reshape(c[0].shape)).reshape(-1)


def _block_cascade(c, offs, bs, nu):
    """The additive block cascade of a 2D operator in FP64: Lambda~_l [nu, nblocks, bs^2, bs^2] on the prescaled
    operator, and the scales w [ny, nx].  The rows E and R of a block are kept over the block's own window of
    columns, (bs + 2 r)^2 nodes."""
    ny, nx = c.shape[-2:]
    c = c.reshape(len(offs), ny, nx)
    centre = offs.index((0, 0, 0))
    w = c[centre].rsqrt()
    nby, nbx = -(-ny // bs), -(-nx // bs)
    py, px = nby * bs, nbx * bs
    At = torch.zeros(len(offs), py, px, dtype=F64, device=DEV)
    for s, (dx, dy, _) in enumerate(offs):
        At[s, :ny, :nx] = w * c[s] * _shift(_shift(w, 0, dy), 1, dx)
    rad = (nu - 1) * bs + 1  # a step reaches one node into the next blocks, whose rows reach bs further each step
    W = bs + 2 * rad
    E = torch.zeros(py, px, W, W, dtype=F64, device=DEV)  # E[i] over the window of i's block
    iy = torch.arange(py, device=DEV)[:, None].expand(py, px)
    ix = torch.arange(px, device=DEV)[None].expand(py, px)
    E[iy, ix, iy % bs + rad, ix % bs + rad] = ((iy < ny) & (ix < nx)).to(F64)
    lams = []
    for _ in range(nu):
        R = torch.zeros_like(E)
        for s, (dx, dy, _) in enumerate(offs):
            # row j = i + (dy, dx) in the window of i's block: j's block may be the next one
            for ly in range(bs):
                for lx in range(bs):
                    by, bx = (ly + dy) // bs, (lx + dx) // bs
                    src = E[(ly + dy) % bs::bs, (lx + dx) % bs::bs]
                    src = _shift(_shift(src, 0, by), 1, bx)
                    src = _shift(_shift(src, 2, -by * bs), 3, -bx * bs)
                    R[ly::bs, lx::bs] += At[s, ly::bs, lx::bs, None, None] * src
        q = bs * bs

        def rows(M):
            return M.reshape(nby, bs, nbx, bs, W * W).permute(0, 2, 1, 3, 4).reshape(nby * nbx, q, W * W)
        Rb, Eb = rows(R), rows(E)
        G, C = Rb @ Rb.transpose(1, 2), Eb @ Rb.transpose(1, 2)
        ev, Q = (torch.cat(t) for t in zip(*(torch.linalg.eigh(part) for part in G.split(16384))))
        keep = ev > 1e-14 * G.diagonal(dim1=1, dim2=2).sum(1, keepdim=True)
        inv = torch.where(keep, 1.0 / torch.where(keep, ev, torch.ones_like(ev)), torch.zeros_like(ev))
        L = C @ (Q * inv[:, None]) @ Q.transpose(1, 2)
        lams.append(L)
        Eb = Eb - L @ Rb
        E = Eb.reshape(nby, nbx, bs, bs, W, W).permute(0, 2, 1, 3, 4, 5).reshape(py, px, W, W).contiguous()
    return torch.stack(lams), w


def _blocks_of(v, bs):
    """v [ny, nx, m] as [nblocks, bs^2, m], absent nodes zero."""
    ny, nx, m = v.shape
    nby, nbx = -(-ny // bs), -(-nx // bs)
    p = torch.zeros(nby * bs, nbx * bs, m, dtype=v.dtype, device=v.device)
    p[:ny, :nx] = v
    return p.reshape(nby, bs, nbx, bs, m).permute(0, 2, 1, 3, 4).reshape(nby * nbx, bs * bs, m)


def _features(c, offs, bs, w):
    ny, nx = w.shape
    win = bs + 2
    nby, nbx = -(-ny // bs), -(-nx // bs)
    F = torch.zeros(nby, nbx, bs * bs, win, win, dtype=F64, device=DEV)
    for s, (dx, dy, _) in enumerate(offs):
        a = w * c.reshape(len(offs), ny, nx)[s] * _shift(_shift(w, 0, dy), 1, dx)
        pad = torch.zeros(nby * bs, nbx * bs, dtype=F64, device=DEV)
        pad[:ny, :nx] = a
        for p in range(bs * bs):
            F[:, :, p, p // bs + dy + 1, p % bs + dx + 1] = pad[p // bs::bs, p % bs::bs]
    return F.reshape(nby * nbx, -1)


def _forward(p, X):
    W = [t.to(torch.bfloat16).to(F64) if t.dim() == 2 else t.to(F64) for t in p]
    Z1 = X.to(F64) @ W[0].T + W[1]
    H1 = Z1.clamp(min=0)
    Z2 = H1 @ W[2].T + W[3]
    H2 = Z2.clamp(min=0)
    return H2 @ W[4].T + W[5], (Z1, H1, Z2, H2, W)


def exact(case, seed):
    f = case["family"]
    if f in ("poisson", "step", "variable"):
        g = _gen(seed)
        c, offs = _operator(case, g)
        return _solve(c, offs, _uniform(g, c[0].numel()))
    if f == "batch":
        out = []
        for c, m, b in _batch_inputs(case, seed):
            cols = [_solve(c, _star(2), b.reshape(-1, m)[:, r].contiguous()) for r in range(m)]
            out.append(torch.stack(cols, 1).reshape(-1))
        return out
    if f == "rhs":
        c, b, x = _rhs_inputs(case, seed)
        n, m = case["n"], case["nrhs"]
        lam, w = _block_cascade(c, _star(2), 2, 1)
        xg, r = x.to(F64).reshape(n, n, m), -b.to(F64).reshape(n, n, m)
        for s, (dx, dy, _) in enumerate(_star(2)):
            r += c[s, 0, :, :, None] * _shift(_shift(xg, 0, dy), 1, dx)
        d = lam[0] @ _blocks_of(w[..., None] * r, 2)
        nb = -(-n // 2)
        d = d.reshape(nb, nb, 2, 2, m).permute(0, 2, 1, 3, 4).reshape(2 * nb, 2 * nb, m)[:n, :n]
        return (xg - w[..., None] * d).reshape(n * n, m)
    if f == "label":
        A = problems.q1_jittered(case["n"], 5000 + seed % 100000)
        c = torch.tensor(A.coeff, device=DEV)
        n, bs = case["n"], case["bs"]
        c = c.reshape(9, n, n)
        lam, w = _block_cascade(c, A.offsets, bs, case["nu"])
        return _features(c, A.offsets, bs, w), lam.permute(1, 0, 2, 3).reshape(lam.shape[1], -1)
    if f == "general":
        u, b = _general(case, seed)
        A = u["A"]
        M = torch.sparse_csr_tensor(torch.tensor(A.indptr).long(), torch.tensor(A.indices).long(),
                                    torch.tensor(A.data), size=A.shape).to(DEV)
        return _cg(lambda x: (M @ x[:, None])[:, 0], torch.tensor(A.diagonal(), device=DEV), b)
    if f in ("gradients", "predict"):
        p, X, T = _network_inputs(case, seed)
        Y, (Z1, H1, Z2, H2, W) = _forward(p, X)
        if f == "predict":
            return Y
        E = Y - T.to(F64)
        dY = 2 * E / E.numel()
        dZ2 = (dY @ W[4]) * (Z2 > 0)
        dZ1 = (dZ2 @ W[2]) * (Z1 > 0)
        g = [dZ1.T @ X.to(F64), dZ1.sum(0), dZ2.T @ H1, dZ2.sum(0), dY.T @ H2, dY.sum(0)]
        return float((E * E).mean()), torch.cat([t.reshape(-1) for t in g])
    A, B = _gemm_inputs(case, seed)
    return A.to(F64) @ B.to(F64).T
