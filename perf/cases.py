"""The measured cases: what a user of the library has it compute, through the public binding.

A case is a dict of plain values.  ``kind`` names the call: ``apply`` (molt_apply_D along every axis), ``heat``,
``wave``, ``hj``, ``advdiff`` (molt_step of that problem), ``batch`` (molt_step of many uneven heat problems) or
``train`` (one minibatch of the weight network: loss, gradient, Adam).  ``listed()`` holds one case of each use,
``draw(rng)`` more of the same ranges.  ``exact`` restates every call in FP64 torch, from the definitions of the
operators (quadrature by Gauss-Legendre, recurrences point by point), without the library.
"""
import math

import numpy as np
import torch

from paper_2007_03041_gb300 import molt as M

TWO_PI = 2.0 * math.pi
PREC = {"f64": M.PREC_F64, "mixed": M.PREC_F32_F64UPDATE, "f32": M.PREC_F32}
WEIGHTS = {"linear": M.W_LINEAR, "wenoz": M.W_WENOZ, "learned": M.W_LEARNED}
OPS = {"L": M.OP_L, "R": M.OP_R, "0": M.OP_0}
HAMS = {"half_sq": M.H_HALF_SQ, "linear": M.H_LINEAR, "affine_sq": M.H_AFFINE_SQ}
SSPRK3 = ((0.0, 1.0), (0.75, 0.25), (1.0 / 3.0, 2.0 / 3.0))


def _case(kind, nx, ny=1, nz=1, **more):
    c = dict(kind=kind, nx=nx, ny=ny, nz=nz, prec="f64", bc="periodic", P=1, quad=6, weights="linear", steps=1)
    c.update(more)
    return c


def listed():
    return [
        # the smallest call: the operator on a small 2-D field, as in a coupling loop or a notebook; launch latency
        _case("apply", 100, 60, name="apply_small_f64", op="0", P=2, nu=0.6, nonuniform=False),
        # the operator on a stretched periodic grid with point-local weights, along x and then y
        _case("apply", 4096, 4096, name="apply_nonuniform_4096_f32", prec="f32", op="0", P=2, nu=0.6,
              nonuniform=True),
        # 2-D heat in FP64, SSP-RK3 with P = 3: a small grid advanced by ten steps, bound by launches and latency
        _case("heat", 256, 256, name="heat_256_f64", P=3, quad=3, steps=10),
        # the first-order diffusion problem in FP64 on its odd 5277^2 grid
        _case("heat", 5277, 5277, name="diffusion_5277_f64", P=1, quad=6, integrator="euler", steps=2),
        # 64 uneven heat problems, sides 128 .. 2048, advanced together
        _case("batch", 2048, 2048, name="batch_64_mixed", prec="mixed", P=3, quad=3, count=64, sides=3, steps=2),
        # the 3-D wave equation between Dirichlet walls, FP32 sweeps with the FP64 update, at full size
        _case("wave", 512, 512, 512, name="wave_512_mixed", prec="mixed", bc="dirichlet", P=2, quad=6, steps=4),
        # the same on a grid whose sides no tile divides
        _case("wave", 201, 151, 101, name="wave_ragged_mixed", prec="mixed", bc="dirichlet", P=2, quad=6, steps=5),
        # Hamilton-Jacobi with WENO-Z weights and the lagged adaptive time step, FP32
        _case("hj", 4096, 4096, name="hj_4096_wenoz_f32", prec="f32", quad=5, weights="wenoz", ham="half_sq",
              cfl=1.5, steps=4),
        # the same with the weights of the network (WENO-Z where the two differ), at full size
        _case("hj", 8192, 8192, name="hj_8192_learned_f32", prec="f32", quad=5, weights="learned", ham="half_sq",
              cfl=1.5, steps=1),
        # H = (1 + u_x + u_y)^2 / 2 with a manufactured source, FP64, on one of that problem's odd grids
        _case("hj", 1759, 1759, name="hj_source_1759_f64", quad=6, ham="affine_sq", cfl=1.0, steps=4),
        # viscous Burgers by flux splitting, WENO-Z weights, FP32
        _case("advdiff", 4096, 4096, name="burgers_4096_wenoz_f32", prec="f32", quad=5, weights="wenoz",
              flux="burgers", integrator="euler", steps=1),
        # one minibatch of the weight network's training: forward, backward, Adam
        _case("train", 16384, name="train_16384", prec="f32", weights="learned"),
    ]


def _log_size(rng, lo, hi):
    """A size spread over the logarithm of lo..hi: a power of two, a multiple of 16 or any (odd) number."""
    n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    how = rng.randrange(3)
    if how == 0:
        n = 1 << max(1, round(math.log2(n)))
    elif how == 1:
        n = max(16, n // 16 * 16)
    else:
        n |= 1
    return max(lo, min(hi, n))


def draw(rng):
    kind = rng.choice(["apply", "apply", "apply_nu", "heat", "diffusion", "batch", "wave", "hj", "hj_learned",
                       "hj_source", "advdiff", "train"])
    if kind == "apply":
        nd = rng.choice([1, 2, 3])
        hi = {1: 8192, 2: 4096, 3: 256}[nd]
        n = [_log_size(rng, 32, hi) for _ in range(nd)]
        return _case("apply", *n, prec=rng.choice(["f64", "mixed", "f32"]), bc=rng.choice(["periodic", "dirichlet"]),
                     op=rng.choice(["L", "R", "0"]), P=rng.choice([1, 2, 3]), quad=rng.choice([3, 5, 6]),
                     nu=round(rng.uniform(0.1, 1.2), 3), nonuniform=False)
    if kind == "apply_nu":
        weno = rng.random() < 0.4
        return _case("apply", _log_size(rng, 64, 4096), _log_size(rng, 64, 4096), prec=rng.choice(["f64", "f32"]),
                     bc=rng.choice(["periodic", "dirichlet"]), op=rng.choice(["L", "R", "0"]),
                     P=rng.choice([1, 2]), quad=5 if weno else rng.choice([3, 5, 6]),
                     weights="wenoz" if weno else "linear", nu=0.6, nonuniform=True)
    if kind == "heat":
        n = _log_size(rng, 64, 1024)
        return _case("heat", n, n, prec=rng.choice(["f64", "mixed"]), P=3, quad=3, steps=rng.choice([1, 2, 5]))
    if kind == "diffusion":
        n = _log_size(rng, 512, 4096)
        return _case("heat", n, n, prec=rng.choice(["f64", "mixed"]), P=1, quad=6, integrator="euler",
                     steps=rng.choice([1, 2]))
    if kind == "batch":
        return _case("batch", 2048, 2048, prec="mixed", P=3, quad=3, count=rng.randrange(4, 49),
                     sides=rng.randrange(1000), steps=rng.choice([1, 2]))
    if kind == "wave":
        n = [_log_size(rng, 32, 400) for _ in range(3)]
        return _case("wave", *n, prec="mixed", bc="dirichlet", P=2, quad=6, steps=rng.choice([1, 2, 5]))
    if kind == "hj":
        n = _log_size(rng, 256, 4096)
        weno = rng.random() < 0.7
        prec = "f32" if n > 2048 else rng.choice(["f32", "f32", "f64"])
        return _case("hj", n, n, prec=prec, quad=5, weights="wenoz" if weno else "linear", ham="half_sq", cfl=1.5,
                     steps=rng.choice([1, 2, 4]))
    if kind == "hj_learned":
        n = _log_size(rng, 256, 4096)
        return _case("hj", n, n, prec="f32", quad=5, weights="learned", ham="half_sq", cfl=1.5,
                     steps=rng.choice([1, 2]))
    if kind == "hj_source":
        n = _log_size(rng, 256, 2500)
        return _case("hj", n, n, prec=rng.choice(["f64", "f32"]), quad=6, ham=rng.choice(["affine_sq", "linear"]),
                     cfl=1.0, steps=rng.choice([1, 2, 4]))
    if kind == "advdiff":
        n = _log_size(rng, 128, 2500)
        weno = rng.random() < 0.6
        prec = rng.choice(["f64", "f32"]) if weno else rng.choice(["f64", "mixed", "f32"])
        return _case("advdiff", n, n, prec=prec, quad=5 if weno else 6, weights="wenoz" if weno else "linear",
                     flux=rng.choice(["burgers", "linear"]), integrator="euler", steps=rng.choice([1, 2]))
    return _case("train", rng.randrange(1024, 65536) // 4 * 4, prec="f32", weights="learned")


# ------------------------------------------------------------------- problems
def _shape(case):
    return [case[k] for k in ("nx", "ny", "nz") if case[k] > 1]


def _lengths(case):
    """Length of the domain along every axis ([0, length])."""
    wide = case["kind"] in ("hj", "advdiff", "apply") or (case["kind"] == "heat" and case.get("integrator") == "euler")
    return [TWO_PI if wide else 1.0] * len(_shape(case))


def _spacings(case):
    return [L / (n if case["bc"] == "periodic" else n - 1) for n, L in zip(_shape(case), _lengths(case))]


def _nodes(case, n):
    """The stretched nodes of a non-uniform axis (one period, or both ends included)."""
    if case["bc"] == "periodic":
        xi = TWO_PI * np.arange(n) / n
        return xi + 0.3 * np.sin(xi)
    t = np.linspace(0.0, 1.0, n)
    x = TWO_PI * (t + 0.3 * np.sin(TWO_PI * t) / TWO_PI)
    x[0], x[-1] = 0.0, TWO_PI
    return x


def _dt(case):
    h = min(_spacings(case))
    if case["kind"] == "wave":
        return 2.0 * h
    if case["kind"] == "heat" and case.get("integrator") == "euler":
        return h
    if case["kind"] == "advdiff":
        return 0.5 * h / 1.2
    return 0.5 * h


def _beta(case):
    return {"heat": 1.0 if case.get("integrator") == "euler" else 0.6, "batch": 0.6, "wave": 0.8, "advdiff": 0.6}.get(
        case["kind"], 1.0)


def _kappa(case):
    return 2e-3 if case["kind"] == "advdiff" else 1.0


def _velocity(case):
    return (1.0, 0.5, 0.0) if case["kind"] == "advdiff" else (1.0, 1.0, 1.0)


def _alpha(case):
    """alpha of the ``apply`` cases: nu over the mean spacing of every axis."""
    return [case["nu"] / h for h in _spacings(case)]


def _desc(case):
    pde = {"heat": M.PDE_HEAT, "batch": M.PDE_HEAT, "wave": M.PDE_WAVE, "hj": M.PDE_HJ, "advdiff": M.PDE_ADVDIFF,
           "apply": M.PDE_HEAT}[case["kind"]]
    nd = len(_shape(case))
    bc = M.BC_PERIODIC if case["bc"] == "periodic" else M.BC_DIRICHLET
    return M.make_desc(_shape(case), lo=[0.0] * nd, hi=_lengths(case), bc=[bc] * nd, P=case["P"],
                       quad_points=case["quad"], weights=WEIGHTS[case["weights"]], beta=_beta(case), pde=pde,
                       c=1.2 if case["kind"] == "advdiff" else 1.0, diffusivity=_kappa(case),
                       cfl=case.get("cfl", 1.0), dt=0.0 if case["kind"] == "hj" else _dt(case),
                       prec=PREC[case["prec"]], hamiltonian=HAMS[case.get("ham", "half_sq")],
                       velocity=_velocity(case), h0=1.0 if case.get("ham") == "affine_sq" else 0.0,
                       integrator=M.INT_EULER if case.get("integrator") == "euler" else M.INT_DEFAULT,
                       flux=M.FLUX_BURGERS if case.get("flux") == "burgers" else M.FLUX_LINEAR)


def _batch_sides(case):
    g = np.random.Generator(np.random.PCG64(case["sides"]))
    return [int(s) for s in g.choice([128, 256, 512, 1024, 2048], size=case["count"])]


def _batch_cases(case):
    return [dict(case, kind="heat", nx=s, ny=s) for s in _batch_sides(case)]


# --------------------------------------------------------------------- inputs
def _axes(case):
    """FP64 coordinates of every axis, shaped to broadcast over [z][y][x]."""
    n = _shape(case)
    out = []
    for k, (m, h) in enumerate(zip(n, _spacings(case))):
        x = torch.arange(m, dtype=torch.float64, device="cuda") * h
        out.append(x.reshape([-1 if len(n) - 1 - d == k else 1 for d in range(len(n))]))
    return out


def _state_dtype(case):
    return torch.float32 if case["prec"] == "f32" else torch.float64


def _field(case, seed):
    """The initial state of a case from its seed."""
    g = np.random.Generator(np.random.PCG64(seed))
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    ax = _axes(case)
    shape = tuple(reversed(_shape(case)))
    u = torch.zeros(shape, dtype=torch.float64, device="cuda")
    if case["kind"] == "wave":
        for _ in range(16):                              # Gaussian bumps, zero on the walls
            c, s = g.uniform(0.0, 1.0, size=3), g.uniform(0.02, 0.1)
            b = None
            for k, x in enumerate(ax):
                e = torch.exp(-(x - c[k]) ** 2 / (2 * s * s))
                b = e if b is None else b * e
            u += b
        for d in range(u.ndim):
            u.select(d, 0).zero_()
            u.select(d, u.shape[d] - 1).zero_()
    elif case["kind"] == "heat":
        u += 1.0                                         # a mean temperature and eight Fourier modes
        w = TWO_PI / _lengths(case)[0]
        for _ in range(8):
            k, a = g.integers(1, 9, size=2), 0.1 * g.standard_normal()
            u += a * torch.cos(w * (int(k[0]) * ax[0] + int(k[1]) * ax[1]))
    elif case["kind"] == "hj" and case.get("ham") == "affine_sq":
        a = 0.02 * g.standard_normal(2)                  # near the manufactured solution's zero state
        u += a[0] * torch.sin(ax[0]) + a[1] * torch.sin(ax[1])
    elif case["kind"] == "hj" and case.get("ham") == "linear":
        p = g.uniform(0.0, TWO_PI, size=2)
        u += 0.25 * (1 - torch.cos(ax[0] - p[0])) * (1 - torch.cos(ax[1] - p[1]))
    elif case["kind"] == "hj":
        p = g.uniform(0.0, TWO_PI, size=2)
        u += -torch.cos(ax[0] - p[0]) - torch.cos(ax[1] - p[1])
        u += 1e-3 * torch.randn(shape, generator=gen, dtype=torch.float64, device="cuda")
    elif case["kind"] == "advdiff":
        p = g.uniform(0.0, TWO_PI, size=2)
        u += 0.3 + 0.5 * torch.sin(ax[0] - p[0]) * torch.sin(ax[1] - p[1])
    else:
        for k, x in enumerate(ax):                       # smooth along every axis, with noise
            u += g.uniform(0.5, 1.5) * torch.cos(x * (1 + k) + g.uniform(0.0, TWO_PI))
        u += 0.1 * torch.randn(shape, generator=gen, dtype=torch.float64, device="cuda")
    return u.to(_state_dtype(case))


def _source(case):
    """F_k of F(x, t) = sum_k t^k F_k(x) for u = t (sin x + sin y), H = (1 + u_x + u_y)^2 / 2."""
    x, y = _axes(case)
    c = torch.cos(x) + torch.cos(y)
    return torch.stack([torch.sin(x) + torch.sin(y) + 0.5, c, 0.5 * c * c]).to(_state_dtype(case))


def _stencils(n, seed):
    """(n, 5) stencils of smooth, noisy, kinked and jumping data, and their WENO-Z weights as targets."""
    g = np.random.Generator(np.random.PCG64(seed))
    j = np.arange(-2, 3, dtype=np.float64)
    kind = g.integers(0, 4, size=(n, 1))
    a = g.uniform(0.5, 2.0, size=(n, 1)) * g.choice([-1.0, 1.0], size=(n, 1))
    x0 = g.uniform(-2.0, 2.0, size=(n, 1))
    smooth = a * np.sin(g.uniform(0.5, 4.0, size=(n, 1)) * 2e-3 * j + g.uniform(0.0, TWO_PI, size=(n, 1)))
    x = np.select([kind == 0, kind == 1, kind == 2], [smooth, smooth + 1e-3 * g.standard_normal((n, 5)),
                                                      a * np.abs(j - x0)], a * (j > x0))
    x = (x + g.uniform(-2.0, 2.0, size=(n, 1))).astype(np.float32).astype(np.float64)
    w = _wenoz_weights([x[:, k] for k in range(5)], _uniform_rule(1.0 / 1.5, 5))
    return x, np.ascontiguousarray(w.T)


def _split(theta):
    """W1, b1, W2, b2, W3, b3 of the 1347 master parameters."""
    out, k = [], 0
    for s in ((32, 5), (32,), (32, 32), (32,), (3, 32), (3,)):
        m = int(np.prod(s))
        out.append(theta[k:k + m].reshape(s))
        k += m
    return out


def _gelu(z):
    return 0.5 * z * (1.0 + torch.tanh(math.sqrt(2.0 / math.pi) * (z + 0.044715 * z ** 3)))


def _round_bf16(x):
    """x rounded to BF16, the rounding taken as the identity by derivatives."""
    return x + (x.detach().to(torch.float32).to(torch.bfloat16).to(x.dtype) - x.detach())


def _network(theta, x, rnd=_round_bf16):
    """Hidden activations and outputs of the network on raw stencils x (n, 5) in x's type; ``rnd`` rounds the inputs of
    every product (the network is defined with BF16 operands)."""
    d = x - x[:, 2:3]
    d = rnd(d / (d.abs().amax(dim=1, keepdim=True) + 1e-30))
    w1, b1, w2, b2, w3, b3 = _split(theta)
    a = rnd(_gelu(rnd(_gelu(d @ w1.T + b1)) @ w2.T + b2))
    return a, torch.softmax(a @ w3.T + b3, dim=1)


_network_kept = []


def _network_params():
    """The network that the learned cases run: seeded random hidden layers, the output layer fitted by least squares
    to the logarithms of the WENO-Z weights (a fixed network, the same in every program that runs these cases)."""
    if not _network_kept:
        g = np.random.Generator(np.random.PCG64(50))
        theta = np.concatenate([g.standard_normal(160) * math.sqrt(2.0 / 5), 0.1 * g.standard_normal(32),
                                g.standard_normal(1024) * math.sqrt(2.0 / 32), 0.1 * g.standard_normal(32),
                                np.zeros(99)])
        x, w = _stencils(20000, 51)
        a, _ = _network(torch.tensor(theta), torch.tensor(x), lambda v: v)
        A = np.concatenate([a.numpy(), np.ones((len(x), 1))], axis=1)
        logits = np.log(np.maximum(w, 1e-4))
        sol = np.linalg.solve(A.T @ A + 1e-3 * np.eye(33), A.T @ (logits - logits.mean(axis=1, keepdims=True)))
        theta[1248:1344] = sol[:32].T.reshape(-1)
        theta[1344:] = sol[32]
        _network_kept.append(theta.astype(np.float32))
    return _network_kept[0]


def _bf16(theta):
    return theta.to(torch.float32).to(torch.bfloat16).to(torch.float64)


class State:
    """What a program holds between calls: its context and arrays."""

    def __init__(self):
        self.ctx = None

    def __del__(self):
        if self.ctx is not None:
            M.molt_destroy(self.ctx)


def prepare(case, seed):
    s = State()
    s.case = case
    if case["kind"] == "train":
        n = case["nx"]
        x, y = _stencils(n, seed)
        g = np.random.Generator(np.random.PCG64(seed + 1))
        f32 = dict(dtype=torch.float32, device="cuda")
        s.x, s.y = torch.tensor(x, **f32), torch.tensor(y, **f32)
        s.theta = torch.tensor(_network_params(), **f32)
        # moments of a run under way
        s.m = torch.tensor(1e-3 * g.standard_normal(M.MLP_PARAMS), **f32)
        s.v = torch.tensor(1e-6 * g.uniform(0.5, 2.0, size=M.MLP_PARAMS), **f32)
        s.grad, s.loss = torch.zeros(M.MLP_PARAMS, **f32), torch.zeros(4, **f32)
        s.blob = torch.empty(M.MLP_BLOB_BYTES, dtype=torch.uint8, device="cuda")
        s.step = 100
        M.molt_mlp_pack(s.theta, s.blob)
        return s
    # small heat steps and batches run on a stream of their own, so that the library can capture them; so do the
    # Hamilton-Jacobi and advection-diffusion runs.  The wave and the bare operator run on the current stream.
    own = case["kind"] in ("heat", "batch", "hj", "advdiff")
    s.stream = torch.cuda.Stream() if own else torch.cuda.current_stream()
    with torch.cuda.stream(s.stream):
        if case["kind"] == "batch":
            each = _batch_cases(case)
            s.u = [_field(c, seed * 1000 + i) for i, c in enumerate(each)]
            s.ctx = M.molt_create([_desc(c) for c in each], s.stream)
            s.t = [0.0] * len(each)
            s.prev = None
        else:
            s.u = _field(case, seed)
            s.ctx = M.molt_create(_desc(case), s.stream)
            s.t = [0.0]
            s.prev = torch.zeros_like(s.u) if case["kind"] == "wave" else None
        if case["kind"] == "apply":
            s.out = [torch.empty_like(s.u) for _ in _shape(case)]
            s.alpha = _alpha(case)
            if case["nonuniform"]:
                for ax, n in enumerate(_shape(case)):
                    M.molt_set_grid_axis(s.ctx, 0, ax, _nodes(case, n))
        if case["weights"] == "learned":
            blob = torch.empty(M.MLP_BLOB_BYTES, dtype=torch.uint8, device="cuda")
            M.molt_mlp_pack(torch.tensor(_network_params(), device="cuda"), blob, s.stream)
            M.molt_set_mlp(s.ctx, blob)
        if case.get("ham") == "affine_sq":
            M.molt_set_source(s.ctx, 0, _source(case))
        s.stream.synchronize()
    return s


def _returns_time(case):
    """The adaptive time of a Hamilton-Jacobi run.  With the network, one point's choice between its weights and the
    WENO-Z weights (a threshold) can set the largest speed, so there the time is seen through the state alone."""
    return case["kind"] == "hj" and case["weights"] != "learned"


def run(s):
    case = s.case
    if case["kind"] == "train":
        M.molt_mlp_loss_grad(s.blob, s.x, s.y, s.grad, s.loss)
        s.step += 1
        M.molt_mlp_adam(s.theta, s.m, s.v, s.grad, s.step, 1e-4, s.blob)
        return {"grad": s.grad, "loss": s.loss[:1], "theta": s.theta, "m": s.m, "v": s.v}
    if case["kind"] == "apply":
        src = s.u
        for ax, out in enumerate(s.out):                 # S_P along x, of that along y, ...
            M.molt_apply_D(s.ctx, 0, ax, OPS[case["op"]], case["P"], s.alpha[ax], src, out)
            src = out
        return list(s.out)
    s.t = M.molt_step(s.ctx, s.u, s.prev, nsteps=case["steps"], t=s.t)
    if case["kind"] == "wave":
        return {"u": s.u, "u_prev": s.prev}
    if _returns_time(case):
        return {"u": s.u, "t": s.t[0]}
    return {"u": s.u}


# ----------------------------------------------------------------------- work
def _per_point(case, dirs):
    """Operations of one D application at one point: the local integrals, recurrences and closures."""
    w = 2 * case["quad"]
    if case["weights"] != "linear":
        w += 60
    if case["weights"] == "learned":
        w += 2 * (5 * 32 + 32 * 32 + 32 * 3) + 64 * 10
    return dirs * (w + 6) + 4


def work(case):
    """One pass: every step (or application) reads its state once and writes it once."""
    if case["kind"] == "train":
        n = case["nx"]
        return {"bytes": n * 8 * 4 + 1347 * 4 * 8, "flops": n * 3 * 2 * (5 * 32 + 32 * 32 + 32 * 3)}
    if case["kind"] == "batch":
        each = [work(c) for c in _batch_cases(case)]
        return {k: sum(w[k] for w in each) for k in ("bytes", "flops")}
    pts = float(np.prod(_shape(case)))
    nd, el = len(_shape(case)), 4 if case["prec"] == "f32" else 8
    if case["kind"] == "apply":
        dirs = 2 if case["op"] == "0" else 1
        # the WENO-Z and point-local tables are small beside the field
        return {"bytes": nd * pts * 2 * el, "flops": nd * pts * case["P"] * _per_point(case, dirs)}
    stages = 3 if case["kind"] == "heat" and case.get("integrator") != "euler" else 1
    flops = pts * nd * stages * case["P"] * _per_point(case, 2) * (2 if case["kind"] == "advdiff" else 1)
    arrays = {"wave": 3, "hj": 5 if case.get("ham") == "affine_sq" else 2}.get(case["kind"], 2)
    return {"bytes": case["steps"] * pts * arrays * el, "flops": case["steps"] * flops}


def tolerance(case):
    """About four times the largest difference from ``exact`` seen over the listed and many drawn cases."""
    if case["kind"] == "train":
        # the gradient's products run in BF16
        return {"rel": 1e-2, "max": 5e-2}
    if case["prec"] == "f64":
        if case["weights"] != "linear":
            # tau = |beta_0 - beta_2| of nearly equal indicators
            return {"rel": 2e-12, "max": 2e-10}
        if case.get("nonuniform"):
            # the cells of a stretched axis are differences of coordinates, 1e-13 of a cell off
            return {"rel": 4e-13, "max": 3e-12}
        return {"rel": 5e-14, "max": 5e-13}
    if case["kind"] == "apply":
        # D = v - L^{-1}[v] cancels: the result is small beside v at small nu
        return {"rel": 4e-6, "max": 4e-5}
    if case["kind"] == "hj":
        # the time comes from the largest of the FP32 derivatives, each a small difference of values of order one
        return {"rel": 4e-5 if _returns_time(case) else 4e-6, "max": 1e-4}
    return {"rel": 2e-6, "max": 2e-5}


# ---------------------------------------------------------------------- exact
_GX, _GW = np.polynomial.legendre.leggauss(40)
OFFSETS = {3: (-1, 0, 1), 5: (-3, -2, -1, 0, 1), 6: (-3, -2, -1, 0, 1, 2)}


def _lagrange(nodes, j, z, order=0):
    """The Lagrange basis polynomial j on ``nodes`` (arrays (k, m)) at z (arrays (q, m)), or its derivative of that
    order; m points of a line at a time."""
    k = nodes.shape[0]
    others = [i for i in range(k) if i != j]
    scale = np.prod([nodes[j] - nodes[i] for i in others], axis=0)

    def drop(left, order):
        if order == 0:
            out = np.ones_like(z)
            for i in left:
                out = out * (z - nodes[i])
            return out
        return sum(drop([i for i in left if i != d], order - 1) for d in left)
    return drop(others, order) / scale


def _rule(nodes, cell, alpha):
    """Weights of alpha int_cell e^{-alpha |s|} p(s) ds (the point at s = 0, p through ``nodes``, relative to it)."""
    a, b = cell
    s = 0.5 * (b - a) * _GX[:, None] + 0.5 * (a + b)
    w = 0.5 * (b - a) * _GW[:, None] * alpha * np.exp(-alpha * np.abs(s))
    return np.stack([np.sum(w * _lagrange(nodes, j, s), axis=0) for j in range(nodes.shape[0])])


def _smoothness(nodes, cell):
    """beta = sum_l dx^{2l-1} int_cell (p^{(l)})^2, l = 1, 2, as the matrix of a quadratic form in the node values."""
    a, b = cell
    dx = b - a
    s = 0.5 * dx * _GX[:, None] + 0.5 * (a + b)
    w = 0.5 * dx * _GW[:, None]
    k = nodes.shape[0]
    out = np.zeros((k, k) + dx.shape)
    for l in (1, 2):
        d = [_lagrange(nodes, j, s, l) for j in range(k)]
        for i in range(k):
            for j in range(k):
                out[i, j] += dx ** (2 * l - 1) * np.sum(w * d[i] * d[j], axis=0)
    return out


def _tables(nodes, cell, alpha, npts):
    """Every constant of one direction: nodes (npts, m) relative to each point, in the order of the J_R offsets."""
    t = {"c": _rule(nodes, cell, alpha)}
    if npts == 5:
        t["sub"] = [_rule(nodes[r:r + 3], cell, alpha) for r in range(3)]
        # sum_r d_r c^{(r)} = c at the outermost nodes fixes d_0 and d_2
        d0, d2 = t["c"][0] / t["sub"][0][0], t["c"][4] / t["sub"][2][2]
        t["d"] = [d0, 1.0 - d0 - d2, d2]
        t["M"] = [_smoothness(nodes[r:r + 3], cell) for r in range(3)]
    return t


def _uniform_rule(nu, npts):
    nodes = np.array(OFFSETS[npts], dtype=np.float64)[:, None]
    t = _tables(nodes, (np.array([-1.0]), np.array([0.0])), nu, npts)
    return t


def _wenoz_weights(vals, t):
    """w_r of the five values in J_R order (numpy arrays or torch tensors), as a stacked array (3, ...)."""
    beta = []
    for r in range(3):
        m = t["M"][r]
        beta.append(sum(m[i][j] * vals[r + i] * vals[r + j] for i in range(3) for j in range(3)))
    tau = abs(beta[0] - beta[2])
    wt = [t["d"][r] * (1.0 + tau / (1e-6 + beta[r])) for r in range(3)]
    tot = wt[0] + wt[1] + wt[2]
    stack = torch.stack if isinstance(vals[0], torch.Tensor) else np.stack
    return stack([w / tot for w in wt])


def _to_dev(t):
    """The tables as FP64 tensors that broadcast over (points, lines)."""
    def dev(a):
        a = np.asarray(a)
        return float(a[0]) if a.shape[-1] == 1 else torch.tensor(a, device="cuda")[:, None]
    out = {"c": [dev(c) for c in t["c"]]}
    if "d" in t:
        out["sub"] = [[dev(c) for c in s] for s in t["sub"]]
        out["d"] = [dev(d) for d in t["d"]]
        out["M"] = [[[dev(m[i, j]) for j in range(3)] for i in range(3)] for m in t["M"]]
    return out


class _Line:
    """Lines of one axis: their tables for alpha, decays and closures."""

    def __init__(self, n, h, alpha, npts, bc, weights, x=None, period=None):
        self.n, self.bc, self.weights, self.npts = n, bc, weights, npts
        off = OFFSETS[npts]
        if x is None:
            r = _uniform_rule(alpha * h, npts)
            self.R, self.L = _to_dev(r), _to_dev(r)
            self.q = [math.exp(-alpha * h)] * (n + 1)    # q[i]: decay of the cell that ends at point i
            self.width = alpha * h * (n if bc == "periodic" else n - 1)
            return
        g = 4                                            # ghost nodes on either side
        if bc == "periodic":
            xe = np.concatenate([x[-g:] - period, x, x[:g] + period])
            self.width = alpha * period
        else:
            xe = np.concatenate([2 * x[0] - x[g:0:-1], x, 2 * x[-1] - x[-2:-g - 2:-1]])
            self.width = alpha * (x[-1] - x[0])
        i = np.arange(n) + g
        self.q = list(np.exp(-alpha * (xe[g:g + n + 1] - xe[g - 1:g + n])))
        self.R = _to_dev(_tables(np.stack([xe[i + l] - xe[i] for l in off]), (xe[i - 1] - xe[i], 0.0 * xe[i]), alpha,
                                 npts))
        self.L = _to_dev(_tables(np.stack([xe[i - l] - xe[i] for l in off]), (0.0 * xe[i], xe[i + 1] - xe[i]), alpha,
                                 npts))

    def local(self, ext, t, sign, net):
        """J of every point; ext has three ghost rows on either side."""
        vals = [ext[3 + sign * l:3 + sign * l + self.n] for l in OFFSETS[self.npts]]
        if self.weights == "linear":
            out = t["c"][0] * vals[0]
            for c, v in zip(t["c"][1:], vals[1:]):
                out = out + c * v
            return out
        w = _wenoz_weights(vals, t)
        if net is not None:
            p = _network(net, torch.stack([v.reshape(-1) for v in vals], dim=1))[1].T.reshape(w.shape)
            near = (p - w).abs().amax(dim=0) <= 1e-2
            w = torch.where(near, p, w)
        return sum(w[r] * sum(t["sub"][r][j] * vals[r + j] for j in range(3)) for r in range(3))

    def inverse(self, v, op, net):
        """L^{-1} of the lines v (points, lines)."""
        n, per = self.n, self.bc == "periodic"
        if per:
            ext = v[torch.arange(-3, n + 3, device=v.device) % n]
        else:
            lo = [2 * v[:1] - v[j:j + 1] for j in (3, 2, 1)]
            hi = [2 * v[n - 1:] - v[n - 1 - j:n - j] for j in (1, 2, 3)]
            ext = torch.cat(lo + [v] + hi)
        mu = math.exp(-self.width)
        right = left = None
        if op != "L":
            right = self.local(ext, self.R, 1, net)
            if not per:
                right[0] = 0.0
            for i in range(1, n):
                right[i].add_(right[i - 1], alpha=self.q[i])
        if op != "R":
            left = self.local(ext, self.L, -1, net)
            if not per:
                left[n - 1] = 0.0
            for i in range(n - 2, -1, -1):
                left[i].add_(left[i + 1], alpha=self.q[i + 1])
        # the decay from the left end (or its periodic image) to every point, and from the right end
        q = torch.tensor(self.q, dtype=torch.float64, device=v.device)
        if per:
            ea = torch.cumprod(q[:n], 0)[:, None]
            eb = torch.cumprod(q[1:].flip(0), 0).flip(0)[:, None]
            if right is not None:
                right = right + ea * (right[n - 1:] / (-math.expm1(-self.width)))
            if left is not None:
                left = left + eb * (left[:1] / (-math.expm1(-self.width)))
            return right if op == "R" else left if op == "L" else 0.5 * (right + left)
        one = torch.ones(1, dtype=torch.float64, device=v.device)
        ea = torch.cat([one, torch.cumprod(q[1:n], 0)])[:, None]
        eb = torch.cat([torch.cumprod(q[1:n].flip(0), 0).flip(0), one])[:, None]
        if op == "R":
            return right + ea * v[:1]
        if op == "L":
            return left + eb * v[n - 1:]
        i0 = 0.5 * (right + left)
        r0, r1 = v[:1] - i0[:1], v[n - 1:] - i0[n - 1:]
        det = -math.expm1(-2.0 * self.width)
        return i0 + ea * ((r0 - mu * r1) / det) + eb * ((r1 - mu * r0) / det)

    def sum(self, v, op, P, net=None):
        out = torch.zeros_like(v)
        for _ in range(P):
            v = v - self.inverse(v, op, net)
            out += v
        return out


def _axis_sum(line, u, ax, op, P, net=None):
    """S_P along axis ax (0 = x, the last dimension) of u, some lines at a time."""
    d = u.ndim - 1 - ax
    v = u.movedim(d, 0)
    flat = v.reshape(v.shape[0], -1)
    out = torch.empty(flat.shape, dtype=u.dtype, device=u.device)
    most = max(1, (1 << (22 if net is not None else 26)) // flat.shape[0])
    for k in range(0, flat.shape[1], most):
        out[:, k:k + most] = line.sum(flat[:, k:k + most].contiguous(), op, P, net)
    return out.reshape(v.shape).movedim(0, d)


def _lines(case, alpha):
    return [_Line(n, h, a, case["quad"], case["bc"], case["weights"])
            for n, h, a in zip(_shape(case), _spacings(case), alpha)]


def _exact_heat(case, u):
    dt, beta = _dt(case), _beta(case)
    lines = _lines(case, [beta / math.sqrt(dt)] * u.ndim)
    rk = ((0.0, 1.0),) if case.get("integrator") == "euler" else SSPRK3
    for _ in range(case["steps"]):
        un = us = u
        for a0, a1 in rk:
            s = sum(_axis_sum(ln, us, ax, "0", case["P"]) for ax, ln in enumerate(lines))
            us = a0 * un + a1 * (us - beta * beta * s)
        u = us
    return u


def _exact_batch(case, seed):
    each = _batch_cases(case)
    out = [None] * len(each)
    for side in sorted(set(c["nx"] for c in each)):
        same = [i for i, c in enumerate(each) if c["nx"] == side]
        # problems of one side as the planes of one array, swept along x and y
        u = torch.stack([_field(each[i], seed * 1000 + i) for i in same])
        c = each[same[0]]
        dt, beta = _dt(c), _beta(c)
        lines = _lines(c, [beta / math.sqrt(dt)] * 2)
        for _ in range(case["steps"]):
            us = u
            for a0, a1 in SSPRK3:
                s = sum(_axis_sum(ln, us, ax, "0", c["P"]) for ax, ln in enumerate(lines))
                us = a0 * u + a1 * (us - beta * beta * s)
            u = us
        for k, i in enumerate(same):
            out[i] = u[k]
    return out


def _exact_wave(case, u):
    beta = _beta(case)
    lines = _lines(case, [beta / _dt(case)] * u.ndim)
    prev = None
    for _ in range(case["steps"]):
        s = sum(_axis_sum(ln, u, ax, "0", case["P"]) for ax, ln in enumerate(lines))
        new = u - 0.5 * beta * beta * s if prev is None else 2.0 * u - prev - beta * beta * s
        prev, u = u, new
    return {"u": u, "u_prev": prev}


def _exact_hj(case, u):
    h = _spacings(case)
    alpha = _beta(case) / (case["cfl"] * min(h))
    lines = _lines(case, [alpha] * u.ndim)
    net = _bf16(torch.tensor(_network_params(), device="cuda")) if case["weights"] == "learned" else None
    src = _source(case).double() if case["ham"] == "affine_sq" else None
    vel = _velocity(case)

    def hamiltonian(u):
        mean, half, r = [], [], []
        for ax, ln in enumerate(lines):
            vm = alpha * _axis_sum(ln, u, ax, "R", 1, net)
            vp = -alpha * _axis_sum(ln, u, ax, "L", 1, net)
            mean.append(0.5 * (vm + vp))
            half.append(0.5 * (vp - vm))
            if case["ham"] == "half_sq":
                r.append(torch.maximum(vm.abs(), vp.abs()))
            elif case["ham"] == "linear":
                r.append(torch.full_like(vm, abs(vel[ax])))
        if case["ham"] == "half_sq":
            H = 0.5 * sum(m * m for m in mean)
        else:
            H = sum(a * m for a, m in zip(vel, mean))
            if case["ham"] == "affine_sq":
                # |dH/dp_d| = |a_d| |1 + a.p|, largest at a corner of the box of one-sided derivatives
                top = (1.0 + H).abs() + sum(abs(a) * d.abs() for a, d in zip(vel, half))
                r = [abs(a) * top for a in vel[:len(mean)]]
                H = 0.5 * (1.0 + H) ** 2
        H = H - sum(a * b for a, b in zip(r, half))
        return H, [float(x.max()) for x in r]

    t, speeds = 0.0, hamiltonian(u)[1]
    for _ in range(case["steps"]):
        dt = min([case["cfl"] * hd / c for hd, c in zip(h, speeds) if c > 0] + [10.0 * min(h)])
        H, speeds = hamiltonian(u)
        if src is not None:
            H = H - (src[0] + t * (src[1] + t * src[2]))
        u = u - dt * H
        t += dt
    return {"u": u, "t": t} if _returns_time(case) else {"u": u}


def _exact_advdiff(case, u):
    dt, beta, c, kappa = _dt(case), _beta(case), 1.2, _kappa(case)
    hyp = _lines(case, [beta / (c * dt)] * u.ndim)
    dif = _lines(case, [beta / math.sqrt(kappa * dt)] * u.ndim)
    for _ in range(case["steps"]):
        f = torch.zeros_like(u)
        for ax in range(u.ndim):
            g = 0.5 * u * u if case["flux"] == "burgers" else _velocity(case)[ax] * u
            f -= beta / c * (_axis_sum(hyp[ax], 0.5 * (g + c * u), ax, "R", case["P"])
                             - _axis_sum(hyp[ax], 0.5 * (g - c * u), ax, "L", case["P"]))
            f -= beta * beta * _axis_sum(dif[ax], u, ax, "0", case["P"])
        u = u + f
    return {"u": u}


def _exact_train(case, seed):
    s = prepare(case, seed)
    theta = _bf16(s.theta).requires_grad_(True)
    p = _network(theta, s.x.double())[1]
    loss = ((p - s.y.double()) ** 2).sum(dim=1).mean()
    loss.backward()
    g = theta.grad
    m, v = 0.9 * s.m.double() + 0.1 * g, 0.999 * s.v.double() + 0.001 * g * g
    k = s.step + 1
    new = s.theta.double() - 1e-4 * (m / (1 - 0.9 ** k)) / (torch.sqrt(v / (1 - 0.999 ** k)) + 1e-8)
    return {"grad": g, "loss": loss.detach().reshape(1), "theta": new, "m": m, "v": v}


def exact(case, seed):
    if case["kind"] == "train":
        return _exact_train(case, seed)
    if case["kind"] == "batch":
        return {"u": _exact_batch(case, seed)}
    u = _field(case, seed).double()
    if case["kind"] == "apply":
        out = []
        for ax, (n, h, a) in enumerate(zip(_shape(case), _spacings(case), _alpha(case))):
            x = _nodes(case, n) if case["nonuniform"] else None
            u = _axis_sum(_Line(n, h, a, case["quad"], case["bc"], case["weights"], x, TWO_PI), u, ax, case["op"],
                          case["P"])
            out.append(u)
        return out
    if case["kind"] == "heat":
        return {"u": _exact_heat(case, u)}
    return {"wave": _exact_wave, "hj": _exact_hj, "advdiff": _exact_advdiff}[case["kind"]](case, u)
