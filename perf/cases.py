"""The library's workloads as measurable cases: what a user of the package runs,
through its public entry points (`ds.PhiSet`, `ds.Plan`, `ds.Batch`, `ds.tucker`,
`adjoint.integrate`).

`listed()` names the cases, `draw(rng)` gives more of the same ranges,
`prepare(case, seed)` makes what a program holds before the call, `run(state)` is
one pass, `work(case)` its compulsory bytes and operations and `exact(case, seed)`
the same outputs in 64-bit torch, from the method's formulas alone.

States.  FP64 runs start from the package's initial data (equilibrium plus white
noise, white noise for FitzHugh-Nagumo).  The reduced precisions start from the
smooth states that a run meets once diffusion has acted, which is where all but
the first few of its steps are spent: a few Neumann cosine modes per direction,
of the initial data's amplitude.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2310_07551_gb300 import adjoint, configs, ds, inputs

SCHNAK, FHN = configs.SCHNAK, configs.FHN
DELTA = {"schnakenberg": (1.0, 10.0), "fhn": (1.0, 42.1887)}
DOMAIN = {"schnakenberg": (0.0, 1.0), "fhn": (-1.0, 1.0)}
PARAMS = {"schnakenberg": SCHNAK, "fhn": FHN}


def listed():
    return [
        # the smallest run: a 64^2 pattern in FP64, launches and latency count
        dict(name="schnak2d_64_f64", kind="run", model="schnakenberg", precision="f64", scheme="exprk3ds_real",
             d=2, n1=64, n2=64, tau=2e-4, steps=10),
        # an ordinary FP64 run on an odd, non-square grid (no padding-friendly size)
        dict(name="schnak2d_301x150_f64", kind="run", model="schnakenberg", precision="f64", scheme="exprk3ds_real",
             d=2, n1=301, n2=150, tau=2e-4, steps=4),
        # the complex two-term split, the paper's second integrator, at its laptop size
        dict(name="schnak2d_150_cplx", kind="run", model="schnakenberg", precision="f64", scheme="exprk3ds_cplx",
             d=2, n1=150, n2=150, tau=2e-4, steps=2),
        # parameter fitting: forward and reverse of two steps with gradients in the
        # state, the reaction parameters and the diffusion scalings, 96^3
        dict(name="fhn3d_96_adjoint", kind="adjoint", model="fhn", d=3, n1=96, n2=96, n3=96, tau=1e-3, steps=2),
        # one step per call with a look at the state in between, small grid
        dict(name="schnak2d_192_bf16x6_step", kind="step", model="schnakenberg", precision="bf16x6",
             scheme="exprk3ds_real", d=2, n1=192, n2=192, tau=2e-4, steps=1),
        # Schnakenberg 1024^2 in the precision recommended for it
        dict(name="schnak2d_1024_bf16x6", kind="run", model="schnakenberg", precision="bf16x6",
             scheme="exprk3ds_real", d=2, n1=1024, n2=1024, tau=1e-4, steps=10),
        # FitzHugh-Nagumo 256^3 in the precision recommended for it (the largest run)
        dict(name="fhn3d_256_f16x10", kind="run", model="fhn", precision="f16x10", scheme="exprk3ds_real",
             d=3, n1=256, n2=256, n3=256, tau=1e-3, steps=4),
        # single-precision CUDA-core run, the paper's GPU arithmetic, at its 100^3 size
        dict(name="fhn3d_100_f32", kind="run", model="fhn", precision="f32", scheme="exprk3ds_real",
             d=3, n1=100, n2=100, n3=100, tau=1e-3, steps=2),
        # a parameter study: uneven independent problems stepped together
        dict(name="batch16_f16x13", kind="batch", precision="f16x13", count=16, family=7, steps=10),
        # the Tucker operator on its own, FP64, three unequal sizes
        dict(name="tucker_201x150x67_f64", kind="tucker", precision="f64", transpose=False,
             d=3, n1=201, n2=150, n3=67),
        # the Tucker operator in split BF16, a large cube
        dict(name="tucker_256_bf16x6", kind="tucker", precision="bf16x6", transpose=False,
             d=3, n1=256, n2=256, n3=256),
        # the phi-matrices of a new time step or diffusion coefficient
        dict(name="phi_setup_256x200", kind="phi", model="schnakenberg", d=2, n1=256, n2=200, tau=2e-4),
    ]


def _log_int(rng, lo, hi, step=1):
    n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi))) / step)) * step
    return max(lo, min(hi, n))


def draw(rng):
    kind = rng.choice(["run64_2d", "run64_3d", "run64_4d", "scheme", "adjoint", "step", "bf16", "fx", "f32", "batch",
                       "tucker64", "tucker16", "phi"])
    tau = math.exp(rng.uniform(math.log(5e-5), math.log(2e-4)))
    real = "exprk3ds_real"
    if kind in ("run64_2d", "scheme"):
        scheme = rng.choice(["etd2rkds", "exprk3ds_cplx"]) if kind == "scheme" else real
        return dict(kind="run", model="schnakenberg", precision="f64", scheme=scheme, d=2,
                    n1=_log_int(rng, 33, 400), n2=_log_int(rng, 33, 400), tau=tau, steps=rng.randint(1, 6))
    if kind == "run64_3d":
        return dict(kind="run", model="fhn", precision="f64", scheme=real, d=3, n1=_log_int(rng, 24, 110),
                    n2=_log_int(rng, 24, 110), n3=_log_int(rng, 24, 110), tau=5 * tau, steps=rng.randint(1, 3))
    if kind == "run64_4d":
        return dict(kind="run", model="fhn", precision="f64", scheme=real, d=4, n1=rng.randint(9, 32),
                    n2=rng.randint(9, 32), n3=rng.randint(9, 32), n4=rng.randint(9, 32), tau=5 * tau, steps=1)
    if kind == "adjoint":
        return dict(kind="adjoint", model="fhn", d=3, n1=_log_int(rng, 20, 96), n2=_log_int(rng, 20, 96),
                    n3=_log_int(rng, 20, 96), tau=5 * tau, steps=rng.randint(1, 3))
    if kind in ("step", "bf16"):
        return dict(kind="step" if kind == "step" else "run", model="schnakenberg", precision="bf16x6", scheme=real,
                    d=2, n1=_log_int(rng, 64, 768, 8), n2=_log_int(rng, 64, 768), tau=tau,
                    steps=1 if kind == "step" else rng.randint(2, 12))
    if kind == "fx":
        return dict(kind="run", model="fhn", precision="f16x10", scheme=real, d=3, n1=_log_int(rng, 64, 256, 8),
                    n2=_log_int(rng, 64, 256), n3=_log_int(rng, 64, 256), tau=5 * tau, steps=rng.randint(2, 4))
    if kind == "f32":
        return dict(kind="run", model="fhn", precision="f32", scheme=real, d=3, n1=_log_int(rng, 32, 128),
                    n2=_log_int(rng, 32, 128), n3=_log_int(rng, 32, 128), tau=5 * tau, steps=rng.randint(1, 3))
    if kind == "batch":
        return dict(kind="batch", precision="f16x13", count=rng.randint(2, 16), family=rng.randint(1, 1000),
                    steps=rng.randint(4, 12))
    if kind == "phi":
        return dict(kind="phi", model="schnakenberg", d=2, n1=_log_int(rng, 33, 300), n2=_log_int(rng, 33, 300),
                    tau=tau)
    if kind == "tucker64":
        return dict(kind="tucker", precision="f64", transpose=rng.random() < 0.5, d=3, n1=_log_int(rng, 24, 240),
                    n2=_log_int(rng, 24, 240), n3=_log_int(rng, 24, 240))
    return dict(kind="tucker", precision="bf16x6", transpose=rng.random() < 0.5, d=3, n1=_log_int(rng, 32, 256, 8),
                n2=_log_int(rng, 32, 256), n3=_log_int(rng, 32, 256))


def _dims(case):
    return tuple(case["n%d" % (q + 1)] for q in range(case["d"]))


def _instances(case):
    return configs.batch_instances(case["count"], case["family"])


def _fd(dims, lo, hi):
    return [inputs.fd_neumann(n, lo, hi) for n in dims]


def _matrices(model, dims):
    Ds = _fd(dims, *DOMAIN[model])
    return [[dl * D for D in Ds] for dl in DELTA[model]]


def _rand(gen, *shape):
    return torch.rand(*shape, dtype=torch.float64, device="cuda", generator=gen)


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _equilibrium(a, b):
    return inputs.schnakenberg_equilibrium(a, b)


def _noise_state(model, dims, gen, a=0.1, b=0.9):
    """The package's initial data (`inputs.initial_state`) from torch's generator."""
    U = _rand(gen, 2, *reversed(dims))
    if model == "fhn":
        return U.mul_(2.0).sub_(1.0)
    for c, e in enumerate(_equilibrium(a, b)):
        U[c].mul_(1e-3).add_(e)
    return U


def _smooth_state(model, dims, gen, a=0.1, b=0.9, modes=6):
    """Random Neumann cosine modes 0 .. modes-1 per direction.  FitzHugh-Nagumo: u of
    order one, v as its fast diffusion leaves it (driven by u mode by mode);
    Schnakenberg: both components near equilibrium, deviations of 1e-3."""
    d = len(dims)
    coef = _rand(gen, 2, *([modes] * d)).mul_(2.0).sub_(1.0) / modes ** (d / 2)
    if model == "fhn":
        k2 = (torch.arange(modes, dtype=torch.float64, device="cuda") * (math.pi / 2)) ** 2
        lam = sum(k2.reshape([-1 if q == r else 1 for r in range(d)]) for q in range(d))
        coef[1] = FHN[0] * coef[0] / (DELTA["fhn"][1] * lam + FHN[0] * FHN[1])
    out = torch.empty((2,) + tuple(reversed(dims)), dtype=torch.float64, device="cuda")
    for c in range(2):
        x = coef[c]
        for n in dims:   # each pass contracts the leading mode axis and appends its grid axis
            j = torch.arange(n, dtype=torch.float64, device="cuda") * (math.pi / (n - 1))
            cos = torch.cos(torch.arange(modes, dtype=torch.float64, device="cuda")[:, None] * j[None, :])
            x = torch.tensordot(x, cos, dims=([0], [0]))
        out[c] = x.permute(*reversed(range(d)))
    if model == "schnakenberg":
        for c, e in enumerate(_equilibrium(a, b)):
            out[c].mul_(1e-3).add_(e)
    return out.contiguous()


def _initial(case, seed):
    make = _noise_state if case.get("precision", "f64") == "f64" else _smooth_state
    return make(case["model"], _dims(case), _gen(seed))


def _tucker_inputs(case, seed):
    gen, dims = _gen(seed), _dims(case)
    X = _rand(gen, *reversed(dims)).mul_(2.0).sub_(1.0)
    return X, [_rand(gen, n, n).mul_(2.0).sub_(1.0) for n in dims]


def _batch_states(case, seed):
    gen = _gen(seed)
    return [_smooth_state("schnakenberg", i.dims, gen, a=i.params[1], b=i.params[2]) for i in _instances(case)]


def _adjoint_inputs(case, seed):
    gen, dims = _gen(seed), _dims(case)
    U0 = _noise_state(case["model"], dims, gen)
    lam = _rand(gen, 2, *reversed(dims)).mul_(2.0).sub_(1.0)
    return U0, lam


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("run", "step"):
        dims = _dims(case)
        phis = ds.PhiSet(dims, _matrices(case["model"], dims), case["tau"], scheme=case["scheme"])
        plan = ds.Plan(phis, case["model"], PARAMS[case["model"]], precision=case["precision"])
        return dict(kind=kind, plan=plan, U=_initial(case, seed), steps=case["steps"])
    if kind == "batch":
        inst = _instances(case)
        As = [[[dl * D for D in _fd(i.dims, 0.0, 1.0)] for dl in i.delta] for i in inst]
        batch = ds.Batch([i.dims for i in inst], As, [i.tau for i in inst], "schnakenberg", [i.params for i in inst],
                         precision=case["precision"])
        return dict(kind=kind, batch=batch, Us=_batch_states(case, seed), steps=case["steps"])
    if kind == "adjoint":
        dims = _dims(case)
        phis = ds.PhiSet(dims, _matrices(case["model"], dims), case["tau"])
        plan = ds.Plan(phis, case["model"], PARAMS[case["model"]], precision="f64")
        U0, lam = _adjoint_inputs(case, seed)
        p = torch.tensor(PARAMS[case["model"]], dtype=torch.float64, device="cuda")
        s = torch.ones(2, dtype=torch.float64, device="cuda")
        return dict(kind=kind, plan=plan, lam=lam, steps=case["steps"],
                    leaves=[t.requires_grad_() for t in (U0, p, s)])
    if kind == "tucker":
        X, Ls = _tucker_inputs(case, seed)
        return dict(kind=kind, X=X, Ls=Ls, transpose=case["transpose"], precision=case["precision"])
    if kind == "phi":
        # the coefficients are the input here: one diffusion coefficient per seed
        dims = _dims(case)
        return dict(kind=kind, dims=dims, tau=case["tau"], As=_phi_matrices(case, seed))
    raise ValueError(kind)


def _phi_scale(seed):
    return 0.5 + float(np.random.default_rng(int(seed)).random())


def _phi_matrices(case, seed):
    dims = _dims(case)
    As = _matrices(case["model"], dims)
    return [As[0], [_phi_scale(seed) * A for A in As[1]]]


def run(state):
    kind = state["kind"]
    if kind == "run":
        return state["plan"].integrate(state["U"], state["steps"])
    if kind == "step":
        return state["plan"].step(state["U"])
    if kind == "batch":
        state["batch"].integrate(state["Us"], state["steps"])
        return list(state["Us"])
    if kind == "adjoint":
        U0, p, s = state["leaves"]
        out = adjoint.integrate(U0, p, state["plan"], state["steps"], ckpt=state["steps"], s=s)
        return [out.detach(), *torch.autograd.grad(out, (U0, p, s), grad_outputs=state["lam"])]
    if kind == "tucker":
        return ds.tucker(state["X"], state["Ls"], transpose=state["transpose"], precision=state["precision"])
    phis = ds.PhiSet(state["dims"], state["As"], state["tau"])
    return [phis.get(c, slot, i, mu) for c in range(2) for slot in range(5) for i in range(2) for mu in range(2)]


# --------------------------------------------------------------------------
# Compulsory work: 2 N n_mu operations per mode product; states, checkpoints
# and matrices read and written once per pass.
# --------------------------------------------------------------------------
def _slots_terms(scheme, d):
    """(Tucker operators per component and step, real products per Tucker operator)"""
    if scheme == "etd2rkds":
        return 2, d
    if scheme == "exprk3ds_cplx":
        return 10, 2 + 4 * (d - 2) + 2
    return 5 * (2 if d == 2 else 3), d


def _step_work(dims, scheme, steps):
    d, N = len(dims), math.prod(dims)
    ops, prods = _slots_terms(scheme, d)
    mats = 2 * ops * sum(n * n for n in dims) * (2 if scheme == "exprk3ds_cplx" else 1)
    # products of one mode all cost 2 N n_mu; the complex split repeats each mode equally
    flops = steps * 2 * ops * (prods / d) * sum(2.0 * N * n for n in dims)
    return {"bytes": 32.0 * N + 8.0 * mats, "flops": flops}


def work(case):
    kind = case["kind"]
    if kind in ("run", "step"):
        return _step_work(_dims(case), case["scheme"], case["steps"])
    if kind == "batch":
        w = [_step_work(i.dims, "exprk3ds_real", case["steps"]) for i in _instances(case)]
        return {k: sum(x[k] for x in w) for k in ("bytes", "flops")}
    dims = _dims(case)
    d, N = len(dims), math.prod(dims)
    if kind == "adjoint":
        # forward step, its recomputation up to U3, the transposed sweep and, per
        # Tucker operator, d operators with one derivative matrix
        fwd = _step_work(dims, "exprk3ds_real", 1)
        steps = case["steps"]
        return {"bytes": 2 * fwd["bytes"] + steps * 16.0 * N, "flops": steps * fwd["flops"] * (1 + 0.6 + 1 + d)}
    if kind == "tucker":
        return {"bytes": 16.0 * N + 8.0 * sum(n * n for n in dims), "flops": sum(2.0 * N * n for n in dims)}
    # phi: 20 matrices per size; scaling to norm 1/2 and degree-16 Taylor with shared
    # powers (a dozen products), then three products per squaring
    flops = nbytes = 0.0
    for n in dims:
        lam = 4.0 * (n - 1) ** 2
        for c in range(2):
            s = max(0.0, math.ceil(math.log2(max(1.0, 2 * case["tau"] * DELTA["schnakenberg"][c] * lam * 2))))
            flops += 10 * (12 + 3 * s) * 2.0 * n ** 3
            nbytes += 8.0 * n * n * 11
    return {"bytes": nbytes, "flops": flops}


# --------------------------------------------------------------------------
# The outputs in 64-bit torch: the split step from its formulas, the phi-functions
# from the closed-form eigenvectors of the Neumann difference matrix.
# --------------------------------------------------------------------------
def _table(d, ell, scheme):
    """[(phi index, eta, alpha per direction)] of the split of phi_ell."""
    if scheme == "etd2rkds":
        return [(ell, 1.0 if ell == 1 else 2.0 ** (d - 1), [1.0] * d)]
    if scheme == "exprk3ds_cplx":
        sc = 2.0 ** (d - 2)
        if ell == 1:
            r = math.sqrt(2.0)
            return [(1, complex(1.75, 1.5 * r), [complex(12 / 11, -4 * r / 11)] * d),
                    (2, complex(-3, -6 * r) * sc, [complex(4 / 3, -2 * r / 3)] * d)]
        r = math.sqrt(3.0)
        return [(1, complex(2 / 3, 2 * r / 3), [complex(0.75, -r / 4)] * d),
                (2, complex(-2 / 3, -8 * r / 3) * sc, [complex(6 / 7, -3 * r / 7)] * d)]
    if d == 2:
        if ell == 1:
            r = math.sqrt(10.0)
            return [(1, -1.25, [4 / 3 + 4 * r / 15, 4 / 3 - 4 * r / 15]),
                    (2, 9.0, [16 / 9 + 2 * r / 9, 16 / 9 - 2 * r / 9])]
        r = math.sqrt(33.0)
        return [(1, -4 / 3, [9 / 8 + r / 8, 9 / 8 - r / 8]), (2, 22 / 3, [1.5 + 3 * r / 22, 1.5 - 3 * r / 22])]
    p = 2.0 ** (d - 3)
    if ell == 1:
        r = math.sqrt(2991111.0)
        m, o, am, ao = 2243 / 1350, 440521 / 675 / r, 3 * 5161 / 15869, 3 * r / 15869
        e2, a2 = -12544 / 675 * p, 45 / 28
    else:
        r = math.sqrt(2391.0)
        m, o, am, ao = 19 / 27, 151 / 27 / r, 3 * 121 / 490, 3 * r / 490
        e2, a2 = -196 / 27 * p, 9 / 7
    return [(1, m + o, [am + ao] * d), (2, e2, [a2] * d), (1, m - o, [am - ao] * d)]


def _phi(ell, z):
    """phi_1 or phi_2 of a vector, by its power series near zero."""
    small = z.abs() < 0.5
    zs = torch.where(small, z, torch.zeros_like(z))
    series = torch.zeros_like(z)
    for j in range(20, -1, -1):
        series = series * zs + 1.0 / math.factorial(j + ell)
    zl = torch.where(small, torch.ones_like(z), z)
    e = torch.exp(zl) - 1.0
    return torch.where(small, series, e / zl if ell == 1 else (e - zl) / (zl * zl))


class _Eigen:
    """The n-point Neumann difference matrix D = V diag(lam) V^-1."""

    def __init__(self, n, lo, hi, dev):
        m, h = n - 1, (hi - lo) / (n - 1)
        k = torch.arange(n, dtype=torch.int64, device=dev)
        self.V = torch.cos(((k[:, None] * k[None, :]) % (2 * m)).to(torch.float64) * (math.pi / m))
        w = torch.ones(n, dtype=torch.float64, device=dev)
        w[0] = w[-1] = 0.5
        self.Vi = (2.0 / m) * w[:, None] * self.V * w[None, :]
        self.lam = -4.0 / (h * h) * torch.sin(k.to(torch.float64) * (math.pi / (2 * m))) ** 2
        self.D = torch.from_numpy(inputs.fd_neumann(n, lo, hi)).to(dev)

    def phi(self, ell, z, s=None):
        """phi_ell(z s D), z a number, s a 0-dim tensor or None"""
        lam = self.lam * z if s is None else self.lam * z * s
        f = _phi(ell, lam)
        return (self.V.to(f.dtype) * f) @ self.Vi.to(f.dtype)


def _mode(X, mu, L):
    axis = X.dim() - 1 - mu
    return torch.movedim(torch.tensordot(L, X, dims=([1], [axis])), 0, axis)


def _chain(X, Ls):
    for mu, L in enumerate(Ls):
        X = _mode(X.to(L.dtype), mu, L)
    return X


def _react(model, p, U):
    u, v = U[0], U[1]
    if model == "schnakenberg":
        w = u * u * v
        return torch.stack([p[0] * (p[1] - u + w), p[0] * (p[2] - w)])
    return torch.stack([u - u ** 3 - v, p[0] * (u - p[1] * v - p[2])])


class _Exact:
    def __init__(self, model, dims, dom, delta, p, tau, scheme="exprk3ds_real", s=None):
        self.model, self.p, self.tau, self.scheme, self.d = model, p, tau, scheme, len(dims)
        eig = {n: _Eigen(n, *dom, "cuda") for n in set(dims)}
        self.eig = [eig[n] for n in dims]
        self.delta, self.s = delta, s
        self.mats = {}

    def _split(self, c, cs, ell, X):
        key = (c, cs, ell)
        if key not in self.mats:
            s = None if self.s is None else self.s[c]
            self.mats[key] = [(eta, [self.eig[mu].phi(li, cs * self.tau * self.delta[c] * al[mu], s)
                                     for mu in range(self.d)])
                              for li, eta, al in _table(self.d, ell, self.scheme)]
        out = 0.0
        for eta, Ls in self.mats[key]:
            Y = eta * _chain(X, Ls)
            out = out + (Y.real if Y.is_complex() else Y)
        return out

    def S(self, cs, ell, X):
        return torch.stack([self._split(c, cs, ell, X[c]) for c in range(2)])

    def K(self, U):
        out = []
        for c in range(2):
            x = sum(_mode(U[c], mu, self.eig[mu].D) for mu in range(self.d)) * self.delta[c]
            out.append(x if self.s is None else x * self.s[c])
        return torch.stack(out)

    def step(self, U):
        t = self.tau
        G = _react(self.model, self.p, U)
        F = self.K(U) + G
        if self.scheme == "etd2rkds":
            U2 = U + t * self.S(1.0, 1, F)
            return U2 + t * self.S(1.0, 2, _react(self.model, self.p, U2) - G)
        U2 = U + t / 3 * self.S(1 / 3, 1, F)
        D2 = _react(self.model, self.p, U2) - G
        U3 = U + 2 * t / 3 * self.S(2 / 3, 1, F) + 4 * t / 3 * self.S(2 / 3, 2, D2)
        D3 = _react(self.model, self.p, U3) - G
        return U + t * self.S(1.0, 1, F) + 1.5 * t * self.S(1.0, 2, D3)


def exact(case, seed):
    kind = case["kind"]
    if kind == "tucker":
        X, Ls = _tucker_inputs(case, seed)
        return _chain(X, [L.t() for L in Ls] if case["transpose"] else Ls)
    if kind == "phi":
        dims = _dims(case)
        eig = [_Eigen(n, *DOMAIN[case["model"]], "cuda") for n in dims]
        dl = [DELTA[case["model"]][0], DELTA[case["model"]][1] * _phi_scale(seed)]
        out = []
        for c in range(2):
            for cs, ell in ((1 / 3, 1), (2 / 3, 1), (2 / 3, 2), (1.0, 1), (1.0, 2)):
                for li, _, al in _table(2, ell, "exprk3ds_real"):
                    out += [eig[mu].phi(li, cs * case["tau"] * dl[c] * al[mu]).cpu().numpy() for mu in range(2)]
        return out
    if kind == "batch":
        out = []
        for i, U in zip(_instances(case), _batch_states(case, seed)):
            ex = _Exact("schnakenberg", i.dims, (0.0, 1.0), i.delta, i.params, i.tau)
            for _ in range(case["steps"]):
                U = ex.step(U)
            out.append(U)
        return out
    model, dims = case["model"], _dims(case)
    if kind == "adjoint":
        U0, lam = _adjoint_inputs(case, seed)
        p = torch.tensor(PARAMS[model], dtype=torch.float64, device="cuda")
        s = torch.ones(2, dtype=torch.float64, device="cuda")
        leaves = [t.requires_grad_() for t in (U0, p, s)]
        ex = _Exact(model, dims, DOMAIN[model], DELTA[model], p, case["tau"], s=s)
        U = U0
        for _ in range(case["steps"]):
            U = ex.step(U)
        return [U.detach(), *torch.autograd.grad(U, leaves, grad_outputs=lam)]
    U = _initial(case, seed)
    ex = _Exact(model, dims, DOMAIN[model], DELTA[model], PARAMS[model], case["tau"], case["scheme"])
    for _ in range(case["steps"]):
        U = ex.step(U)
    return U
