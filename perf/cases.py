"""What this library is measured on: its public calls over the meshes, degrees and precisions they
are used with.

Sizes are those of the repository's own workloads: the 8^3 p = 2 cavity (the smallest configuration,
bound by latency), the 32^3 p = 3 cavity (the FP64 sweep), the 64^3 p = 3 cavity (gradients), the
16^3 .. 48^3 p = 2 .. 4 meshes of the batch, the 128^3 p = 3 cavity (the headline), and 61^3 p = 2 as
a mesh nothing was tuned on.

Kinds (each is one call of `Stokes` or of the autograd functions):
  apply_K      y = K x in FP64, banded Kronecker form or (forward = quadrature) the matrix-free
               quadrature form
  apply_K_f32  y = K x for an FP32 x in pair-of-FP32 arithmetic (the `outer = pair` option)
  apply_P      the base block preconditioner (fast diagonalisation)
  hyperpower   the order-q, s-step preconditioner; FP64, or TF32 / BF16 for one or several
               right-hand sides
  solve        the preconditioned Krylov solve of a cavity with a random body force. FP64 MINRES
               stops at 1e-8, the tolerance of every FP64 workload here. Flexible GMRES with a
               reduced-precision preconditioner stops at 1e-12: the mixed form where the caller
               wants an FP64-accurate solution (its error at 1e-8 depends on the last bit of every
               rounding in the preconditioner, so two correct runs agree to that tolerance only).
  gradient     forward solve, adjoint solve and the gradient of a velocity misfit
"""
import math

import numpy as np
import torch

from paper_2311_06926_gb300 import Stokes, synthetic
from paper_2311_06926_gb300.adjoint import cavity_solve, mass_misfit

C_PEN = 14.0       # the library's default Nitsche constant
N_THETA = 16       # lid-profile coefficients of the gradient workload


def _case(kind, n, p, nu=1.0, **more):
    c = {"kind": kind, "n": n, "p": p, "nu": nu}
    c.update(more)
    return c


def listed():
    named = [
        # the smallest operator call: four short launches, host call and latency
        ("apply_K_8_p2", _case("apply_K", 8, 2)),
        # the operator of every outer iteration of the headline solve
        ("apply_K_128_p3", _case("apply_K", 128, 3)),
        # the operator of the paper's timings, formed by quadrature on the fly
        ("apply_K_quad_32_p3", _case("apply_K", 32, 3, forward="quadrature")),
        # the Arnoldi product of the pair-of-FP32 option at the headline size
        ("apply_K_f32_128_p3", _case("apply_K_f32", 128, 3)),
        # the FP64 base preconditioner: the sweep's mesh, and the headline's
        ("apply_P_32_p3", _case("apply_P", 32, 3)),
        ("apply_P_128_p3", _case("apply_P", 128, 3)),
        # an FP64 polynomial preconditioner on an odd mesh, another viscosity and Schur sequence
        ("hyper_fp64_61_p2", _case("hyperpower", 61, 2, 0.1, precision="fp64", order=3, steps=1,
                                   schur="none", nrhs=1)),
        # the headline's preconditioner on the tensor cores
        ("hyper_tf32_128_p3", _case("hyperpower", 128, 3, precision="tf32", order=3, steps=1,
                                    schur="inner", nrhs=1)),
        # the batch workload's largest mesh with its right-hand sides, in BF16
        ("hyper_bf16_48x6_p4", _case("hyperpower", 48, 4, precision="bf16", order=2, steps=2,
                                     schur="inner", nrhs=6)),
        # a whole FP64 solve of the sweep
        ("solve_minres_32_p3", _case("solve", 32, 3, precision="fp64", order=2, steps=2)),
        # a whole mixed-precision solve at the headline size
        ("solve_tf32_128_p3", _case("solve", 128, 3, precision="tf32", order=3, steps=1)),
        # differentiation through the solver
        ("gradient_64_p3", _case("gradient", 64, 3, order=2, steps=1)),
    ]
    return [dict(c, name=name) for name, c in named]


def _mesh(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["apply_K", "apply_K", "apply_K_f32", "apply_P", "apply_P", "hyperpower",
                       "hyperpower", "hyperpower", "solve", "solve", "gradient"])
    nu = round(math.exp(rng.uniform(math.log(0.05), math.log(20.0))), 3)
    p = rng.choice([1, 2, 2, 3, 3, 4])
    if kind == "apply_K" and rng.random() < 0.25:
        return _case(kind, _mesh(rng, 4, 40), p, nu, forward="quadrature")
    if kind in ("apply_K", "apply_K_f32"):
        return _case(kind, _mesh(rng, 4, 128), p, nu)
    if kind == "apply_P":
        return _case(kind, _mesh(rng, 4, 128), p, nu)
    if kind == "hyperpower":
        precision = rng.choice(["fp64", "fp64", "tf32", "bf16"])
        order, steps = rng.choice([(2, 1), (2, 2), (3, 1)])
        nrhs = 1 if precision == "fp64" else rng.choice([1, 1, 3, 6])
        return _case(kind, _mesh(rng, 6, 128 if nrhs == 1 else 48), p, nu, precision=precision,
                     order=order, steps=steps, schur=rng.choice(["inner", "inner", "none"]),
                     nrhs=nrhs)
    if kind == "solve":
        precision = rng.choice(["fp64", "tf32", "bf16"])
        order, steps = rng.choice([(2, 0), (2, 1), (2, 2), (3, 1)])
        return _case(kind, _mesh(rng, 6, 48 if precision == "fp64" else 96), p, nu,
                     precision=precision, order=order, steps=steps)
    return _case(kind, _mesh(rng, 6, 48), p, nu, order=2, steps=rng.choice([0, 1]))


def _tol(case):
    return 1e-8 if case.get("precision", "fp64") == "fp64" else 1e-12


def _context(case):
    kind, kw = case["kind"], {"nu": case["nu"]}
    if kind == "apply_K":
        kw.update(max_order=2, max_steps=0, forward=case.get("forward", "kronecker"))
    elif kind == "apply_K_f32":
        kw.update(max_order=2, max_steps=0, precision="tf32", outer="pair")
    elif kind == "apply_P":
        kw.update(max_order=2, max_steps=0)
    else:
        kw.update(max_order=case["order"], max_steps=case["steps"])
        if kind == "hyperpower":
            kw.update(precision=case["precision"], schur=case["schur"], nrhs=case["nrhs"])
        elif kind == "solve":
            kw.update(precision=case["precision"])
    G = Stokes(case["n"], case["p"], **kw)
    if kind in ("solve", "gradient"):
        G.set_preconditioner(case["order"], case["steps"])
    return G


def _vector(case, seed, nrhs=1):
    """A vector as the solver meets it: noise concentrated near the lid (x2 = 1), where the
    residual of a cavity lives, fading over two orders of magnitude away from it."""
    n, p = case["n"], case["p"]
    a, b = n + p - 1, n + p
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    out = []
    for _ in range(nrhs):
        for e1, e2, e3 in ((a, b, b), (b, a, b), (b, b, a), (b, b, b)):
            fade = torch.exp(torch.linspace(-5.0, 0.0, e2, dtype=torch.float64, device="cuda"))
            t = torch.randn(e3, e2, e1, dtype=torch.float64, device="cuda", generator=g)
            out.append((t * fade[None, :, None]).reshape(-1))
    return torch.cat(out)


def _lid_theta(seed):
    return np.random.default_rng(seed).uniform(0.5, 1.5, N_THETA)


def prepare(case, seed):
    G = _context(case)
    s = {"case": case, "G": G}
    kind = case["kind"]
    if kind in ("apply_K", "apply_P"):
        s["x"] = _vector(case, seed)
    elif kind == "apply_K_f32":
        s["x"] = _vector(case, seed).float()
    elif kind == "hyperpower":
        s["x"] = _vector(case, seed, case["nrhs"])
    elif kind == "solve":
        f = G.rhs_cavity(synthetic.lid_speed(seed))
        coef, waves = synthetic.forcing_modes(seed)
        s["x"] = G.rhs_body(coef, waves, accumulate=True, out=f)
    else:
        coef, waves = synthetic.forcing_modes(seed)
        s["waves"] = waves
        s["theta"] = torch.tensor(_lid_theta(seed), requires_grad=True)
        s["coef"] = torch.tensor(coef, requires_grad=True)
        s["nu"] = torch.tensor(case["nu"], dtype=torch.float64, requires_grad=True)
        s["target"] = torch.from_numpy(synthetic.random_vector(G.n_vel, seed + 1000) * 0.01).cuda()
        return s
    s["y"] = G.empty(G.batch_size)
    return s


def run(state):
    case, G = state["case"], state["G"]
    kind = case["kind"]
    if kind == "apply_K":
        return G.apply_K(state["x"], out=state["y"])
    if kind == "apply_K_f32":
        return G.apply_K_f32(state["x"], out=state["y"])
    if kind == "apply_P":
        return G.apply_P(state["x"], out=state["y"])
    if kind == "hyperpower":
        return G.apply_hyperpower(case["order"], case["steps"], state["x"], out=state["y"])
    if kind == "solve":
        x, its, _, _ = G.solve(state["x"], _tol(case), out=state["y"])
        # the FP64 count is determined by the method, the mixed one also by the roundings
        return {"x": x, "iterations": its} if case["precision"] == "fp64" else {"x": x}
    for leaf in (state["theta"], state["coef"], state["nu"]):
        leaf.grad = None
    x = cavity_solve(G, state["theta"], state["coef"], state["nu"], state["waves"], 1e-8)
    J = mass_misfit(G, x, state["target"])
    J.backward()
    return {"J": J.detach(), "x": x.detach(), "theta": state["theta"].grad,
            "coef": state["coef"].grad, "nu": state["nu"].grad}


def work(case):
    """Inputs read once and outputs written once; flops of the factored operators (bands of 2p+3
    and 2p+1 entries; even and odd modes apart). A solve's are those of about as many iterations as
    its preconditioner needs for the first eight digits."""
    n, p, kind = case["n"], case["p"], case["kind"]
    a, b = n + p - 1, n + p
    nv, npr = 3 * a * b * b, b ** 3
    size = nv + npr
    k_apply = nv * (4 * (2 * p + 3) + 10 * (2 * p + 1) + 4) + npr * (12 * (2 * p + 1) + 10)
    a_apply = nv * (4 * (2 * p + 3) + 10 * (2 * p + 1) + 4) + npr * (6 * (2 * p + 1) + 6)
    b_apply = npr * 6 * (2 * p + 1) + 3 * nv
    pv, pq = nv * (6 * b + 1), npr * 12 * (p + 1)

    def hyper(q, s, schur):
        m = q ** s
        v = m * pv + (m - 1) * a_apply
        inner = 1 if (s == 1 or schur == "none") else m
        return v + m * pq + (m - 1) * (2 * b_apply + inner * pv + (inner - 1) * a_apply)

    if kind in ("apply_K", "apply_K_f32"):
        return {"bytes": (16 if kind == "apply_K" else 12) * size, "flops": k_apply}
    if kind == "apply_P":
        return {"bytes": 16 * size, "flops": pv + pq}
    if kind == "hyperpower":
        r = case["nrhs"]
        return {"bytes": 16 * size * r,
                "flops": r * hyper(case["order"], case["steps"], case["schur"])}
    its = {1: 56, 2: 30, 3: 23, 4: 20}[case["order"] ** case["steps"]]
    one = its * (k_apply + hyper(case["order"], case["steps"], "inner"))
    return {"bytes": 16 * size, "flops": one if kind == "solve" else 2 * one}


# ---- the same quantities by the textbook formulas in 64 bits --------------------------------------


def _bsplines(t, d, x):
    """Values of the degree-d B-splines of the knots t at x in [0, 1] (Cox-de Boor)."""
    last = int(np.max(np.nonzero(t < t[-1])[0]))
    s = np.minimum(np.searchsorted(t, x, side="right") - 1, last)
    N = np.zeros((len(x), len(t) - 1))
    N[np.arange(len(x)), s] = 1.0
    for k in range(1, d + 1):
        up = np.zeros((len(x), N.shape[1] - 1))
        for i in range(up.shape[1]):
            if t[i + k] > t[i]:
                up[:, i] += (x - t[i]) / (t[i + k] - t[i]) * N[:, i]
            if t[i + k + 1] > t[i + 1]:
                up[:, i] += (t[i + k + 1] - x) / (t[i + k + 1] - t[i + 1]) * N[:, i + 1]
        N = up
    return N


def _basis(n, d, x, unit):
    """Values and derivatives of the degree-d splines on n elements; unit: scaled to integral 1."""
    t = np.concatenate([np.zeros(d), np.linspace(0.0, 1.0, n + 1), np.ones(d)])
    v, low = _bsplines(t, d, x), _bsplines(t, d - 1, x)
    dv = np.zeros_like(v)
    for i in range(v.shape[1]):
        if t[i + d] > t[i]:
            dv[:, i] += d / (t[i + d] - t[i]) * low[:, i]
        if t[i + d + 1] > t[i + 1]:
            dv[:, i] -= d / (t[i + d + 1] - t[i + 1]) * low[:, i + 1]
    integral = (t[d + 1:] - t[:-d - 1]) / (d + 1)
    return (v / integral, dv / integral, integral) if unit else (v, dv, integral)


def _gauss(breaks, q):
    g, w = np.polynomial.legendre.leggauss(q)
    x = np.concatenate([0.5 * (lo + hi) + 0.5 * (hi - lo) * g
                        for lo, hi in zip(breaks[:-1], breaks[1:])])
    return x, np.concatenate([0.5 * (hi - lo) * w for lo, hi in zip(breaks[:-1], breaks[1:])])


def _eig(K, M):
    """Generalised eigenpairs: U^T K U = diag(lam), U^T M U = 1."""
    Li = np.linalg.inv(np.linalg.cholesky(M))
    lam, V = np.linalg.eigh(Li @ K @ Li.T)
    return lam, Li.T @ V


class _Plain:
    """The discrete Stokes system by dense 1D factors: 15 Kronecker products for A, three for B."""

    def __init__(self, n, p, nu):
        self.n, self.p, self.nu = n, p, nu
        a, b = self.a, self.b = n + p - 1, n + p
        self.shapes = [(b, b, a), (b, a, b), (a, b, b), (b, b, b)]     # (x3, x2, x1)
        self.sizes = [math.prod(s) for s in self.shapes]
        self.n_vel = sum(self.sizes[:3])
        breaks = np.linspace(0.0, 1.0, n + 1)
        x, w = _gauss(breaks, p + 2)
        N, dN, _ = _basis(n, p + 1, x, False)
        N, dN = N[:, 1:n + p], dN[:, 1:n + p]
        M, dM, self.int_Np = _basis(n, p, x, True)
        W = w[:, None]
        ends = np.array([0.0, 1.0])
        Me, dMe, _ = _basis(n, p, ends, True)
        self.M1, self.dM1 = Me[1], dMe[1]
        pen = np.outer(Me[1], Me[1]) + np.outer(Me[0], Me[0])
        flux = np.outer(Me[1], dMe[1]) - np.outer(Me[0], dMe[0])
        mats = {"M": N.T @ (W * N), "K": dN.T @ (W * dN), "C": N.T @ (W * dM),
                "Mc": M.T @ (W * M), "Cc": dN.T @ (W * M)}
        mats["T"] = 0.5 * (dM.T @ (W * dM) + 2.0 * C_PEN * n * pen - flux - flux.T)
        self.int_N = N.T @ w
        lN, UN = _eig(mats["K"], mats["M"])
        lT, UT = _eig(mats["T"], mats["Mc"])
        dev = lambda v: torch.from_numpy(np.ascontiguousarray(v)).cuda()  # noqa: E731
        self.m = {k: dev(v) for k, v in mats.items()}
        self.m["Mi"] = dev(np.linalg.inv(mats["Mc"]))
        self.lam, self.U = {"N": dev(lN), "T": dev(lT)}, {"N": dev(UN), "T": dev(UT)}
        self.const = dev(np.einsum("i,j,k->ijk", *[self.int_Np] * 3).reshape(-1))

    @staticmethod
    def kron(D3, D2, D1, t):
        t = t @ D1.T
        t = torch.matmul(D2, t)
        return (D3 @ t.reshape(t.shape[0], -1)).reshape(D3.shape[0], t.shape[1], t.shape[2])

    def split(self, x):
        return [t.reshape(s) for t, s in zip(x.split(self.sizes), self.shapes)]

    @staticmethod
    def join(ts):
        return torch.cat([t.reshape(-1) for t in ts])

    def velocity(self, u):
        """A u for the three components."""
        m, k, nu = self.m, self.kron, self.nu
        M, K, C, Mc, T = m["M"], m["K"], m["C"], m["Mc"], m["T"]
        Ct = C.T
        u1, u2, u3 = u
        return [2 * nu * (k(Mc, Mc, K, u1) + k(Mc, T, M, u1) + k(T, Mc, M, u1))
                + nu * (k(Mc, Ct, C, u2) + k(Ct, Mc, C, u3)),
                2 * nu * (k(Mc, M, T, u2) + k(Mc, K, Mc, u2) + k(T, M, Mc, u2))
                + nu * (k(Mc, C, Ct, u1) + k(Ct, C, Mc, u3)),
                2 * nu * (k(M, Mc, T, u3) + k(M, T, Mc, u3) + k(K, Mc, Mc, u3))
                + nu * (k(C, Mc, Ct, u1) + k(C, Ct, Mc, u2))]

    def grad(self, q):
        Mc, Cc, k = self.m["Mc"], self.m["Cc"], self.kron
        return [k(Mc, Mc, Cc, q), k(Mc, Cc, Mc, q), k(Cc, Mc, Mc, q)]

    def div(self, u):
        Mc, Ct, k = self.m["Mc"], self.m["Cc"].T, self.kron
        return k(Mc, Mc, Ct, u[0]) + k(Mc, Ct, Mc, u[1]) + k(Ct, Mc, Mc, u[2])

    def saddle(self, x):
        *u, q = self.split(x)
        return self.join([s + t for s, t in zip(self.velocity(u), self.grad(q))] + [self.div(u)])

    def base_v(self, u):
        out = []
        for c, t in enumerate(u):
            f = ["N" if d == c else "T" for d in range(3)]      # directions 1, 2, 3
            U1, U2, U3 = (self.U[k] for k in f)
            l1, l2, l3 = (self.lam[k] for k in f)
            t = self.kron(U3.T, U2.T, U1.T, t)
            t = t / (2 * self.nu * (l3[:, None, None] + l2[None, :, None] + l1[None, None, :]))
            out.append(self.kron(U3, U2, U1, t))
        return out

    def base_q(self, q):
        Mi = self.m["Mi"]
        return 2 * self.nu * self.kron(Mi, Mi, Mi, q)

    @staticmethod
    def _power(x, base, apply, q, s):
        if s == 0:
            return base(x)
        prev = lambda v: _Plain._power(v, base, apply, q, s - 1)  # noqa: E731
        r, acc = x, x
        for _ in range(q - 1):
            r = [i - j for i, j in zip(r, apply(prev(r), s))]
            acc = [i + j for i, j in zip(acc, r)]
        return prev(acc)

    def hyper(self, x, q, s, schur="inner"):
        *u, pr = self.split(x)
        v_level = lambda v, l: self._power(v, self.base_v, lambda t, _: self.velocity(t), q, l)  # noqa: E731
        schur_apply = lambda t, m: [self.div(v_level(self.grad(t[0]), 0 if (m == 1 or schur == "none") else m))]  # noqa: E731,E501
        yq = self._power([pr], lambda t: [self.base_q(t[0])], schur_apply, q, s)
        return self.join(v_level(u, s) + yq)

    def zero_mean(self, x):
        x = x.clone()
        q = x[self.n_vel:]
        x[self.n_vel:] = q - q.sum() * self.const
        return x

    def _minres(self, f, tol, maxit=300):
        """Preconditioned MINRES (base preconditioner) from zero."""
        prec = lambda v: self.hyper(v, 2, 0)  # noqa: E731
        x = torch.zeros_like(f)
        v_old, v = torch.zeros_like(f), f.clone()
        z = prec(v)
        g = math.sqrt(float(z @ v))
        eta, g_old, s_old, s, c_old, c = g, 1.0, 0.0, 0.0, 1.0, 1.0
        w_old, w = torch.zeros_like(f), torch.zeros_like(f)
        first = eta
        for _ in range(maxit):
            z = z / g
            kz = self.saddle(z)
            d = float(kz @ z)
            v_new = kz - (d / g) * v - (g / g_old) * v_old
            z_new = prec(v_new)
            g_new = math.sqrt(max(0.0, float(z_new @ v_new)))
            a0 = c * d - c_old * s * g
            a1 = math.hypot(a0, g_new)
            a2, a3 = s * d + c_old * c * g, s_old * g
            c_old, s_old, c, s = c, s, a0 / a1, g_new / a1
            w_old, w = w, (z - a3 * w_old - a2 * w) / a1
            x = x + (c * eta) * w
            eta = -s * eta
            if abs(eta) <= tol * first or g_new == 0.0:
                break
            v_old, v, z, g_old, g = v, v_new, z_new, g, g_new
        return x

    def solve(self, f):
        """K^-1 f with zero-mean pressure, refined until the residual is at rounding level."""
        x = torch.zeros_like(f)
        for _ in range(3):
            x = x + self._minres(f - self.saddle(x) if x.any() else f, 1e-7)
        return self.zero_mean(x)

    # loads and the misfit of the gradient workload
    def _axis_loads(self, k):
        """int sin(k pi x) times the N and the M functions."""
        x, w = _gauss(np.linspace(0.0, 1.0, self.n + 1), 24)
        s = w * np.sin(k * np.pi * x)
        return (s @ _basis(self.n, self.p + 1, x, False)[0][:, 1:self.n + self.p],
                s @ _basis(self.n, self.p, x, True)[0])

    @staticmethod
    def _outer(l1, l2, l3):
        t = [torch.from_numpy(np.ascontiguousarray(v)).cuda() for v in (l1, l2, l3)]
        return (t[2][:, None, None] * t[1][None, :, None] * t[0][None, None, :]).reshape(-1)

    def body_modes(self, waves):
        """(c, m, the load of that unit mode on component c) of every mode."""
        loads = {int(k): self._axis_loads(int(k)) for k in np.unique(waves)}
        for c in range(3):
            for m in range(waves.shape[1]):
                yield c, m, self._outer(*[loads[int(waves[c, m, d])][0 if d == c else 1]
                                          for d in range(3)])

    def body(self, coef, waves):
        f = torch.zeros(sum(self.sizes), dtype=torch.float64, device="cuda")
        at = np.concatenate([[0], np.cumsum(self.sizes)])
        for c, m, load in self.body_modes(waves):
            f[at[c]:at[c + 1]] += float(coef[c, m]) * load
        return f

    def lid(self, along_x1):
        """Load of the lid velocity whose integrals against the N functions are given."""
        g2 = self.nu * (2.0 * C_PEN * self.n * self.M1 - self.dM1)
        f = torch.zeros(sum(self.sizes), dtype=torch.float64, device="cuda")
        f[:self.sizes[0]] = self._outer(along_x1, g2, np.ones(self.b))
        return f

    def lid_matrix(self):
        nel = N_THETA - 3
        x, w = _gauss(np.union1d(np.linspace(0, 1, self.n + 1), np.linspace(0, 1, nel + 1)),
                      self.p + 6)
        N = _basis(self.n, self.p + 1, x, False)[0][:, 1:self.n + self.p]
        return N.T @ (w[:, None] * _basis(nel, 3, x, False)[0])

    def mass(self, u):
        M, Mc, k = self.m["M"], self.m["Mc"], self.kron
        return [k(Mc, Mc, M, u[0]), k(Mc, M, Mc, u[1]), k(M, Mc, Mc, u[2])]

    def gradient(self, theta, coef, waves, target):
        L = self.lid_matrix()
        f_lid = self.lid(L @ theta)
        x = self.solve(f_lid + self.body(coef, waves))
        pad = torch.zeros(self.sizes[3], dtype=torch.float64, device="cuda")
        e = x[:self.n_vel] - target
        Me = self.join(self.mass(self.split(torch.cat([e, pad]))[:3]))
        lam = self.solve(torch.cat([Me, pad]))
        at = np.concatenate([[0], np.cumsum(self.sizes)])
        g_coef = torch.zeros(coef.shape, dtype=torch.float64)
        for c, m, load in self.body_modes(waves):
            g_coef[c, m] = float(lam[at[c]:at[c + 1]] @ load)
        g_theta = torch.tensor([float(lam @ self.lid(L[:, k])) for k in range(N_THETA)],
                               dtype=torch.float64)
        Ax = self.join(self.velocity(self.split(x)[:3]))
        g_nu = (float(lam @ f_lid) - float(lam[:self.n_vel] @ Ax)) / self.nu
        return {"J": 0.5 * (e @ Me), "x": x, "theta": g_theta, "coef": g_coef,
                "nu": torch.tensor(g_nu, dtype=torch.float64)}


def exact(case, seed):
    S = _Plain(case["n"], case["p"], case["nu"])
    kind = case["kind"]
    if kind == "apply_K":
        return S.saddle(_vector(case, seed))
    if kind == "apply_K_f32":
        return S.saddle(_vector(case, seed).float().double())
    if kind == "apply_P":
        return S.hyper(_vector(case, seed), 2, 0)
    if kind == "hyperpower":
        x = _vector(case, seed, case["nrhs"])
        return torch.cat([S.hyper(t, case["order"], case["steps"], case["schur"])
                          for t in x.split(sum(S.sizes))])
    coef, waves = synthetic.forcing_modes(seed)
    if kind == "solve":
        x = S.solve(S.lid(synthetic.lid_speed(seed) * S.int_N) + S.body(coef, waves))
        return {"x": x, "iterations": None} if case["precision"] == "fp64" else {"x": x}
    target = torch.from_numpy(synthetic.random_vector(S.n_vel, seed + 1000) * 0.01).cuda()
    return S.gradient(_lid_theta(seed), coef, waves, target)
