"""Work that a user has the MG-CCCS library do, as timed cases.

Each case is one call (or the few calls a program makes together) through the public
binding: preconditioner applications and stand-alone iterations for a caller's own outer
solver, one Gram-Schmidt pass of a caller's Arnoldi loop, whole GMRES solves in both
precisions, setups, a point of an energy scan, adjoint gradients and a batch.  Problems are
Temkin-Poet on the exterior-scaled square box [0, L]^2 (R0 = 2L/3, theta = pi/6) with the
impact-ionisation source plus complex noise; sizes are those of the repository's benchmark,
sweeps and tests.

`exact` restates the method in plain torch complex128: level operators, V-cycle, bound
states, CCCS with dense or block-Thomas solves, and a GMRES run to the rounding level.
"""
import math

import numpy as np
import torch

from paper_1412_1953_gb300 import adjoint
from paper_1412_1953_gb300 import mgcccs as M

THETA = math.pi / 6
OMEGA = 2.0 / 3.0
GAMMA = M.COARSE_GAMMA_DEFAULT
C128, C64 = torch.complex128, torch.complex64


def _case(kind, nx, levels, n_b, ny=None, L=30.0, E=0.5, nu1=1, nu2=1, precision=0, k=11, count=1, rtol=1e-10):
    return {"kind": kind, "nx": nx, "ny": nx if ny is None else ny, "L": L, "E": E, "levels": levels, "nu1": nu1,
            "nu2": nu2, "n_b": n_b, "precision": precision, "k": k, "count": count, "rtol": rtol}


def listed():
    return [
        # the smallest problem of the parity tests and the smoke run: a preconditioner call
        # inside a caller's own Krylov loop, all launch latency
        dict(_case("precond", 128, 5, 3), name="precond_128"),
        # the benchmark's grid, block-reduction coarsest solve: what every FP64 Arnoldi step runs
        dict(_case("precond", 1024, 5, 3), name="precond_1024"),
        # the complex64 preconditioner of a mixed-precision handle on a grid of the batch workload
        dict(_case("precond", 384, 5, 3, precision=1), name="precond_384_c64"),
        # stand-alone MG-CCCS iteration (no Krylov) on a non-square grid with odd row lengths, V(2,1)
        dict(_case("iterate", 768, 5, 1, ny=512, nu1=2), name="iterate_768x512"),
        # operator and one Gram-Schmidt pass of an Arnoldi step at the mean column count of GMRES(20)
        dict(_case("arnoldi", 1024, 5, 0, k=11), name="arnoldi_1024"),
        # the same on complex64 vectors, as the mixed form's cycles do, on the largest grid
        dict(_case("arnoldi", 2048, 6, 0, L=60.0, precision=1, k=11), name="arnoldi_2048_c64"),
        # the headline: one GMRES(20) solve to 1e-10 in complex128
        dict(_case("solve", 1024, 5, 3), name="solve_1024"),
        # the precision form: complex64 cycles in FP64 refinement, six states per axis, the largest grid
        dict(_case("solve", 2048, 6, 6, L=60.0, precision=1), name="solve_2048_mixed"),
        # a new potential: full setup (bound states, coarsest factors, channel factors) and the
        # first preconditioner application
        dict(_case("setup", 1024, 5, 3), name="setup_1024"),
        # one point of an energy scan: setup from the states already known (31^2 coarsest grid,
        # dense inverse), then the mixed-precision solve
        dict(_case("energy", 512, 5, 3, precision=1, E=0.8), name="energy_512"),
        # gradients of the amplitude in E, Z and the potential: setup, forward and adjoint solves
        dict(_case("gradient", 256, 4, 3, L=15.0, rtol=1e-11), name="gradient_256"),
        # several energies and grids at once as one graph launch, the batch's tuned V(2,2)
        dict(_case("batch", 384, 4, 3, L=22.5, nu1=2, nu2=2, precision=1, count=6), name="batch_6"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: kinds as listed, grids from 64 to 2048 cells per axis with 16 to 64
    coarsest cells (so odd multiples, non-square grids and both coarsest solvers occur)."""
    kind = rng.choice(["precond", "precond", "iterate", "arnoldi", "arnoldi", "solve", "setup", "energy", "gradient",
                       "batch"])
    top = {"precond": 2048, "iterate": 1024, "arnoldi": 2048, "solve": 1000, "setup": 900, "energy": 640,
           "gradient": 320, "batch": 420}[kind]
    n = _log_int(rng, 96, top)
    levels = rng.choice([v for v in range(2, 7) if 16 <= n >> (v - 1) <= 62])
    s = 1 << (levels - 1)
    nx = max(16, n // s) * s
    ny = nx
    if kind in ("precond", "iterate", "arnoldi", "solve") and rng.random() < 0.4:
        ny = max(16, int(n * rng.uniform(0.6, 1.0)) // s) * s
    L = 30.0 if n < 768 else rng.choice([30.0, 45.0])
    if kind in ("gradient", "batch"):
        L = 30.0 * nx / 512 if nx >= 256 else 15.0
    # a complex64 cycle amplifies its own rounding on large grids; there only a solve's result is comparable
    both = kind in ("arnoldi", "solve", "energy", "batch") or (kind in ("precond", "setup") and n <= 400)
    return _case(kind, nx, levels, 0 if kind == "arnoldi" else rng.choice([1, 2, 3, 3, 4, 5, 6]), ny=ny, L=L,
                 E=round(rng.uniform(0.3, 1.2), 3), nu1=1 if kind in ("solve", "energy") else rng.choice([1, 1, 2]),
                 nu2=rng.choice([1, 1, 2]), precision=rng.choice([0, 1]) if both else 0,
                 k=rng.randint(2, 20), count=rng.randint(2, 6), rtol=1e-11 if kind == "gradient" else 1e-10)


# ---------------------------------------------------------------- inputs

def _rand(shape, gen):
    return torch.complex(torch.randn(shape, generator=gen, device="cuda", dtype=torch.float64),
                         torch.randn(shape, generator=gen, device="cuda", dtype=torch.float64))


def _nodes(n, L):
    """Interior node parameters x and their exterior-scaled images z."""
    x = torch.arange(1, n, dtype=torch.float64, device="cuda") * (L / n)
    R0 = 2.0 * L / 3.0
    z = x.to(C128)
    return x, torch.where(x > R0, R0 + (x - R0) * complex(math.cos(THETA), math.sin(THETA)), z)


class Problem:
    """Potentials and source of one problem; the seed moves the charge by up to 1% and draws
    the source noise."""

    def __init__(self, c, seed, nx=None, ny=None, L=None, E=None):
        self.nx, self.ny = nx or c["nx"], ny or c["ny"]
        self.L, self.E = L or c["L"], E or c["E"]
        gen = torch.Generator(device="cuda")
        gen.manual_seed(int(seed))
        self.Z = 1.0 + 0.01 * (2.0 * float(torch.rand((), generator=gen, device="cuda", dtype=torch.float64)) - 1.0)
        x, zx = _nodes(self.nx, self.L)
        y, zy = _nodes(self.ny, self.L)
        self.v1, self.v2 = -self.Z / zx, -self.Z / zy
        zmax = torch.where(x[None, :] >= y[:, None], zx[None, :], zy[:, None])
        self.v12 = (1.0 / zmax).contiguous()
        k = math.sqrt(2.0 * self.E)
        src = 2.0 * zx[None, :] * torch.exp(-zx)[None, :] * (1.0 / zmax - 1.0 / zy[:, None]) * torch.sin(k * zy)[:, None]
        self.f = (src + 1e-3 * _rand(src.shape, gen)).contiguous()
        self.gen = gen

    def params(self, c, precision=None):
        R0 = 2.0 * self.L / 3.0
        return M.make_params(self.nx, self.ny, self.L, self.L, R0, R0, THETA, self.E, levels=c["levels"], nu1=c["nu1"],
                             nu2=c["nu2"], n_b=c["n_b"], krylov_restart=20,
                             precision=c["precision"] if precision is None else precision)

    def solver(self, c, **kw):
        return M.Solver(self.params(c), self.v1, self.v2, self.v12, **kw)


def _batch_member(c, seed, q):
    """Problem q of a batch: its own energy, and a grid that halves and thirds around the case's."""
    s = 1 << (c["levels"] - 1)
    nx = max(16, int(c["nx"] * (1.0, 2.0 / 3.0, 5.0 / 6.0)[q % 3]) // s) * s
    E = c["E"] * (0.8 + 0.4 * q / max(1, c["count"] - 1))
    return Problem(c, 1000 * seed + q, nx=nx, ny=nx, L=c["L"] * nx / c["nx"], E=E)


def _gradient_args(c, P):
    n, L = P.nx, P.L
    x = torch.arange(1, n, dtype=torch.float64, device="cuda") * (L / n)
    w = torch.exp(-(x - L / 2) ** 2 / 8.0)
    dV = 1e-2 * torch.randn((n - 1, n - 1), generator=P.gen, device="cuda", dtype=torch.float64)
    geom = {"n": n, "L": L, "R0": 2.0 * L / 3.0, "theta": THETA}
    kw = {"levels": c["levels"], "nu1": c["nu1"], "nu2": c["nu2"], "n_b": c["n_b"], "krylov_restart": 20,
          "precision": c["precision"]}
    return dV, (w[None, :] * w[:, None]).to(C128).contiguous(), geom, kw


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        S = {"case": case, "probs": [_batch_member(case, seed, q) for q in range(case["count"])]}
        S["solvers"] = [P.solver(case, stream=torch.cuda.Stream()) for P in S["probs"]]
        S["u"] = [torch.zeros_like(P.f) for P in S["probs"]]
        torch.cuda.synchronize()
        S["batch"] = M.Batch(S["solvers"], S["u"], [P.f for P in S["probs"]])
        return S
    P = Problem(case, seed)
    S = {"case": case, "prob": P, "u": torch.zeros_like(P.f), "z": torch.zeros_like(P.f)}
    if kind in ("precond", "iterate", "arnoldi", "solve"):
        S["solver"] = P.solver(case)
    if kind == "iterate":
        S["u0"] = _rand(P.f.shape, P.gen)
    if kind == "arnoldi":
        n, ld = P.f.numel(), (P.f.numel() + 31) // 32 * 32
        dt = C64 if case["precision"] else C128
        # a basis of near-orthonormal random vectors in the solver's padded layout
        V = torch.zeros((case["k"], ld), dtype=dt, device="cuda")
        V[:, :n] = (_rand((case["k"], n), P.gen) / math.sqrt(2.0 * n)).to(dt)
        S["V"], S["h"] = V, torch.zeros(case["k"], dtype=C128, device="cuda")
        S["x"] = _rand(P.f.shape, P.gen) / math.sqrt(2.0 * n)
        S["w0"] = (_rand(P.f.shape, P.gen) / math.sqrt(2.0 * n)).to(dt).reshape(-1) + V[0, :n]
        S["w"] = torch.zeros_like(S["w0"])
    if kind == "energy":
        P.solver(case, reuse_states=True).close()      # the scan's first point left its states behind
    if kind == "gradient":
        S["dV"], S["g"], S["geom"], S["kw"] = _gradient_args(case, P)
    return S


def run(S):
    c = S["case"]
    kind = c["kind"]
    if kind == "batch":
        for u in S["u"]:
            u.zero_()
        S["batch"].run(rtol=c["rtol"], max_iter=600)
        return S["u"]
    P, u = S["prob"], S["u"]
    if kind == "precond":
        S["solver"].precond_apply(S["z"], P.f)
        # a mixed handle's result is the widening of complex64 values
        return S["z"].to(C64) if c["precision"] else S["z"]
    if kind == "iterate":
        u.copy_(S["u0"])
        S["solver"].vcycle(u, P.f)
        S["solver"].cccs(u, P.f)
        return u
    if kind == "arnoldi":
        sv, w, h = S["solver"], S["w"], S["h"]
        if c["precision"]:
            w.copy_(S["w0"])
            sv.gs_dots_c64(S["V"], c["k"], w, h)
            sv.gs_update_c64(S["V"], c["k"], h, w)
            return w, h.to(C64)                          # sums of complex64 products
        sv.matvec(S["x"], w)
        sv.gs_dots(S["V"], c["k"], w, h)
        sv.gs_update(S["V"], c["k"], h, w)
        return w, h
    if kind == "solve":
        u.zero_()
        S["solver"].solve(u, P.f, rtol=c["rtol"], max_iter=600)
        return u
    if kind == "setup":
        sv = P.solver(c)
        sv.precond_apply(S["z"], P.f)
        out = list(sv.bound_states()) + [S["z"].to(C64) if c["precision"] else S["z"]]
        sv.close()
        return out
    if kind == "energy":
        sv = P.solver(c, reuse_states=True)
        u.zero_()
        sv.solve(u, P.f, rtol=c["rtol"], max_iter=600)
        sv.close()
        return u
    r = adjoint.amplitude_and_gradients(P.E, P.Z, S["dV"], P.f, S["g"], S["geom"], S["kw"], rtol=c["rtol"])
    return [complex(r["J"]).real, complex(r["J"]).imag] + [np.array([r["dE"], r["dZ"]]), r["ddV"], r["u"], r["mu"]]


# ---------------------------------------------------------------- what a pass cannot do without

def _iteration_flops(n, c):
    """FP operations of one V(nu1,nu2) cycle (real coefficients in the box) and one CCCS."""
    return n * (4.0 / 3.0 * (18.0 * (c["nu1"] + c["nu2"]) + 22.0 + 4.5 + 4.0) + (22.0 + 32.0 * c["n_b"] if c["n_b"] else 0))


def work(case):
    e = 8.0 if case["precision"] and case["kind"] != "batch" else 16.0
    n = float((case["nx"] - 1) * (case["ny"] - 1))
    kind = case["kind"]
    it = _iteration_flops(n, case)
    if kind == "batch":
        sizes = [_batch_nx(case, q) for q in range(case["count"])]
        n = float(sum((s - 1) ** 2 for s in sizes))
        return {"bytes": 48.0 * n, "flops": _iteration_flops(n, case)}
    if kind == "arnoldi":
        return {"bytes": n * (e * (case["k"] + 2) + (0.0 if case["precision"] else 32.0)),
                "flops": n * (16.0 * case["k"] + (0.0 if case["precision"] else 22.0))}
    if kind == "iterate":
        return {"bytes": 64.0 * n, "flops": it}
    if kind == "precond":
        return {"bytes": 32.0 * n + e * n, "flops": it}
    if kind == "setup":
        return {"bytes": 48.0 * n + 32.0 * case["n_b"] * (case["nx"] + case["ny"]), "flops": it}
    if kind == "gradient":
        return {"bytes": 16.0 * n * 6 + 8.0 * n, "flops": 2.0 * it}
    return {"bytes": 48.0 * n, "flops": it}            # a solve: potential and source in, u out; at least one step


def _batch_nx(c, q):
    s = 1 << (c["levels"] - 1)
    return max(16, int(c["nx"] * (1.0, 2.0 / 3.0, 5.0 / 6.0)[q % 3]) // s) * s


# ---------------------------------------------------------------- the method in plain torch

class _Axis:
    """Second-difference coefficients of one axis of one level."""

    def __init__(self, n, L, gamma):
        x = np.arange(n + 1) * (L / n)
        R0 = 2.0 * L / 3.0
        z = x.astype(np.complex128)
        far = x > R0
        z[far] = R0 + (x[far] - R0) * np.exp(1j * THETA)
        z = z * np.exp(1j * gamma) if gamma else z
        h = np.diff(z)
        s = h[:-1] + h[1:]
        self.west, self.east = -1.0 / (s * h[:-1]), -1.0 / (s * h[1:])
        self.diag, self.w = -(self.west + self.east), 0.5 * s


def _t(a):
    return torch.as_tensor(np.ascontiguousarray(a)).to("cuda")


def _operator(P, l, v12):
    """West, east, south and north couplings and the diagonal of level l."""
    ax, ay = (_Axis(n >> l, P.L, GAMMA if l else 0.0) for n in (P.nx, P.ny))
    s = 1 << l
    D = _t(ax.diag)[None, :] + _t(ay.diag)[:, None] + P.v1[s - 1::s][None, :] + P.v2[s - 1::s][:, None] \
        + v12[s - 1::s, s - 1::s] - P.E
    return _t(ax.west), _t(ax.east), _t(ay.west)[:, None], _t(ay.east)[:, None], D


def _apply(op, u):
    W, E, S, N, D = op
    r = D * u
    r[:, 1:] += W[1:] * u[:, :-1]
    r[:, :-1] += E[:-1] * u[:, 1:]
    r[1:] += S[1:] * u[:-1]
    r[:-1] += N[:-1] * u[1:]
    return r


class Plain:
    """One MG-CCCS preconditioner as the paper states it, complex128 throughout."""

    def __init__(self, c, P, extra=None):
        self.c, self.P = c, P
        v12 = P.v12 if extra is None else P.v12 + extra
        self.ops = [_operator(P, l, v12) for l in range(c["levels"])]
        W, E, S, N, D = self.ops[-1]
        my, mx = D.shape
        A = torch.diag(D.reshape(-1))
        p = torch.arange(mx * my, device="cuda").reshape(my, mx)
        A[p[:, 1:], p[:, :-1]] = W[1:].expand(my, -1)
        A[p[:, :-1], p[:, 1:]] = E[:-1].expand(my, -1)
        A[p[1:], p[:-1]] = S[1:].expand(-1, mx)
        A[p[:-1], p[1:]] = N[:-1].expand(-1, mx)
        self.coarse = torch.linalg.lu_factor(A)
        if c["n_b"]:
            self._channels(v12)

    def vcycle(self, l, u, f):
        if l == len(self.ops) - 1:
            return torch.linalg.lu_solve(*self.coarse, f.reshape(-1, 1)).reshape(f.shape)
        D = self.ops[l][4]
        for _ in range(self.c["nu1"]):
            u = u + OMEGA / D * (f - _apply(self.ops[l], u))
        r = f - _apply(self.ops[l], u)
        r = 0.25 * (r[0:-2:2] + 2.0 * r[1:-1:2] + r[2::2])
        r = 0.25 * (r[:, 0:-2:2] + 2.0 * r[:, 1:-1:2] + r[:, 2::2])
        e = self.vcycle(l + 1, torch.zeros_like(r), r)
        for axis in (0, 1):
            e = e.movedim(axis, 0)
            g = torch.zeros((2 * e.shape[0] + 1,) + e.shape[1:], dtype=C128, device="cuda")
            g[1::2] = e
            g[0:-2:2] += 0.5 * e
            g[2::2] += 0.5 * e
            e = g.movedim(0, axis)
        u = u + e
        for _ in range(self.c["nu2"]):
            u = u + OMEGA / D * (f - _apply(self.ops[l], u))
        return u

    def states(self, n, v):
        """The n_b eigenpairs of the axis operator with the smallest real parts."""
        nb, a = self.c["n_b"], _Axis(n, self.P.L, 0.0)

        def dense(a, v):
            return np.diag(a.diag + v) + np.diag(a.west[1:], -1) + np.diag(a.east[:-1], 1)

        half = n > 1100 and n % 2 == 0
        b = _Axis(n // 2, self.P.L, 0.0) if half else a
        ev = np.linalg.eigvals(dense(b, v[1::2] if half else v))
        ev = ev[np.argsort(ev.real)][:nb + (2 if half else 0)]
        H, w = _t(dense(a, v)), _t(a.w)
        I, got = torch.eye(n - 1, dtype=C128, device="cuda"), []
        for lam in ev:
            lam = complex(lam) * (1 + 1e-9)
            x = torch.ones((n - 1, 1), dtype=C128, device="cuda")
            for it in range(8):
                x = torch.linalg.solve(H - lam * I, x)
                x = x / x.abs().max()
                new = complex((w[:, None] * x * (H @ x)).sum() / (w[:, None] * x * x).sum())
                if it >= 2:
                    lam, last = new * (1 + 1e-13) if it < 6 else new, new
            x = x[:, 0] / torch.sqrt((w * x[:, 0] ** 2).sum())
            x = -x if float(x[x.abs().argmax()].real) < 0 else x
            got.append((last, x))
        got = sorted(got, key=lambda t: t[0].real)[:nb]
        return np.array([t[0] for t in got]), torch.stack([t[1] for t in got]), w

    def _channels(self, v12):
        P = self.P
        v1, v2 = P.v1.cpu().numpy(), P.v2.cpu().numpy()
        self.lam, self.phi, wx = self.states(P.nx, v1)
        same = P.nx == P.ny
        self.mu, self.vphi, wy = (self.lam, self.phi, wx) if same else self.states(P.ny, v2)
        self.wphi, self.wvphi = wx * self.phi, wy * self.vphi
        VA = torch.einsum("ai,bi,ji->jab", self.wphi, self.phi, v12).cpu().numpy()
        VB = torch.einsum("aj,bj,ji->iab", self.wvphi, self.vphi, v12).cpu().numpy()
        self.sysA = self._factor(_Axis(P.ny, P.L, 0.0), v2 - P.E, self.lam, VA)
        self.sysB = self._factor(_Axis(P.nx, P.L, 0.0), v1 - P.E, self.mu, VB)

    def _factor(self, a, v, lam, V):
        """Block Thomas factors of the coupled-channel system along one axis."""
        nb, m = self.c["n_b"], len(a.diag)
        B = V + np.eye(nb) * (a.diag + v)[:, None, None] + np.diag(lam)
        inv = np.empty_like(B)
        inv[0] = np.linalg.inv(B[0])
        for k in range(1, m):
            inv[k] = np.linalg.inv(B[k] - a.west[k] * a.east[k - 1] * inv[k - 1])
        return a, inv

    @staticmethod
    def _channel_solve(sys, r):
        a, inv = sys
        x = r.T.cpu().numpy().copy()
        m = len(x)
        for k in range(1, m):
            x[k] -= a.west[k] * (inv[k - 1] @ x[k - 1])
        x[m - 1] = inv[m - 1] @ x[m - 1]
        for k in range(m - 2, -1, -1):
            x[k] = inv[k] @ (x[k] - a.east[k] * x[k + 1])
        return _t(x.T)

    def cccs(self, u, f):
        r = f - _apply(self.ops[0], u)
        Px, Py = self.wphi @ r.T, self.wvphi @ r
        cm = Px @ self.wvphi.T
        nb = self.c["n_b"]
        up = torch.triu(torch.ones((nb, nb), device="cuda"), 1).to(C128)
        eA = self._channel_solve(self.sysA, Px - (cm * up) @ self.vphi)
        eB = self._channel_solve(self.sysB, Py - (cm * (1 - up)).T @ self.phi)
        return u + eA.T @ self.phi + self.vphi.T @ eB

    def precond(self, f):
        z = self.vcycle(0, torch.zeros_like(f), f)
        return self.cccs(z, f) if self.c["n_b"] else z

    def solve(self, f, m=40):
        """GMRES to the rounding level of the residual."""
        u, shape, best = torch.zeros_like(f), f.shape, math.inf
        fn = float(torch.linalg.vector_norm(f))
        for _ in range(12):
            r = f - _apply(self.ops[0], u)
            beta = float(torch.linalg.vector_norm(r))
            if beta <= 3e-14 * fn or beta > 0.5 * best:
                break
            best = beta
            V = torch.zeros((m + 1, f.numel()), dtype=C128, device="cuda")
            Z = torch.zeros((m, f.numel()), dtype=C128, device="cuda")
            H = np.zeros((m + 1, m), dtype=np.complex128)
            V[0] = r.reshape(-1) / beta
            for j in range(m):
                z = self.precond(V[j].reshape(shape))
                Z[j] = z.reshape(-1)
                w = _apply(self.ops[0], z).reshape(-1)
                for _ in range(2):
                    h = (V[:j + 1] * w.conj()).sum(1).conj()
                    w = w - h @ V[:j + 1]
                    H[:j + 1, j] += h.cpu().numpy()
                H[j + 1, j] = float(torch.linalg.vector_norm(w))
                V[j + 1] = w / H[j + 1, j].real
                e = np.zeros(j + 2, dtype=np.complex128)
                e[0] = beta
                y = np.linalg.lstsq(H[:j + 2, :j + 1], e, rcond=None)[0]
                if np.linalg.norm(e - H[:j + 2, :j + 1] @ y) <= max(1e-14 * fn, 1e-10 * beta):
                    break
            u = u + (_t(y) @ Z[:len(y)]).reshape(shape)
        return u


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        probs = [_batch_member(case, seed, q) for q in range(case["count"])]
        return [Plain(case, P).solve(P.f) for P in probs]
    S = None
    if kind in ("iterate", "arnoldi"):
        S = prepare(case, seed)
        P = S["prob"]
    else:
        P = Problem(case, seed)
    if kind == "arnoldi":
        n, V = P.f.numel(), S["V"]
        if case["precision"]:
            w = S["w0"].to(C128)
        else:
            w = _apply(_operator(P, 0, P.v12), S["x"]).reshape(-1)
        h = torch.stack([(V[i, :n].to(C128).conj() * w).sum() for i in range(case["k"])])
        for i in range(case["k"]):
            w = w - h[i] * V[i, :n].to(C128)
        return w, h
    if kind == "gradient":
        dV, g, geom, kw = _gradient_args(case, P)
        A = Plain(case, P, extra=dV.to(C128))
        u, mu = A.solve(P.f), A.solve(g)
        a = _Axis(P.nx, P.L, 0.0)
        W = _t(a.w)[:, None] * _t(a.w)[None, :]
        zx = _nodes(P.nx, P.L)[1]
        J, dE = (complex((W * b * u).sum()) for b in (g, mu))
        dZ = -complex((W * mu * u * (-1.0 / zx[None, :] - 1.0 / zx[:, None])).sum())
        return [J.real, J.imag, np.array([dE, dZ]), -W * mu * u, u, mu]
    A = Plain(case, P)
    if kind == "precond":
        return A.precond(P.f)
    if kind == "iterate":
        return A.cccs(A.vcycle(0, S["u0"], P.f), P.f)
    if kind == "setup":
        return [A.lam, A.phi, A.mu, A.vphi, A.precond(P.f)]
    return A.solve(P.f)
