"""The V-cycle's sums on the integer pipes leave no mean: a constant error per node is a smooth
residual, which the coarser levels amplify by the operator's condition.

V-cycles on rough data against the same cycle in extended precision with the device's own
coefficients, read through the one-step residual: each pass rounds as often as the one-step FP64
kernels, so its error is within 1.5 times theirs."""
import math

import numpy as np
import pytest

from paper_1412_1953_gb300 import build, inputs
from paper_1412_1953_gb300 import mgcccs as M

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]
E = np.clongdouble


def _problem(nx, ny):
    return inputs.temkin_poet(nx, L=30.0, R0=20.0, theta=math.pi / 6, E=0.5, seed=3, ny=ny)


def _coefficients(sv, l, shape):
    """Centre, west, east, south and north of every node: a node and its neighbours differ in colour."""
    colour = np.add.outer(2 * np.arange(shape[0]), np.arange(shape[1])) % 5
    out = [np.zeros(shape, E) for _ in range(5)]
    for c in range(5):
        x = torch.as_tensor((colour == c).astype(complex).ravel()).to("cuda")
        r = torch.empty_like(x)
        sv.level_residual(l, x, torch.zeros_like(x), r)
        r = -r.cpu().numpy().reshape(shape)
        for o, step in zip(out, (0, -1, 1, -2, 2)):
            o[(colour + step) % 5 == c] = r[(colour + step) % 5 == c]
    return out


def _apply(A, v):
    d, w, e, s, n = A
    r = d * v
    r[:, 1:] += w[:, 1:] * v[:, :-1]
    r[:, :-1] += e[:, :-1] * v[:, 1:]
    r[1:] += s[1:] * v[:-1]
    r[:-1] += n[:-1] * v[1:]
    return r


def _two_grid(sv, A, u, f, nu1, nu2, correct):
    w = E(2) / 3 / A[0]
    for _ in range(nu1):
        u = u + w * (f - _apply(A, u))
    r = f - _apply(A, u)
    for ax in (0, 1):
        r = np.moveaxis(r, ax, 0)
        r = np.moveaxis((r[0:-2:2] + 2 * r[1:-1:2] + r[2::2]) / 4, 0, ax)
    e = correct(r)
    for ax in (0, 1):
        e = np.moveaxis(e, ax, 0)
        g = np.zeros((2 * e.shape[0] + 1,) + e.shape[1:], dtype=E)
        g[1::2] = e
        g[0:-2:2] += e / 2
        g[2::2] += e / 2
        e = np.moveaxis(g, 0, ax)
    u = u + e
    for _ in range(nu2):
        u = u + w * (f - _apply(A, u))
    return u


@pytest.mark.parametrize("nx,ny,levels,nu1,nu2", [(256, 256, 4, 1, 1), (592, 432, 5, 2, 1)])
def test_cycle_error_is_that_of_fp64(nx, ny, levels, nu1, nu2):
    build.build()
    prob = _problem(nx, ny)
    sv = M.Solver(M.params_for(prob, levels=levels, nu1=nu1, nu2=nu2, n_b=0), prob.v1, prob.v2, prob.v12)
    shapes = [prob.f.shape]
    for _ in range(levels - 1):
        shapes.append(tuple((n - 1) // 2 for n in shapes[-1]))
    A = [_coefficients(sv, l, s) for l, s in enumerate(shapes)]
    n = shapes[-1][0] * shapes[-1][1]
    A64 = [a.astype(np.complex128) for a in A[-1]]
    inv = np.linalg.inv(np.stack([_apply(A64, e.reshape(shapes[-1])).ravel() for e in np.eye(n, dtype=complex)], 1))

    def coarsest(f):
        x = np.zeros_like(f)
        for _ in range(4):
            x = x + (inv @ (f - _apply(A[-1], x)).ravel().astype(complex)).reshape(f.shape)
        return x

    def cycle(l, u, f):
        if l == levels - 1:
            return coarsest(f)
        return _two_grid(sv, A[l], u, f, nu1, nu2,
                         lambda r: cycle(l + 1, np.zeros_like(r), r))

    g = np.random.default_rng(7)
    start = g.standard_normal(prob.f.shape) + 1j * g.standard_normal(prob.f.shape)
    ref = cycle(0, start.astype(E), prob.f.astype(E))
    f = torch.as_tensor(prob.f).to("cuda")
    u = torch.as_tensor(start).to("cuda")
    # the one-step calls, which use FP64 instructions
    zeros = lambda l: torch.zeros(sv.level_size(l), dtype=torch.complex128, device="cuda")
    fs, us = [f.reshape(-1)], []
    for l in range(levels - 1):
        v = u.reshape(-1).clone() if l == 0 else zeros(l)
        sv.smooth(l, v, fs[l], nu1)
        r, fc = zeros(l), zeros(l + 1)
        sv.level_residual(l, v, fs[l], r)
        sv.restrict(l, r, fc)
        us.append(v)
        fs.append(fc)
    e = zeros(levels - 1)
    sv.coarse_solve(fs[-1], e)
    for l in reversed(range(levels - 1)):
        sv.prolong_add(l, e, us[l])
        sv.smooth(l, us[l], fs[l], nu2)
        e = us[l]
    sv.vcycle(u, f)
    torch.cuda.synchronize()
    off = lambda x: float(np.linalg.norm((x.cpu().numpy().reshape(ref.shape) - ref).astype(complex)))
    assert off(u) <= 1.5 * off(e)
    sv.close()
