"""The complex128 level passes that run on the integer pipes (levels of at least 60000 nodes whose
coefficients share an exponent) against the same cycle composed from the one-step C-ABI calls, which
use FP64 instructions: ragged tiles, non-square grids, sweep counts that take every branch, values
scaled into the range where the passes use FP64 instructions themselves, a level whose diagonal is
spread too far, and NaN.

Bound: each pass rounds values to 2^-57 of its tile's largest and its results to doubles, the one-step
kernels round each operation to 2^-53 of its result; a cycle amplifies either by the operator's norm
over the smoothed part, so the two agree to 1e-13 of the largest value (the composed cycles of the FP64
passes are held to 1e-14 at a sixteenth of these sizes)."""
import math

import numpy as np
import pytest

from paper_1412_1953_gb300 import build, inputs
from paper_1412_1953_gb300 import mgcccs as M

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()


def _composed(sv, levels, f, u, nu1, nu2):
    """V(nu1, nu2) from u by the one-step calls."""
    zeros = lambda l: torch.zeros(sv.level_size(l), dtype=torch.complex128, device="cuda")
    fs, us = [f], []
    for l in range(levels - 1):
        v = u.clone() if l == 0 else zeros(l)
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
    return e


def _rel(a, b):
    torch.cuda.synchronize()
    return float((a - b).abs().max() / b.abs().max())


@pytest.mark.parametrize("nx,ny,levels,nu1,nu2", [(256, 256, 4, 1, 1), (320, 272, 4, 1, 1), (592, 432, 5, 2, 1),
                                                  (272, 320, 4, 1, 2), (320, 320, 4, 0, 1), (320, 256, 4, 1, 0)])
@pytest.mark.parametrize("scale,spike", [(1.0, 0.0), (2.0 ** 200, 0.0), (2.0 ** -480, 0.0), (1.0, 1e6)])
def test_cycle_equals_composed_steps(nx, ny, levels, nu1, nu2, scale, spike):
    prob = inputs.temkin_poet(nx, L=30.0, R0=20.0, theta=math.pi / 6, E=0.5, seed=3, ny=ny)
    v12 = prob.v12.copy()
    v12[ny // 3, nx // 5] += spike
    sv = M.Solver(M.params_for(prob, levels=levels, nu1=nu1, nu2=nu2, n_b=0), prob.v1, prob.v2, v12)
    g = np.random.default_rng(nx)
    f = torch.as_tensor(prob.f.reshape(-1) * scale).to("cuda")
    u0 = torch.as_tensor((g.standard_normal(f.numel()) + 1j * g.standard_normal(f.numel())) * scale).to("cuda")
    u = u0.clone()
    sv.vcycle(u, f)
    assert _rel(u, _composed(sv, levels, f, u0, nu1, nu2)) <= 1e-13
    z = torch.zeros_like(f)
    sv.precond_apply(z, f)
    assert _rel(z, _composed(sv, levels, f, torch.zeros_like(f), nu1, nu2)) <= 1e-13
    # the operator: f - (f - A u) from the FP64 residual
    y, r = torch.empty_like(f), torch.empty_like(f)
    sv.matvec(u0, y)
    sv.level_residual(0, u0, torch.zeros_like(f), r)
    assert _rel(y, -r) <= 1e-14
    sv.close()


def test_nan_spreads_only_as_far_as_the_stencils():
    prob = inputs.temkin_poet(320, L=30.0, R0=20.0, theta=math.pi / 6, E=0.5, seed=3)
    sv = M.Solver(M.params_for(prob, levels=4, n_b=0), prob.v1, prob.v2, prob.v12)
    f = torch.as_tensor(prob.f).to("cuda")
    x = f.clone()
    x[100, 200] = complex(np.nan, 0.0)
    y = torch.empty_like(f)
    sv.matvec(x, y)
    bad = ~torch.isfinite(torch.view_as_real(y)).all(-1)
    ref = torch.zeros_like(bad)
    ref[100, 199:202] = ref[99:102, 200] = True
    assert bool((bad == ref).all())
    z = torch.zeros_like(f)
    sv.precond_apply(z, x)
    assert not bool(torch.isfinite(torch.view_as_real(z)).any())     # the coarsest solve couples every node
