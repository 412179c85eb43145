"""The complex128 Gram-Schmidt pair, whose products are summed on the integer pipes, against
extended-precision sums: edges of the tiles and of the vector groups, operands of very different
size inside a tile, magnitudes for which it uses FP64 instructions, and non-finite entries.

Bounds, derived before the first run: a product carries 2^-56 of the largest one its warp has met,
a partial sum is rounded to 2^-53 of itself, and the block sums add a few units of 2^-53 of the
partial sums, so a dot product is good to 8 units of 2^-53 |V_i| |w|, and an entry of the update to
8 units of 2^-53 of the largest sum of absolute terms among the entries (both are normwise bounds
that FP64 multiply-adds meet as well)."""
import math

import numpy as np
import pytest

from paper_1412_1953_gb300 import build, inputs
from paper_1412_1953_gb300 import mgcccs as M

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]
EPS = 2.0 ** -53


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()


def _solver(nx, ny, m=60):
    prob = inputs.temkin_poet(nx, L=30.0, R0=20.0, theta=math.pi / 6, seed=1, ny=ny)
    return M.Solver(M.params_for(prob, levels=1 if nx * ny < 1100 else 5 if nx > 512 else 4, n_b=0, krylov_restart=m), prob.v1, prob.v2,
                    prob.v12)


def _ext(a):
    return np.asarray(a.real, dtype=np.longdouble), np.asarray(a.imag, dtype=np.longdouble)


def _run(sv, V, k, w):
    V, w0 = torch.as_tensor(V).to("cuda"), torch.as_tensor(w).to("cuda")
    h, w1 = torch.empty(k, dtype=torch.complex128, device="cuda"), w0.clone()
    sv.gs_dots(V, k, w0, h)
    sv.gs_update(V, k, h, w1)
    torch.cuda.synchronize()
    return h.cpu().numpy(), w1.cpu().numpy()


def _check(V, k, w, h, w1):
    n = w.size
    (vr, vi), (wr, wi), (hr, hi) = _ext(V[:k, :n]), _ext(w), _ext(h)
    dr, di = (vr * wr + vi * wi).sum(1), (vr * wi - vi * wr).sum(1)
    nv, nw = np.sqrt((vr ** 2 + vi ** 2).sum(1)), np.sqrt((wr ** 2 + wi ** 2).sum())
    assert np.all(np.hypot(hr - dr, hi - di) <= 8 * EPS * nv * nw)
    ur = wr - (hr[:, None] * vr - hi[:, None] * vi).sum(0)
    ui = wi - (hr[:, None] * vi + hi[:, None] * vr).sum(0)
    size = np.hypot(wr, wi) + (np.hypot(hr, hi)[:, None] * np.hypot(vr, vi)).sum(0)
    assert np.max(np.hypot(w1.real - ur, w1.imag - ui)) <= 8 * EPS * size.max()


# 1 to 961 points around the tiles of 64 and 128; 16641 and 130816 points on many blocks and, with
# four points a lane, several tiles a warp; 1 to 60 vectors around the groups of 4 and of 8 terms
@pytest.mark.parametrize("nx,ny,k", [(2, 2, 1), (2, 64, 3), (2, 66, 4), (9, 9, 5), (32, 32, 9), (136, 128, 60),
                                     (256, 512, 12), (1024, 512, 8)])
@pytest.mark.parametrize("kind", ["gauss", "decaying", "spikes"])
def test_pair_against_extended_sums(nx, ny, k, kind):
    sv = _solver(nx, ny)
    n, ld = sv.n, sv.n + 3
    g = np.random.default_rng(n + k)
    V = (g.standard_normal((k, ld)) + 1j * g.standard_normal((k, ld))) / math.sqrt(2 * n)
    w = (g.standard_normal(n) + 1j * g.standard_normal(n)) / math.sqrt(2 * n) + V[0, :n]
    if kind == "decaying":                            # 2^-100 over the vector, coefficients of all sizes
        f = np.exp2(-100.0 * np.arange(n) / n)
        V[:, :n] *= f
        w = w * f
        V *= np.exp2(-7.0 * np.arange(k))[:, None]
    if kind == "spikes":                              # neighbours 2^40 apart, zeros, a vector of zeros
        V[:, :n] *= np.where(g.random(n) < 0.05, 2.0 ** 20, 2.0 ** -20)
        w[::7] = 0.0
        V[k - 1] = 0.0
    h, w1 = _run(sv, V, k, w)
    _check(V, k, w, h, w1)


def test_scales_outside_the_integer_range():
    sv = _solver(32, 32)
    g = np.random.default_rng(5)
    n = sv.n
    V = g.standard_normal((3, n)) + 1j * g.standard_normal((3, n))
    w = g.standard_normal(n) + 1j * g.standard_normal(n)
    for sv_, sw in ((2.0 ** 600, 2.0 ** -300), (2.0 ** -500, 2.0 ** 450), (1.0, 2.0 ** -480)):
        h, w1 = _run(sv, V * sv_ / math.sqrt(n), 3, w * sw)
        _check(V * sv_ / math.sqrt(n), 3, w * sw, h, w1) if sv_ < 2.0 ** 100 else \
            np.testing.assert_allclose(h, (V.conj() @ w) * (sv_ * sw / math.sqrt(n)), rtol=1e-12)


def test_non_finite_entries_stay_where_they_belong():
    sv = _solver(32, 32)
    g = np.random.default_rng(6)
    n = sv.n
    V = (g.standard_normal((3, n)) + 1j * g.standard_normal((3, n))) / math.sqrt(n)
    w = g.standard_normal(n) + 1j * g.standard_normal(n)
    bad = V.copy()
    bad[1, 700] = complex(np.inf, 0.0)
    h, _ = _run(sv, bad, 3, w)
    assert not np.isfinite(h[1]) and np.isfinite(h[0]) and np.isfinite(h[2])
    c = torch.as_tensor(V[:, :3].copy().diagonal().copy()).to("cuda")
    wd = torch.as_tensor(w).to("cuda")
    sv.gs_update(torch.as_tensor(bad).to("cuda"), 3, c, wd)
    out = wd.cpu().numpy()
    fine = np.ones(n, bool)
    fine[700] = False
    assert not np.isfinite(out[700]) and np.all(np.isfinite(out[fine]))
    ref = w - c.cpu().numpy() @ V
    assert np.abs(out[fine] - ref[fine]).max() <= 1e-14 * np.abs(ref).max()
    nanw = w.copy()
    nanw[3] = np.nan
    h, w1 = _run(sv, V, 3, nanw)
    assert not np.any(np.isfinite(h)) and not np.any(np.isfinite(w1))


# tiles of 8, 16 and 32 rows (by the number of blocks), ragged last tiles, sums that carry (more
# than 8 products a node), sources scaled into the range of the FP64 instructions and back
@pytest.mark.parametrize("nx,ny,levels,nb", [(16, 24, 3, 1), (64, 136, 4, 8), (416, 432, 4, 5), (608, 592, 5, 3)])
@pytest.mark.parametrize("scale", [1.0, 2.0 ** 60, 2.0 ** -460])
def test_cccs_tiles(nx, ny, levels, nb, scale):
    from oracle import mgcccs_oracle as O
    L = 30.0 * nx / 128 if nx < 128 else 30.0
    prob = inputs.temkin_poet(nx, L=L, R0=2 * L / 3, theta=math.pi / 6, E=0.5, seed=4, ny=ny)
    so = O.Solver(O.params_from_problem(prob, levels=levels, n_b=nb), prob.v1, prob.v2, prob.v12)
    sg = M.Solver(M.params_for(prob, levels=levels, n_b=nb), prob.v1, prob.v2, prob.v12)
    g = np.random.default_rng(nx)
    u = g.standard_normal(prob.f.shape) + 1j * g.standard_normal(prob.f.shape)
    ref = so.cccs(u, prob.f)                           # linear in (u, f): a power of two scales exactly
    ud = torch.as_tensor(u * scale).to("cuda")
    sg.cccs(ud, torch.as_tensor(prob.f * scale).to("cuda"))
    # the bound of the oracle parity tests at these sizes
    assert np.abs(ud.cpu().numpy() / scale - ref).max() <= 1e-9 * np.abs(ref).max()
    ud = torch.as_tensor(u).to("cuda")
    ud[3, 5] = complex(np.nan, 0.0)
    sg.cccs(ud, torch.as_tensor(prob.f).to("cuda"))
    assert not bool(torch.isfinite(torch.view_as_real(ud)).any())    # a NaN reaches every node
