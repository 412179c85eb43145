"""Setup kernels at the sizes where their split can go wrong: the eigenvalue iteration's lanes per
approximation, the bound states' scan over threads (odd, tiny, and beyond shared memory), the
channel factors for every block size the library takes, and the block-wise dense inverse in both
orderings with its fallback."""
import math

import numpy as np
import pytest

from oracle import mgcccs_oracle as O
from paper_1412_1953_gb300 import build, inputs
from paper_1412_1953_gb300 import mgcccs as M

torch = pytest.importorskip("torch")
scipy_opt = pytest.importorskip("scipy.optimize")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()


def _problem(nx, ny=None):
    L = 30.0 * nx / 128 if nx <= 128 else 30.0
    return inputs.temkin_poet(nx, L=L, R0=2 * L / 3, theta=math.pi / 6, E=0.5, seed=3, ny=ny)


def _dense_axis(n, prob, v):
    return O.tridiag_1d(O.make_axis(n, prob.Lx, prob.R0x, prob.theta), v).toarray()


# lanes per approximation follow from the row count and the block size: one row block short of,
# at and beyond a power of two, and few enough rows for 32 lanes or so many that only 8 are used
@pytest.mark.parametrize("n", [3, 6, 34, 66, 130, 500, 1300])
def test_spectrum_sizes(n):
    prob = _problem(n, 2 if n % 2 else 4)
    sv = M.Solver(M.params_for(prob, levels=1 if n % 2 else 2, n_b=0), prob.v1, prob.v2, prob.v12)
    ev = np.linalg.eigvals(_dense_axis(n, prob, prob.v1))
    lam = sv.axis_spectrum(0, method=0)
    D = np.abs(lam[:, None] - ev[None, :])
    r, c = scipy_opt.linear_sum_assignment(D)
    assert D[r, c].max() <= 1e-11 * np.abs(ev).max()


# residual of the eigenpairs: backward errors of a few units in the last place of the matrix
# scale; 4095 rows do not fit in shared memory, 300 are no multiple of the threads
@pytest.mark.parametrize("nx,ny,levels,nb", [(4, 4, 1, 2), (6, 10, 1, 4), (301, 4, 1, 3), (608, 304, 5, 6),
                                             (4096, 128, 7, 2)])
def test_bound_state_residuals(nx, ny, levels, nb):
    prob = _problem(nx, ny)
    sv = M.Solver(M.params_for(prob, levels=levels, n_b=nb), prob.v1, prob.v2, prob.v12)
    assert sv.eig_fallbacks() == 0
    lam, phi, mu, vphi = sv.bound_states()
    for n, v, l, p, R0, L in ((nx, prob.v1, lam, phi, prob.R0x, prob.Lx), (ny, prob.v2, mu, vphi, prob.R0y, prob.Ly)):
        ax = O.make_axis(n, L, R0, prob.theta)
        H = O.tridiag_1d(ax, v)
        p = p.cpu().numpy()
        scale = np.abs(H.diagonal()).max()
        assert np.all(np.diff(l.real) >= 0)
        for k in range(nb):
            assert np.abs(H @ p[k] - l[k] * p[k]).max() <= 16 * 2.0 ** -52 * scale * np.abs(p[k]).max()
            assert abs((ax.w * p[k] ** 2).sum() - 1) <= 1e-12
            assert p[k][np.abs(p[k]).argmax()].real > 0
        if n <= 700:
            ev = np.linalg.eigvals(H.toarray())
            ev = ev[np.argsort(ev.real)][:nb]
            assert np.abs(np.sort(l.real) - ev.real).max() <= 1e-11 * scale


# every block size, rows short of and beyond a multiple of the rows per block, and (from 128 rows
# on, by n_b) one to four elimination levels with different counts on the two axes
@pytest.mark.parametrize("nx,ny,nb", [(16, 24, 1), (24, 16, 2), (40, 24, 4), (64, 72, 5), (48, 64, 7), (72, 40, 8),
                                      (4, 4, 2), (152, 248, 8), (496, 208, 4), (368, 496, 6)])
def test_channel_factors(nx, ny, nb):
    prob = _problem(nx, ny)
    levels = 1 if nx < 8 else 4 if nx > 128 else 3
    so = O.Solver(O.params_from_problem(prob, levels=levels, n_b=nb), prob.v1, prob.v2, prob.v12)
    sg = M.Solver(M.params_for(prob, levels=levels, n_b=nb), prob.v1, prob.v2, prob.v12)
    g = np.random.default_rng(nb)
    u = g.standard_normal(prob.f.shape) + 1j * g.standard_normal(prob.f.shape)
    ud = torch.as_tensor(u).to("cuda")
    sg.cccs(ud, torch.as_tensor(prob.f).to("cuda"))
    ref = so.cccs(u, prob.f)
    # the bound of the oracle parity tests (1e-11 at up to 6 states), for up to 8 near-continuum states
    assert np.abs(ud.cpu().numpy() - ref).max() <= 1e-10 * np.abs(ref).max()


@pytest.mark.parametrize("nx,ny", [(2, 2), (3, 2), (2, 1025), (1025, 2), (33, 33), (33, 20), (20, 33), (9, 114),
                                   (129, 5), (5, 8)])
def test_dense_inverse_shapes(nx, ny):
    prob = _problem(nx, ny)
    sv = M.Solver(M.params_for(prob, levels=1, n_b=0), prob.v1, prob.v2, prob.v12)
    so = O.Solver(O.params_from_problem(prob, levels=1, n_b=0), prob.v1, prob.v2, prob.v12)
    g = np.random.default_rng(nx + ny)
    f = g.standard_normal(prob.f.shape) + 1j * g.standard_normal(prob.f.shape)
    u = torch.empty(prob.f.shape, dtype=torch.complex128, device="cuda")
    sv.coarse_solve(torch.as_tensor(f).to("cuda"), u)
    u = u.cpu().numpy()
    A = O.assemble_unweighted(so.levels[0])
    # normwise backward error
    assert np.abs(A @ u.ravel() - f.ravel()).max() <= 1e-13 * (abs(A).sum(1).max() * np.abs(u).max() + np.abs(f).max())


def test_dense_inverse_with_a_singular_block():
    """The first row of the grid alone is singular to rounding, the operator is not: elimination
    within block rows meets a tiny pivot, and setup falls back to pivoting over all rows."""
    prob = _problem(4, 4)
    lev = O.Solver(O.params_from_problem(prob, levels=1, n_b=0), prob.v1, prob.v2, prob.v12).levels[0]
    D = lev.diagonal()
    west, east = lev.ax.west, lev.ax.east
    v12 = prob.v12.copy()
    # the determinant of the first 3 x 3 row block becomes zero
    v12[0, 0] += east[0] * west[1] / (D[0, 1] - east[1] * west[2] / D[0, 2]) - D[0, 0]
    so = O.Solver(O.params_from_problem(prob, levels=1, n_b=0), prob.v1, prob.v2, v12)
    A = O.assemble_unweighted(so.levels[0]).toarray()
    sv = M.Solver(M.params_for(prob, levels=1, n_b=0), prob.v1, prob.v2, v12)
    f = np.arange(9).reshape(3, 3) + 1j
    u = torch.empty((3, 3), dtype=torch.complex128, device="cuda")
    sv.coarse_solve(torch.as_tensor(f).to("cuda"), u)
    ref = np.linalg.solve(A, f.ravel()).reshape(3, 3)
    assert np.abs(u.cpu().numpy() - ref).max() <= 1e-13 * np.linalg.cond(A) * np.abs(ref).max()
