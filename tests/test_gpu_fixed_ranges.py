"""Complex128 results entry by entry, on operands of very different size side by side and on operators
with a small or widely spread diagonal: passes that sum on a common exponent must not lose what is
small beside what is large."""
import math

import numpy as np
import pytest

from paper_1412_1953_gb300 import build, inputs
from paper_1412_1953_gb300 import mgcccs as M
from test_gpu_fixed_bias import _apply, _coefficients

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()


def _problem(nx, ny, E=0.5):
    return inputs.temkin_poet(nx, L=30.0, R0=20.0, theta=math.pi / 6, E=E, seed=3, ny=ny)


def _solver(prob, levels, **kw):
    return M.Solver(M.params_for(prob, levels=levels, **{"n_b": 0, **kw}), prob.v1, prob.v2, prob.v12)


def _composed(sv, levels, f, u, nu1, nu2):
    """V(nu1, nu2) from u by the one-step calls, which use FP64 instructions."""
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
    return e.reshape(u.shape)


# An energy near the diagonal's 2/h^2, or a large omega, makes |omega/D| times a row's coefficients
# large: 14, 47, 72 and 32 against 2.7 (an update in 64-bit integers on v's unit wraps beyond 30).
# The two forms agree to 1e-13 at 2.7 (test_gpu_fixed_stencils.py); a sweep on either level amplifies a
# difference by this factor, 72/2.7 squared: 1e-10.
@pytest.mark.parametrize("E,omega", [(130.0, 2 / 3), (135.0, 2 / 3), (140.0, 2 / 3), (0.5, 8.0)])
def test_updates_beyond_64_bits(E, omega):
    prob = _problem(256, 256, E=E)
    sv = _solver(prob, 3, omega=omega, nu1=0, nu2=1)
    f = torch.full(prob.f.shape, 1e-3, dtype=torch.complex128, device="cuda")
    sign = torch.as_tensor(1.0 - 2.0 * (np.indices(prob.f.shape).sum(0) % 2)).to("cuda")
    for u0 in (torch.full_like(f, 1.9), 1.9 * sign.to(f.dtype)):
        u = u0.clone()
        sv.vcycle(u, f)
        ref = _composed(sv, 3, f, u0, 0, 1)
        assert float((u - ref).abs().max() / ref.abs().max()) <= 1e-10
    sv.close()


# Cells of aspect 1 to 4: the coefficients spread over 3 to 6 powers of two.  A unit vector's image is a
# column of coefficients: to half a unit of 2^-53 of its modulus in either part (the larger one exact),
# exact in the real box.
@pytest.mark.parametrize("nx,ny", [(256, 256), (512, 256), (768, 256), (1024, 256)])
def test_coefficients_keep_their_bits(nx, ny):
    prob = _problem(nx, ny)
    sv = _solver(prob, 5)
    x = torch.zeros(prob.f.shape, dtype=torch.complex128, device="cuda")
    x[1::4, 1::4] = 1.0                              # columns that do not meet
    y, r = torch.empty_like(x), torch.empty_like(x)
    sv.matvec(x, y)
    sv.level_residual(0, x.reshape(-1), torch.zeros(x.numel(), dtype=x.dtype, device="cuda"), r.reshape(-1))
    d = torch.view_as_real(y + r).abs().amax(-1)
    assert bool((d <= 2.0 ** -54 * r.abs()).all())
    box = (slice(0, ny * 2 // 3 - 2), slice(0, nx * 2 // 3 - 2))
    assert bool((y[box] == -r[box]).all())
    sv.close()


# Every rounding is to the nearest, so a cycle is odd to the last bit (ties, one in 2^28 sums, apart): a
# rounding towards one side would show in some 3% of the nodes, half of its unit in a double's 16.
@pytest.mark.parametrize("nx,ny,levels,nu1,nu2", [(256, 256, 4, 1, 1), (592, 432, 5, 0, 1)])
def test_cycle_is_odd(nx, ny, levels, nu1, nu2):
    prob = _problem(nx, ny)
    sv = _solver(prob, levels, nu1=nu1, nu2=nu2)
    g = np.random.default_rng(11)
    u = torch.as_tensor(g.standard_normal(prob.f.shape) + 1j * g.standard_normal(prob.f.shape)).to("cuda")
    f = torch.as_tensor(prob.f).to("cuda")
    v, z, zm = -u, torch.zeros_like(f), torch.zeros_like(f)
    sv.vcycle(u, f)
    sv.vcycle(v, -f)
    sv.precond_apply(z, f)
    sv.precond_apply(zm, -f)
    assert bool((u == -v).all()) and bool((z == -zm).all())
    sv.close()


def _field(kind, shape, g):
    """Values of very different size: entries of 2^60 among ones; 2^-2 a node along x, 2^-1 along y; parts of
    different size; zeros but for a few patches; standing waves with nodal lines."""
    u = g.standard_normal(shape) + 1j * g.standard_normal(shape)
    j, i = np.indices(shape)
    if kind == "spikes":
        u[::37, ::23] = 2.0 ** 60
    elif kind == "decaying":
        u *= np.exp2(-2.0 * (i % 250) - 1.0 * j)
    elif kind == "parts":
        u = u.real * 2.0 ** 50 + 1j * u.imag
    elif kind == "patches":
        u[(i // 10 + j // 10) % 7 > 0] = 0.0
    elif kind == "waves":
        u = np.sin(0.11 * i) * np.sin(0.07 * j) * (1.0 + 1j)
    return u


FIELDS = ["gauss", "spikes", "decaying", "parts", "patches", "waves"]


def _moduli(A, v, f=0.0):
    """|f| + the sum of the moduli of a node's five terms."""
    return np.abs(f) + _apply([np.abs(a) for a in A], np.abs(v))


# Ten multiply-adds a part are within 14 units of 2^-53 of the sum of moduli; up to 32 for sums in integers.
@pytest.mark.parametrize("kind", FIELDS)
def test_operator_entry_by_entry(kind):
    prob = _problem(320, 256)
    sv = _solver(prob, 4)
    A = _coefficients(sv, 0, prob.f.shape)
    x = _field(kind, prob.f.shape, np.random.default_rng(3))
    y = torch.empty(prob.f.shape, dtype=torch.complex128, device="cuda")
    sv.matvec(torch.as_tensor(x).to("cuda"), y)
    y, v = y.cpu().numpy(), x.astype(np.clongdouble)
    assert (np.abs(y - _apply(A, v)) <= 32 * 2.0 ** -53 * _moduli(A, v)).all()
    if kind == "parts":                              # real coefficients keep the parts apart
        box = (slice(0, 168), slice(0, 210))
        im = v.imag.astype(np.clongdouble)
        assert (np.abs(y.imag - _apply(A, im).real) <= 32 * 2.0 ** -53 * _moduli(A, im))[box].all()
    sv.close()


# At E = -200 the operator's inverse decays from node to node on every level, so more than 30 nodes from a
# spike of 2^70 an entry is far below the 2^13 that the last bit of its tile's largest is worth. There
# the cycle agrees with the one-step calls to 1e-12 of the largest entry within 4 nodes (1e-13 of the
# largest of all on ordinary data): both take the spike's remainder through the same coarse levels.
@pytest.mark.parametrize("nu1,nu2", [(1, 0), (0, 1), (1, 1)])
def test_cycle_beside_spikes(nu1, nu2):
    prob = _problem(256, 256, E=-200.0)
    sv = _solver(prob, 4, nu1=nu1, nu2=nu2)
    g = np.random.default_rng(17)
    shape = prob.f.shape
    far = np.ones(shape, bool)
    j, i = np.indices(shape)
    spikes = np.zeros(shape, complex)
    for b in range(0, shape[0], 64):
        for a in range(0, shape[1], 96):             # the corner of a 32 x 16 and of a 32 x 8 tile
            spikes[b, a] = 2.0 ** 70
            far &= abs(i - a) + abs(j - b) > 30
    f, u0 = (g.standard_normal(shape) + 1j * g.standard_normal(shape) for _ in range(2))
    far = torch.as_tensor(far).to("cuda")
    near = lambda x: torch.nn.functional.max_pool2d(x.abs()[None], 9, 1, 4)[0]   # the largest within 4 nodes
    for df, du in ((300.0, 0.0), (0.0, 1.0)):
        fd, u = (torch.as_tensor(x).to("cuda") for x in (300.0 * f + df * spikes, u0 + du * spikes))
        ref = _composed(sv, 4, fd, u, nu1, nu2)
        sv.vcycle(u, fd)
        assert bool(((u - ref).abs() <= 1e-12 * near(ref))[far].all())
        z = torch.zeros_like(fd)
        sv.precond_apply(z, fd)
        ref = _composed(sv, 4, fd, torch.zeros_like(fd), nu1, nu2)
        assert bool(((z - ref).abs() <= 1e-12 * near(ref))[far].all())
    sv.close()


# Without complex scaling and rotation everything is real, and the two parts are two separate cycles: one
# 2^-70 of the other is as precise as alone.
@pytest.mark.parametrize("nu1,nu2", [(1, 0), (0, 1), (1, 1)])
def test_parts_of_different_size(nu1, nu2):
    prob = inputs.temkin_poet(256, L=30.0, R0=30.0, theta=0.0, E=-400.0, seed=3, ny=256)
    sv = _solver(prob, 4, nu1=nu1, nu2=nu2, coarse_gamma=0.0)
    g = np.random.default_rng(19)
    f, u0 = (torch.as_tensor(g.standard_normal((2,) + prob.f.shape)).to("cuda") for _ in range(2))
    join = lambda a, s: torch.complex(a[0] * s, a[1])
    u, v = join(u0, 2.0 ** 70), join(u0, 1.0)
    sv.vcycle(u, join(f, 2.0 ** 79))
    sv.vcycle(v, join(f, 2.0 ** 9))
    assert float((u.real / 2.0 ** 70 - v.real).abs().max() / v.real.abs().max()) <= 1e-13
    f[1] *= 2.0 ** 9
    u, v = join(u0, 2.0 ** 70), join(u0, 1.0)
    sv.vcycle(u, join(f, 2.0 ** 79))
    sv.vcycle(v, join(f, 2.0 ** 9))
    assert float((u.imag - v.imag).abs().max() / v.imag.abs().max()) <= 1e-13
    sv.close()


# A spike of 2^60 where the states are 2^-22, in the corner of a tile of 32 columns and 32, 16 or 8 rows: 22
# nodes on, its share of the projections has decayed (by 2^-2.4 a node and more at these energies), and the rest of
# the row's (column's) projection comes from where the states are large.  The correction there
# agrees with the oracle's to 1e-9, the bound of the parity tests, of the largest within 4 nodes.
@pytest.mark.parametrize("n,E,rows", [(640, -800.0, 32), (512, -500.0, 16), (256, -200.0, 8)])
@pytest.mark.parametrize("where", ["f", "u"])
def test_correction_beside_a_spike(n, E, rows, where):
    from oracle import mgcccs_oracle as O
    prob = _problem(n, n, E=E)
    levels = 5
    so = O.Solver(O.params_from_problem(prob, levels=levels, n_b=1), prob.v1, prob.v2, prob.v12)
    sv = _solver(prob, levels, n_b=1)
    g = np.random.default_rng(n)
    f, u = (g.standard_normal(prob.f.shape) + 1j * g.standard_normal(prob.f.shape) for _ in range(2))
    f *= -E
    a = int(18.0 * n / 30.0) // 32 * 32
    if where == "f":
        f[a, a] = 2.0 ** 60
    else:
        u[a, a] = 2.0 ** 60
    ref = so.cccs(u, f) - u
    ud = torch.as_tensor(u).to("cuda")
    sv.cccs(ud, torch.as_tensor(f).to("cuda"))
    d = torch.as_tensor(ud.cpu().numpy() - u - ref)
    near = torch.nn.functional.max_pool2d(torch.as_tensor(ref).abs()[None], 9, 1, 4)[0]
    near += torch.as_tensor(np.abs(u)) * 1e-6            # the rounding of u itself
    own = slice(a + 22, a + 32)
    assert bool((d.abs() <= 1e-9 * near)[:a // 2, own].all())
    if rows == 32:
        assert bool((d.abs() <= 1e-9 * near)[own, :a // 2].all())
    sv.close()


def _basis(kind, k, n, g):
    """Vectors and w of ordinary size; entries of 2^45 and 2^-45 that meet the other's 2^-45 and 2^45; 2^-90 over
    the vector in one and growing in the other; spikes of 2^60 in the vectors only; a step of 2^80 on the way."""
    V, w = (g.standard_normal(s) + 1j * g.standard_normal(s) for s in ((k, n), (n,)))
    q = np.arange(n)
    if kind == "opposed":
        s = np.where(q % 3 == 0, 2.0 ** 45, 2.0 ** -45)
        V, w = V * s, w / s
    elif kind == "slopes":
        s = np.exp2(-90.0 * q / n)
        V, w = V * s, w / s
    elif kind == "spikes":
        V[:, ::997] *= 2.0 ** 60
        w[::997] = 0.0
    elif kind == "step":
        V[:, :n // 2] *= 2.0 ** 80
        w[:n // 2] *= 2.0 ** -80
    return V, w


BASES = ["gauss", "opposed", "slopes", "spikes", "step"]


# A dot product is good to a few units of 2^-53 of the sum of its terms' moduli, as FP64 multiply-adds give
# it: some 30 partial sums a thread and block, and what a chunk's conversions leave, 2^-59 of its largest
# operands' product a term, 12 units of its largest term's 2^-53 at the guard for 96 terms that all err one way.
@pytest.mark.parametrize("nx,ny,k", [(32, 32, 5), (320, 256, 9), (1024, 512, 4)])
@pytest.mark.parametrize("kind", BASES)
def test_dots_term_by_term(nx, ny, k, kind):
    prob = _problem(nx, ny)
    sv = _solver(prob, 1 if nx == 32 else 5, krylov_restart=20)
    V, w = _basis(kind, k, sv.n, np.random.default_rng(k))
    h = torch.empty(k, dtype=torch.complex128, device="cuda")
    sv.gs_dots(torch.as_tensor(V).to("cuda"), k, torch.as_tensor(w).to("cuda"), h)
    terms = V.conj().astype(np.clongdouble) * w
    assert (np.abs(h.cpu().numpy() - terms.sum(1)) <= 32 * 2.0 ** -53 * np.abs(terms).sum(1)).all()
    sv.close()



def test_partial_sums_are_added_exactly():
    """One product of 2^60, 1, -2^60 or 1 in each tile of 1024 points, a tile a block: the partial sums are
    exact, and so is their sum."""
    sv = _solver(_problem(320, 256), 5, krylov_restart=20)
    V = np.zeros((2, sv.n), complex)
    at = np.arange(0, sv.n, 1024)
    V[0, at] = np.resize([2.0 ** 60, 1.0, 1.0, -2.0 ** 60], at.size)
    V[1, at] = np.resize([1j, 2.0 ** 60, -2.0 ** 60, 3.0], at.size)
    w = np.ones(sv.n, complex)
    h = torch.empty(2, dtype=torch.complex128, device="cuda")
    sv.gs_dots(torch.as_tensor(V).to("cuda"), 2, torch.as_tensor(w).to("cuda"), h)
    assert at.size % 4 == 0
    assert h.tolist() == [at.size / 2, at.size / 4 * (3.0 - 1j)]
    sv.close()


# An entry of the update is good to the roundings of its own 2 k multiply-adds a part, as FP64 instructions
# give it, and as much again for k conversions at the guard.
@pytest.mark.parametrize("nx,ny,k", [(32, 32, 5), (320, 256, 9), (1024, 512, 4)])
@pytest.mark.parametrize("kind", BASES + ["coefficients"])
def test_update_entry_by_entry(nx, ny, k, kind):
    prob = _problem(nx, ny)
    sv = _solver(prob, 1 if nx == 32 else 5, krylov_restart=20)
    g = np.random.default_rng(k)
    V, w = _basis(kind, k, sv.n, g)
    c = g.standard_normal(k) + 1j * g.standard_normal(k)
    if kind == "coefficients":                       # the largest coefficient on a vector that is zero in places
        c *= np.exp2(-30.0 * np.arange(k))
        V[0, :sv.n // 2] = 0.0
        w[:sv.n // 2] *= 2.0 ** -60
    wd = torch.as_tensor(w).to("cuda")
    sv.gs_update(torch.as_tensor(V).to("cuda"), k, torch.as_tensor(c).to("cuda"), wd)
    terms = c[:, None].astype(np.clongdouble) * V
    size = np.abs(w) + np.abs(terms).sum(0)
    assert (np.abs(wd.cpu().numpy() - (w - terms.sum(0))) <= (8 * k + 16) * 2.0 ** -53 * size).all()
    sv.close()


def test_coarsest_solve_beside_a_spike():
    """At E = -2000 the coarsest operator (63 x 63, block reduction) couples a node to the next by 2^-9: 12
    nodes on, a spike of 2^60 adds less than 2^-48 of an entry, and FP64 sums leave the entries there as they
    are without it, to the 1e-13 of the solve."""
    sv = _solver(_problem(256, 256, E=-2000.0), 3)
    g = np.random.default_rng(23)
    f = g.standard_normal((63, 63)) + 1j * g.standard_normal((63, 63))
    spike = np.zeros((63, 63))
    spike[31, 20] = 2.0 ** 60
    j, i = np.indices((63, 63))
    far = abs(i - 20) + abs(j - 31) >= 12
    u = []
    for x in (f, f + spike):
        out = torch.empty(f.size, dtype=torch.complex128, device="cuda")
        sv.coarse_solve(torch.as_tensor(x.reshape(-1)).to("cuda"), out)
        u.append(out.cpu().numpy().reshape(63, 63))
    assert (np.abs(u[1] - u[0]) <= 1e-13 * np.abs(u[0]).max())[far].all()
    sv.close()


# Gauss-Jordan elimination over all rows leaves 4e-15 to 1.3e-14 here, and takes over from the block-wise
# inverse where that leaves more than 1e-14; the residual's own rounding adds less than half of it.
@pytest.mark.parametrize("n,levels,E,gamma", [(128, 3, 0.5, M.COARSE_GAMMA_DEFAULT), (512, 5, 0.8, M.COARSE_GAMMA_DEFAULT),
                                              (512, 5, 2.0, 0.0)])
def test_dense_inverse_residual(n, levels, E, gamma):
    sv = _solver(_problem(n, n, E=E), levels, coarse_gamma=gamma)
    m = sv.level_size(levels - 1)
    one, worst = torch.zeros(m, dtype=torch.complex128, device="cuda"), 0.0
    x, r = torch.empty_like(one), torch.empty_like(one)
    for k in range(m):
        one.zero_()
        one[k] = 1.0
        sv.coarse_solve(one, x)
        sv.level_residual(levels - 1, x, one, r)
        worst = max(worst, float(torch.view_as_real(r).abs().sum(-1).max()))
    assert worst <= 2e-14
    sv.close()
