"""The block-reduction coarsest solve multiplies on the integer pipes; right-hand sides outside their
exponent range (huge, tiny) take FP64 instructions with the same factors.  The solve is linear, so
both give the same up to a power of two: each of the at most 8 levels rounds a sum of 3 m products,
about 100 units of 2^-53 with the reduction's growth, 1e-13 together."""
import math

import numpy as np
import pytest

from paper_1412_1953_gb300 import build, inputs
from paper_1412_1953_gb300 import mgcccs as M

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


@pytest.mark.parametrize("nx,ny", [(256, 256), (136, 272), (132, 256), (260, 132), (128, 512)])
def test_block_reduction_on_integers_equals_fp64(nx, ny):
    build.build()
    prob = inputs.temkin_poet(nx, L=30.0, R0=20.0, theta=math.pi / 6, E=0.5, seed=3, ny=ny)
    sv = M.Solver(M.params_for(prob, levels=3, n_b=0), prob.v1, prob.v2, prob.v12)
    g = np.random.default_rng(nx + ny)
    n = sv.level_size(2)
    f = torch.as_tensor(g.standard_normal(n) + 1j * g.standard_normal(n)).to("cuda")
    f[n // 2] = 0.0
    us = []
    for scale in (1.0, 2.0 ** 470, 2.0 ** -480):
        u = torch.empty_like(f)
        sv.coarse_solve(f * scale, u)
        us.append(u / scale)
    torch.cuda.synchronize()
    for u in us[1:]:
        assert float((u - us[0]).abs().max() / us[0].abs().max()) <= 1e-13
    bad = f.clone()
    bad[3] = complex(np.inf, 0.0)
    u = torch.empty_like(f)
    sv.coarse_solve(bad, u)
    torch.cuda.synchronize()
    assert not bool(torch.isfinite(torch.view_as_real(u)).all(-1).any())   # the inverse couples every node
    sv.close()
