"""A batch of the smallest grids, whose channel systems have at most one row per CTA and so no factors
to fetch: each member equals its own solve to the rounding of the channel solve's two forms."""
import math

import pytest

from paper_1412_1953_gb300 import build, inputs
from paper_1412_1953_gb300 import mgcccs as M

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


@pytest.mark.parametrize("n", [16, 32])
def test_smallest_batch(n):
    build.build()
    L = 30.0 * n / 512
    probs = [inputs.temkin_poet(n, L=L, R0=2 * L / 3, theta=math.pi / 6, E=E, seed=3) for E in (0.5, 1.1)]
    svs = [M.Solver(M.params_for(p, levels=2, n_b=2, krylov_restart=20), p.v1, p.v2, p.v12, stream=torch.cuda.Stream())
           for p in probs]
    fs = [torch.as_tensor(p.f).to("cuda") for p in probs]
    us = [torch.zeros_like(f) for f in fs]
    torch.cuda.synchronize()
    M.Batch(svs, us, fs).run(rtol=1e-10, max_iter=400)
    for sv, f, u in zip(svs, fs, us):
        v = torch.zeros_like(f)
        sv.solve(v, f, rtol=1e-10, max_iter=400)
        torch.cuda.synchronize()
        assert float((u - v).abs().max() / v.abs().max()) <= 1e-8
