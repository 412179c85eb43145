"""Where the complex128 passes on the integer pipes apply: which levels setup puts there, operators
whose updates do not fit 64 bits, and operands of very different size inside a tile."""
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


def _problem(nx, ny, E=0.5):
    return inputs.temkin_poet(nx, L=30.0, R0=20.0, theta=math.pi / 6, E=E, seed=3, ny=ny)


def _solver(prob, levels, spike=0.0, **kw):
    v12 = prob.v12.copy()
    v12[prob.ny // 3, prob.nx // 5] += spike
    return M.Solver(M.params_for(prob, levels=levels, **{"n_b": 0, **kw}), prob.v1, prob.v2, v12)


# 60000 nodes and more: 255 x 255, 511 x 511 with 255 x 255, 591 x 431 with 295 x 215; a coarsest level multiplies
# nothing itself; one large potential value spreads the fine diagonal
@pytest.mark.parametrize("nx,ny,levels,spike,on", [(240, 240, 4, 0.0, []), (256, 256, 4, 0.0, [0]),
                                                   (512, 512, 5, 0.0, [0, 1]), (592, 432, 5, 0.0, [0, 1]),
                                                   (592, 432, 5, 1e6, [1])])
def test_levels_on_the_integer_pipes(nx, ny, levels, spike, on):
    sv = _solver(_problem(nx, ny), levels, spike)
    assert sv.integer_passes() == (on, False)
    sv.close()
