"""Where the one-block step of 1D FP64 problems ends: 512 cells are one launch,
513 are the kernels of the general step, both the oracle's step."""
import numpy as np
import pytest

import oracle as O
import paper_2110_08683_gb300 as gp
from paper_2110_08683_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx", [512, 513])
@pytest.mark.parametrize("R", [0, 1, 2, 3])
def test_each_side_of_the_limit(nx, R):
    p = I.sod_1d(n=nx, R=max(R, 1), ell_cells=6.0)
    p["cascade"] = list(range(R, -1, -1))
    U = p["U0"] * (1.0 + 0.05 * np.random.default_rng(nx + R).standard_normal((1, 1, nx)))
    g = gp.GPMood(p)
    g.set_state(U)
    g.step()
    assert (g.last_launches() == 1) == (nx == 512)
    Ug, (o, b, _) = g.get_state(), g.flags()
    g.close()
    Uo, _, oo, bo = O.Oracle(p).step(U, 0.0)
    assert np.abs(Ug - Uo).max() <= 1e-12 * np.abs(Uo).max()
    assert (o == oo).all() and (b == bo).all()
