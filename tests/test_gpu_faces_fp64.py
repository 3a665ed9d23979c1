"""The FP64 face kernel (bands of 4 rows walked by a block, 31 faces a
segment, states in fixed point) against the oracle where its tiling and its
scaling can go wrong: grids of one cell more and fewer than a segment or a
band, several bands a block, and stencils whose values span many orders."""
import numpy as np
import pytest

import oracle as O
import paper_2110_08683_gb300 as gp
from paper_2110_08683_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def relerr(a, b):
    return max(np.abs(a[v] - b[v]).max() / max(np.abs(b[v]).max(), 1e-300) for v in range(4))


def step_both(p, U):
    g = gp.GPMood(p)
    g.set_state(U)
    g.step()
    Ug = g.get_state()
    og, bg, _ = g.flags()
    g.close()
    Uo, _, oo, bo = O.Oracle(p).step(U, 0.0)
    return Ug, Uo, og, oo, bg, bo


@pytest.mark.parametrize("R", [1, 2, 3])
@pytest.mark.parametrize("nx,ny", [(30, 3 + 1), (31, 5), (32, 6), (33, 7), (61, 8), (62, 9),
                                   (63, 11), (94, 67), (5, 131), (200, 4)])
def test_tile_edges(nx, ny, R):
    p = I.density_wave(nx=max(nx, R + 1), ny=max(ny, R + 1), amp=0.2, R=R, ell=0.1, kx=1, ky=1)
    Ug, Uo, og, oo, _, _ = step_both(p, p["U0"])
    assert relerr(Ug, Uo) <= 1e-12
    assert (og == oo).all()


@pytest.mark.parametrize("R", [1, 2, 3])
def test_large_contrast_and_zero_momentum(R):
    """a quiet gas with a zero momentum component and a hot dense spot 1e7
    times the pressure around it"""
    p = I.uniform(40, 37, R=R, state=(1.0, 0.3, 0.0, 1.0), bc="outflow", ell=0.3)
    p["cascade"] = list(range(R, -1, -1))
    U = p["U0"].copy()
    U[0, 17:20, 20:23] *= 50.0
    U[1, 17:20, 20:23] *= 50.0
    U[3, 17:20, 20:23] = 2.5e7
    Ug, Uo, og, oo, bg, bo = step_both(p, U)
    assert relerr(Ug, Uo) <= 1e-12
    assert (og == oo).all() and (bg == bo).all()


@pytest.mark.parametrize("spread", [1e-3, 1e-5, 1e-7, 1e-9])
def test_detection_near_the_csd_threshold(spread):
    """first-pass flags where the normalised pressure gradient straddles its
    threshold (5) by relative steps of `spread`: the FP64 path's float
    pre-test may only decide what FP64 decides the same"""
    nx, ny = 61, 40
    p = I.uniform(nx, ny, R=2, state=(1.0, 0.0, 0.0, 1.0), bc="outflow", ell=0.2)
    dx = 1.0 / nx
    # p[i+1] / p[i-1] = 1 + 2 dx s[i], s around 5 (pW is the smaller side)
    s = 5.0 * (1.0 + spread * (np.arange(nx) - nx // 2))
    pr = np.ones(nx)
    for i in range(1, nx - 1):
        pr[i + 1] = pr[i - 1] * (1.0 + 2.0 * dx * s[i])
    rho = 1.0 + 0.1 * np.random.default_rng(3).standard_normal((ny, nx))
    U = np.zeros((4, ny, nx))
    U[0] = rho
    U[3] = pr[None, :] / 0.4
    Ug, Uo, og, oo, bg, bo = step_both(p, U)
    assert 0 < bo[0].sum() < bo[0].size
    assert (bg[0] == bo[0]).all() and (og[0] == oo[0]).all()
