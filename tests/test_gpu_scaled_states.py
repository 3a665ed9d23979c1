"""The FP64 step has no scale of its own on an unflagged flow: the same smooth
problem with all averages times a power of two, down to where their squares are
far below the smallest double, gives the same step times that power, for both
Riemann solvers, in the face kernel of 2D grids and the one-block 1D kernel."""
import numpy as np
import pytest

import oracle as O
import paper_2110_08683_gb300 as gp
from paper_2110_08683_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def problem(dim, riemann):
    if dim == 2:
        p = I.density_wave(nx=45, ny=38, amp=0.2, R=2, ell=0.1, kx=1, ky=2)
    else:
        p = I.sod_1d(n=128, R=2)
        x = (np.arange(128) + 0.5) / 128
        rho = 1.0 + 0.2 * np.sin(2.0 * np.pi * x)
        p["bc"] = ["periodic"] * 4
        p["U0"] = np.stack([rho, 0.7 * rho, 0.0 * rho, 2.5 + 0.245 * rho])[:, None, :]
    p["riemann"] = riemann
    return p


def step(p, U):
    g = gp.GPMood(p)
    g.set_state(U)
    g.step()
    out, bad = g.get_state(), g.flags()[1]
    g.close()
    return out, bad


@pytest.mark.parametrize("riemann", ["hllc", "hll"])
@pytest.mark.parametrize("dim", [1, 2])
def test_step_in_other_units(dim, riemann):
    p = problem(dim, riemann)
    ref, st, _, bad = O.Oracle(p).step(p["U0"], 0.0)
    assert not bad.any()
    for k in (0, -300, -505, -515, -530, -600, -900, 300, 505):
        U, bad = step(p, p["U0"] * 2.0**k)
        assert not bad.any(), k
        for v in range(4):
            assert np.abs(U[v] * 2.0**-k - ref[v]).max() <= 1e-12 * max(np.abs(ref[v]).max(), 1e-300), (k, v)


@pytest.mark.parametrize("riemann", ["hllc", "hll"])
@pytest.mark.parametrize("dim", [1, 2])
def test_first_order_where_squares_overflow(dim, riemann):
    """above 2^512 the squares of the momenta are infinite, positivity is not
    shown and every cell ends at first order, with a finite flux: the step of
    the first-order scheme, times the scale"""
    p = problem(dim, riemann)
    q = dict(p, cascade=[0])
    ref = O.Oracle(q).step(p["U0"], 0.0)[0]
    for k in (515, 700, 900):
        U, _ = step(p, p["U0"] * 2.0**k)
        for v in range(4):
            assert np.abs(U[v] * 2.0**-k - ref[v]).max() <= 1e-12 * max(np.abs(ref[v]).max(), 1e-300), (k, v)
