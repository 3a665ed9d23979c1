"""The FP64 face kernel at the edges of its tiles (segments of 31 faces, bands of
4 rows) for every radius and both Riemann solvers: against the oracle, against
itself one direction a launch, and on mirrored and transposed problems."""
import numpy as np
import pytest

import oracle as O
import paper_2110_08683_gb300 as gp
from paper_2110_08683_gb300 import inputs as I

pytestmark = pytest.mark.gpu

SIZES = [(30, 4), (31, 5), (32, 7), (33, 8), (62, 9), (63, 11), (5, 35), (94, 31)]


def problem(nx, ny, R, riemann, bc="outflow", seed=0):
    """smooth waves with noise of a few per cent, momenta of either sign; the length
    scale is at most 6 cells either way (at 40 and more the two binary128 weight
    solves themselves differ by 1e-12)"""
    p = I.uniform(nx, ny, R=max(R, 1), state=(1.0, 0.2, -0.1, 1.0), bc=bc, ell=6.0 / max(nx, ny))
    p["cascade"], p["riemann"] = list(range(R, -1, -1)), riemann
    rng = np.random.default_rng(seed + nx)
    x, y = (np.arange(nx) + 0.5) / nx, (np.arange(ny)[:, None] + 0.5) / ny
    rho = 1.0 + 0.2 * np.sin(2 * np.pi * (x + y)) + 0.02 * rng.standard_normal((ny, nx))
    u = 0.3 * np.sin(2 * np.pi * x) + 0.0 * y
    v = -0.2 * np.cos(2 * np.pi * y) + 0.05 * rng.standard_normal((ny, nx))
    pr = 1.0 + 0.1 * np.cos(2 * np.pi * (x - y))
    p["U0"] = np.stack([rho, rho * u, rho * v, pr / 0.4 + 0.5 * rho * (u * u + v * v)])
    return p


def run(p, U, steps=1):
    g = gp.GPMood(p)
    g.set_state(U)
    for _ in range(steps):
        g.step()
    out, (o, b, _) = g.get_state(), g.flags()
    g.close()
    return out, o, b


@pytest.mark.parametrize("riemann", ["hllc", "hll"])
@pytest.mark.parametrize("R", [0, 1, 2, 3])
@pytest.mark.parametrize("nx,ny", SIZES)
def test_against_the_oracle_and_split(nx, ny, R, riemann):
    p = problem(nx, max(ny, R + 1), R, riemann)
    U, o, b = run(p, p["U0"])
    Uo, _, oo, bo = O.Oracle(p).step(p["U0"], 0.0)
    for v in range(4):
        assert np.abs(U[v] - Uo[v]).max() <= 1e-12 * np.abs(Uo[v]).max()
    assert (o == oo).all() and (b == bo).all()
    Us, os_, bs = run(dict(p, split_faces=1), p["U0"])
    assert np.array_equal(U, Us) and np.array_equal(o, os_) and np.array_equal(b, bs)


@pytest.mark.parametrize("riemann", ["hllc", "hll"])
@pytest.mark.parametrize("R", [1, 2, 3])
@pytest.mark.parametrize("bc", ["outflow", "reflect", "periodic"])
def test_mirror_images(R, bc, riemann):
    """face states, HLL and the update are odd and even bit for bit; the contact
    speed of HLLC adds its two sides in order, a rounding each of 18 stages"""
    p = problem(61, 35, R, riemann, bc)
    U, o, _ = run(p, p["U0"], steps=6)
    for axis, mom in ((2, 1), (1, 2)):
        W = np.flip(p["U0"], axis).copy()
        W[mom] = -W[mom]
        V, om, _ = run(p, np.ascontiguousarray(W), steps=6)
        V = np.flip(V, axis).copy()
        V[mom] = -V[mom]
        if riemann == "hll":
            assert np.array_equal(V, U) and np.array_equal(np.flip(om, axis), o), axis
        else:
            assert np.abs(V - U).max() <= 18 * 16 * 2.0**-53 * np.abs(U).max(), axis


@pytest.mark.parametrize("riemann", ["hllc", "hll"])
@pytest.mark.parametrize("R", [1, 2, 3])
def test_transposed_problem(R, riemann):
    """sums over x and y terms change places: a rounding each, 2^-53 of the sums"""
    p = problem(45, 45, R, riemann)
    U, o, _ = run(p, p["U0"])
    W = np.ascontiguousarray(np.transpose(p["U0"], (0, 2, 1))[[0, 2, 1, 3]])
    V, om, _ = run(p, W)
    V = np.transpose(V, (0, 2, 1))[[0, 2, 1, 3]]
    for v in range(4):
        assert np.abs(V[v] - U[v]).max() <= 2e-14 * max(np.abs(U).max(), 1.0)
    assert np.array_equal(np.transpose(om, (0, 2, 1)), o)
