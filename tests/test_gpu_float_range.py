"""Detection on the FP64 path where single precision runs out: the same flow in
units that make densities, energies and cells very small or very large.  The
scheme has no scale of its own for positivity, so first-pass flags and final
radii have to be the oracle's (float pre-tests may only decide what FP64
decides the same)."""
import numpy as np
import pytest

import oracle as O
import paper_2110_08683_gb300 as gp
from paper_2110_08683_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def cold_stream(scale, size, sigma):
    """a cold supersonic stream with noise: some candidates of the first pass
    have a negative pressure"""
    nx, ny = 45, 38
    p = I.uniform(nx, ny, R=2, state=(1.0, 0.0, 0.0, 1.0), bc="periodic", ell=0.2)
    p["cascade"], p["sigma_v"], p["sigma_p"] = [2, 1, 0], sigma, sigma
    rng = np.random.default_rng(1)
    rho = 1.0 + 0.3 * rng.random((ny, nx))
    u = 1.0 + 0.05 * rng.standard_normal((ny, nx))
    v = -0.7 + 0.05 * rng.standard_normal((ny, nx))
    pr = 2e-3 * (1.0 + rng.random((ny, nx)))
    p["U0"] = scale * np.stack([rho, rho * u, rho * v, pr / 0.4 + 0.5 * rho * (u * u + v * v)])
    for k in ("x0", "x1", "y0", "y1", "ell"):
        p[k] *= size
    return p


@pytest.mark.parametrize("scale", [1.0, 1e-10, 1e-18, 1e-20, 1e-22, 1e-24, 1e-30, 1e-37, 1e-45,
                                   1e-100, 1e20, 1e30, 1e40])
@pytest.mark.parametrize("size,sigma", [(1.0, 1e6), (1.0, 5.0), (1e-14, 5.0), (1e-14, 1e19),
                                        (1e12, 1e-12), (1e25, 5.0)])
def test_flags_in_other_units(scale, size, sigma):
    p = cold_stream(scale, size, sigma)
    Uo, so, oo, bo = O.Oracle(p).step(p["U0"], 0.0)
    assert 0 < bo[0].sum() < bo[0].size and (oo < 2).any()
    g = gp.GPMood(p)
    g.set_state(p["U0"])
    g.step()
    og, bg, _ = g.flags()
    Ug = g.get_state()
    g.close()
    assert (bg[0] == bo[0]).all() and (og[0] == oo[0]).all()
    assert (bg == bo).all() and (og == oo).all()
    for v in range(4):
        assert np.abs(Ug[v] - Uo[v]).max() <= 1e-12 * np.abs(Uo[v]).max()
