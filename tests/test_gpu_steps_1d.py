"""Short 1D FP64 problems step in a one-block kernel (several steps a launch in
run()); the general step of many kernels is what an eager handle takes.  Both
over what the entry points accept: radii, boundaries, solvers, integrators,
Poly3, lengths around the warp and the kernel's limit."""
import numpy as np
import pytest

import oracle as O
import paper_2110_08683_gb300 as gp
from paper_2110_08683_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def tube(nx, R, bc="outflow", riemann="hllc", rk=3, recon="gp", seed=0):
    p = I.sod_1d(n=nx, R=max(R, 1), ell_cells=6.0)
    p["cascade"] = list(range(R, -1, -1))
    p["bc"] = [bc, bc, "outflow", "outflow"]
    if bc == "dirichlet":
        p["bc_prim"] = [[1.0, 0.0, 0.0, 1.0], [0.125, 0.0, 0.0, 0.1]] + [[1.0, 0.0, 0.0, 1.0]] * 2
    p["riemann"], p["rk"], p["recon"] = riemann, rk, recon
    rng = np.random.default_rng(seed)
    U = p["U0"] * (1.0 + 0.05 * rng.standard_normal((1, 1, nx)))
    p["U0"] = U
    return p


def both(p, steps, run_to=None):
    out = []
    for eager in (False, True):
        g = gp.GPMood(p, eager=eager)
        g.set_state(p["U0"])
        if run_to is None:
            for _ in range(steps):
                g.step()
        else:
            g.run(run_to)
        o, f, st = g.flags()
        out.append((g.get_state(), o, f, st, g.last_launches()))
        g.close()
    return out


@pytest.mark.parametrize("kw", [
    dict(nx=128, R=2), dict(nx=128, R=0), dict(nx=33, R=1), dict(nx=31, R=3), dict(nx=4, R=2),
    dict(nx=511, R=3), dict(nx=512, R=1), dict(nx=100, R=2, bc="periodic"),
    dict(nx=100, R=3, bc="reflect"), dict(nx=65, R=2, bc="dirichlet"),
    dict(nx=129, R=3, riemann="hll"), dict(nx=200, R=3, rk=4), dict(nx=90, R=1, recon="poly3"),
])
def test_one_block_steps_equal_the_general_steps(kw):
    (U1, o1, f1, s1, n1), (U0, o0, f0, s0, n0) = both(tube(**kw), 6)
    assert n1 == 1 and n0 > 1
    scale = np.abs(U0).max(axis=(1, 2), keepdims=True) + 1e-300
    assert (np.abs(U1 - U0) / scale).max() <= 1e-14
    assert np.array_equal(o1, o0) and np.array_equal(f1, f0)
    assert s1["iters"] == s0["iters"] and s1["nbad_total"] == s0["nbad_total"]
    assert s1["nsteps"] == s0["nsteps"] == 6


def test_run_takes_many_steps_a_launch():
    p = tube(128, 2)
    (U1, _, _, s1, _), (U0, _, _, s0, _) = both(p, 0, run_to=0.05)
    assert s1["nsteps"] == s0["nsteps"] > 10
    assert abs(s1["t"] - 0.05) <= 1e-15
    assert np.abs(U1 - U0).max() <= 1e-12


def test_above_the_limit_the_general_step_runs():
    for R in (0, 2):
        p = tube(1025, R)
        g = gp.GPMood(p)
        g.set_state(p["U0"])
        g.step()
        assert g.last_launches() > 1
        Uo = O.Oracle(p).step(p["U0"], 0.0)[0]
        assert np.abs(g.get_state() - Uo).max() <= 1e-12 * np.abs(Uo).max()
        g.close()


def test_errors_stop_a_run_where_the_general_step_stops():
    p = tube(64, 2)
    U = p["U0"].copy()
    U[0, 0, 10] = -1.0  # no admissible time step
    for eager in (False, True):
        g = gp.GPMood(p, eager=eager)
        g.set_state(U)
        with pytest.raises(gp.GpmoodError) as e:
            g.run(0.1)
        assert e.value.code == -6
        assert g.flags(maps=False)[2]["nsteps"] == 0
        assert np.array_equal(g.get_state(), U)
        g.close()
