"""What a cell's cotangent reaches through the FP64 gather, cell by cell: a NaN or
an infinity goes where a finite one goes and nowhere else, and small gradients
keep their accuracy next to cells whose large ones do not reach them (faces
below the top radius) and at the rim of what a localised cotangent reaches."""
import numpy as np
import pytest

import paper_2110_08683_gb300 as gp
from paper_2110_08683_gb300 import inputs as I

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

NX, NY = 40, 36


def problem(R):
    p = I.density_wave(nx=NX, ny=NY, amp=0.2, R=R, ell=0.2)
    p["bc"] = ["outflow"] * 4
    return p


def radii(R, kind, seed=0):
    if kind == "mixed":
        return np.random.default_rng(seed).integers(0, R + 1, (3, NY, NX))
    return np.full((3, NY, NX), min(kind, R))


def stages(p, ords, dt):
    from oracle.frozen_torch import FrozenStep

    fs, U = FrozenStep(p), torch.tensor(p["U0"])
    with torch.no_grad():
        Y1 = U - dt * fs.residual(U, ords[0])
        X3 = 0.25 * (3.0 * U + Y1 - dt * fs.residual(Y1, ords[1]))
    return fs, torch.stack([U, Y1, X3]).numpy()


def vjp(p, tape, ords, lam, dt):
    t = torch.tensor(tape, device="cuda")
    o = torch.tensor(ords, dtype=torch.uint8, device="cuda").contiguous()
    l = torch.tensor(lam, device="cuda")
    out = torch.empty_like(l)
    g = gp.GPMood(p)
    g.set_state(p["U0"])
    g.step_adjoint(t.data_ptr(), o.data_ptr(), dt, 0.0, l.data_ptr(), out.data_ptr())
    got = out.cpu().numpy()
    g.close()
    return got


@pytest.mark.parametrize("R", [1, 2, 3])
@pytest.mark.parametrize("kind", [0, 1, 3, "mixed"])
def test_non_finite_cotangents_stay_in_reach(R, kind):
    p, ords = problem(R), radii(R, kind)
    _, tape = stages(p, ords, 1e-3)
    lam = np.zeros_like(p["U0"])
    lam[:, 18, 20] = 1.0
    reach = (vjp(p, tape, ords, lam, 1e-3) != 0.0).any(axis=0)
    assert 13 <= reach.sum() < reach.size
    for bad in (np.nan, np.inf, -np.inf):
        lam[:, 18, 20] = bad
        out = vjp(p, tape, ords, lam, 1e-3)
        assert np.array_equal(~np.isfinite(out).all(axis=0), reach)


@pytest.mark.parametrize("R", [1, 2, 3])
@pytest.mark.parametrize("kind", [0, 1, 3, "mixed"])
def test_small_gradients_next_to_large_ones(R, kind):
    """a cotangent of one in one cell among ones of 1e-12: every cell that the
    large one does not reach has the gradient it has without it, bit for bit up
    to the rounding of its own sums"""
    p, ords = problem(R), radii(R, kind, seed=1)
    _, tape = stages(p, ords, 1e-3)
    rng = np.random.default_rng(2)
    lam = 1e-12 * (1.0 + rng.random(p["U0"].shape))
    big = np.zeros_like(lam)
    big[:, 18, 20] = 1.0
    reach = (vjp(p, tape, ords, big, 1e-3) != 0.0).any(axis=0)
    alone = vjp(p, tape, ords, lam, 1e-3)
    beside = vjp(p, tape, ords, lam + big, 1e-3)
    # a cell's own sums: tens of products of size 1e-12 / 36, dt / dx = 0.04 of
    # them against the identity part: a few 2^-53 of 1e-12
    assert np.abs(beside - alone)[:, ~reach].max() <= 8 * 2.0**-53 * 2e-12


@pytest.mark.parametrize("R", [1, 2, 3])
def test_rim_of_a_localised_cotangent(R):
    """relative to the size of each cell's own gradient (the largest of its four
    values), against autograd of the CPU restatement"""
    p, ords = problem(R), radii(R, 3)
    dt = 1e-3
    fs, tape = stages(p, ords, dt)
    lam = np.zeros_like(p["U0"])
    lam[:, 18, 20] = [1.0, -0.5, 0.7, 0.2]
    got = vjp(p, tape, ords, lam, dt)
    U = torch.tensor(p["U0"], requires_grad=True)
    (ref,) = torch.autograd.grad((fs.step(U, ords, dt) * torch.tensor(lam)).sum(), U)
    ref = ref.numpy()
    size = np.abs(ref).max(axis=0)
    on = size > 0.0
    assert np.array_equal(on, (got != 0.0).any(axis=0))
    # the reference rounds like a chain of FP64 sums whose terms cancel at the rim
    rel = (np.abs(got - ref).max(axis=0)[on] / size[on])
    assert np.median(rel) <= 1e-13 and rel.max() <= 1e-8
