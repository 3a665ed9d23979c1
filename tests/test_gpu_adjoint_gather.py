"""The FP64 gather of the adjoint (tiles of 32 x 8 cells, fixed point with one
exponent a cell) against autograd of the CPU restatement: grids around the
tile, every radius, radius maps with lowered cells, cotangents of very
different sizes side by side."""
import numpy as np
import pytest

import paper_2110_08683_gb300 as gp
from paper_2110_08683_gb300 import inputs as I

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("lowered", [False, True])
@pytest.mark.parametrize("nx,ny,R,bc", [(24, 5, 1, "periodic"), (31, 9, 2, "outflow"),
                                        (33, 8, 3, "periodic"), (26, 17, 3, "dirichlet"),
                                        (60, 7, 2, "periodic")])
def test_vjp_with_given_radii(nx, ny, R, bc, lowered):
    from oracle.frozen_torch import FrozenStep

    p = I.density_wave(nx=nx, ny=ny, amp=0.2, R=R, ell=0.2)
    p["bc"], p["bc_prim"] = [bc] * 4, [[1.1, 0.9, 1.05, 1.0]] * 4
    rng = np.random.default_rng(nx + ny)
    ords = np.full((3, ny, nx), R)
    if lowered:
        ords = np.where(rng.random(ords.shape) < 0.2, rng.integers(0, R + 1, ords.shape), R)
    dt = 0.1 / max(nx, ny)
    fs = FrozenStep(p)
    U = torch.tensor(p["U0"], requires_grad=True)
    # the stage inputs of the step with these radii
    with torch.no_grad():
        Y1 = U - dt * fs.residual(U, ords[0])
        X3 = 0.25 * (3.0 * U + Y1 - dt * fs.residual(Y1, ords[1]))
        tape = torch.stack([U, Y1, X3]).cuda().contiguous()
    otape = torch.tensor(ords, dtype=torch.uint8).cuda().contiguous()
    # cotangents over eight orders of magnitude
    lam = rng.standard_normal(p["U0"].shape) * 10.0 ** rng.uniform(-8, 0, (1, ny, nx))
    lam_d = torch.as_tensor(lam, device="cuda").contiguous()
    out = torch.empty_like(lam_d)
    g = gp.GPMood(p)
    g.set_state(p["U0"])
    g.step_adjoint(tape.data_ptr(), otape.data_ptr(), dt, 0.0, lam_d.data_ptr(), out.data_ptr())
    got = out.cpu().numpy()
    g.close()
    (ref,) = torch.autograd.grad((fs.step(U, ords, dt) * torch.tensor(lam)).sum(), U)
    ref = ref.numpy()
    assert np.abs(got - ref).max() <= 1e-12 * np.abs(ref).max()
