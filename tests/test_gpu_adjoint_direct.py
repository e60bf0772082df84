"""The hand-derived adjoint of the 2-D step against forward mode (the same
derivative by the chain rule per operation) on every face type and corner it
accepts, with solids next to faces, odd extents and both objectives; the
cases it leaves to the tape (convective outlet, cells with a link through
two open faces, omega_hi != 1) too.  Both are exact derivatives of the same
discrete step: they differ by rounding, a few thousand FP64 operations per
cell and step, so 1e-9 of the largest theta_k dJ/dtheta_k.  The FP32-forward
form differentiates the FP32 trajectory: within 2e-3 of the FP64 gradient,
the bar of the gradient tests."""
import numpy as np
import pytest

from paper_2304_05657_gb300 import grad, inputs, lbfd
from test_gpu_small_grids import FACES, state

pytestmark = pytest.mark.gpu


def gradients(cfg, solid, T, Y, g, steps, objective, every):
    out = {}
    for prec in ("fp64", "mixed", "tangent"):
        s = lbfd.Solver(dict(cfg, precision=prec), solid)
        s.set_state(T, Y, g)
        if prec == "tangent":
            s.step(steps)
            out[prec] = s.gradient(objective)
        else:
            s.adjoint_setup(every)
            out[prec] = s.adjoint_run(steps, objective)
        s.close()
    return out


def check(cfg, solid, T, Y, g, steps=9, every=4, objective=lbfd.OBJ_FLAME_POSITION):
    r = gradients(cfg, solid, T, Y, g, steps, objective, every)
    theta = grad.theta_of(cfg)
    (Ja, ga), (Jt, gt), (_, gm) = r["fp64"], r["tangent"], r["mixed"]
    scale = np.abs(gt * theta).max()
    assert abs(Ja - Jt) <= 1e-11 * abs(Jt)
    assert np.abs((ga - gt) * theta).max() <= 1e-9 * scale, (ga, gt)
    assert np.abs((gm - gt) * theta).max() <= 2e-3 * scale, (gm, gt)


@pytest.mark.parametrize("faces", sorted(FACES))
@pytest.mark.parametrize("solids", [False, True])
def test_faces_and_solids(lbfd_lib, faces, solids):
    check(*state(29, 21, faces, solids, seed=7, u_in=0.02))


@pytest.mark.parametrize("nx,ny", [(3, 3), (8, 4), (9, 5), (40, 1), (17, 30)])
def test_extents(lbfd_lib, nx, ny):
    check(*state(nx, ny, "flow", False, seed=nx + ny, u_in=0.02))


def test_poiseuille_quench_distance_and_periodic(lbfd_lib):
    check(*state(33, 18, "flow", True, seed=3, u_in=0.02, poiseuille_inlet=True), objective=lbfd.OBJ_QUENCH_DISTANCE)
    cfg, solid, T, Y, g = state(24, 20, "periodic", True, seed=4, u_in=0.02)
    check(cfg, solid, T, Y, g, objective=lbfd.OBJ_QUENCH_DISTANCE)


def test_tape_with_other_omega_hi(lbfd_lib):
    check(*state(25, 14, "flow", True, seed=9, u_in=0.02, omega_hi=1.2))
