"""Derivatives of the step for small WENO3 epsilons (the weights hold eps^2 in
FP32), where the mixture is nearly uniform: the FP32 forms against the FP64
ones from the same state.

Mixed forward mode: the derivative fields of T and of the species after 4
steps, relative L2 <= 1e-3 of the FP64 tangent (for a species, of the largest
species' derivative).  FP32 rounding carried over 4 steps is about 1e-6; where
the differences of Y lie near FP32 resolution (noise of 1e-6 against 6e-8) the
weights' partials may be off by a few per cent, and they enter with u = 0.02 of
derivatives that live next to the walls and in the flame, where the field is
smooth or the convection centred.

FP32-forward adjoint through the tape (omega_hi != 1): the gradient within 2e-3
of the FP64 one per component, the bar of the gradient tests."""
import numpy as np
import pytest

from paper_2304_05657_gb300 import inputs, lbfd

pytestmark = pytest.mark.gpu


def nearly_uniform(eps):
    cfg, solid, T, Y = inputs.channel(nx=48, ny=16, walls="isothermal", T_wall=350.0, u_in=0.02, weno_eps=eps)
    rng = np.random.Generator(np.random.PCG64(4))
    Y = Y * (1.0 + 1e-6 * rng.standard_normal(Y.shape))
    return cfg, solid, T.astype(np.float32).astype(np.float64), Y.astype(np.float32).astype(np.float64)


@pytest.mark.parametrize("eps", [1e-6, 1e-10, 1e-12, 1e-14, 1e-16, 1e-18])
def test_mixed_tangent_matches_fp64_tangent(lbfd_lib, eps):
    cfg, solid, T, Y = nearly_uniform(eps)
    d = {}
    for prec in ("tangent", "tangent_mixed"):
        s = lbfd.Solver(dict(cfg, precision=prec), solid)
        s.set_state(T, Y)
        s.step(4)
        d[prec] = [[s.read_tangent(f, k) for f in [lbfd.FIELD_T] + [lbfd.FIELD_Y0 + j for j in range(5)]]
                   for k in range(4)]
        s.close()
    for k, (mixed, ref) in enumerate(zip(d["tangent_mixed"], d["tangent"])):
        scale = [np.linalg.norm(ref[0])] + [max(np.linalg.norm(r) for r in ref[1:])] * 5
        for j, (a, b) in enumerate(zip(mixed, ref)):
            assert np.isfinite(a).all(), (lbfd.THETA[k], j)
            assert np.linalg.norm(a - b) <= 1e-3 * scale[j], (lbfd.THETA[k], j, np.linalg.norm(a - b) / scale[j])


@pytest.mark.parametrize("eps", [1e-6, 1e-10, 1e-12, 1e-14, 1e-16, 1e-18, 1e-20])
def test_mixed_adjoint_tape_matches_fp64_adjoint(lbfd_lib, eps):
    cfg, solid, T, Y = nearly_uniform(eps)
    r = {}
    for prec in ("fp64", "mixed"):
        s = lbfd.Solver(dict(cfg, precision=prec, omega_hi=1.3), solid)
        s.set_state(T, Y)
        s.adjoint_setup(4)
        r[prec] = s.adjoint_run(9)[1]
        s.close()
    assert np.all(np.abs(r["mixed"] - r["fp64"]) <= 2e-3 * np.abs(r["fp64"])), r
