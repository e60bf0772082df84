"""A uniform mixture without reaction stays uniform, bit for bit, whatever its
temperature does: every line of Y_k, 1/W and Y_k W is constant, so that each
cell adds the same number to its Y_k (the stencils' rounding of a constant) and
nothing else.  At the largest diffusivities that the scheme accepts, where a
rounding of T in W would move Y by whole ulp a step.  All of a domain's cells
go through one kernel (periodic, no solids)."""
import numpy as np
import pytest

from paper_2304_05657_gb300 import inputs

pytestmark = pytest.mark.gpu

SMALL, LARGE, CUBE = (96, 80), (1280, 512), (48, 32, 24)


@pytest.mark.parametrize("extents,precision,variants", [
    (SMALL, "fp64", [0, 1]), (SMALL, "mixed", [0, 1]), (LARGE, "fp64", [1, 6]), (LARGE, "mixed", [1, 6, 9, 12]),
    (CUBE, "fp64", [0, 1, 4]), (CUBE, "mixed", [0, 1, 4])])
def test_species_stay_uniform(lbfd_lib, extents, precision, variants):
    dim = len(extents)
    cfg = inputs.base_config(dim=dim, bc=["periodic"] * 6, nu=0.1 if dim == 2 else 0.07, A=0.0, precision=precision,
                             **dict(zip(("nx", "ny", "nz"), extents)))
    solid = np.zeros(extents[::-1], np.uint8)
    N = solid.size
    rng = np.random.Generator(np.random.PCG64(3))
    T = 1100.0 + 800.0 * np.cos(2 * np.pi * (np.arange(N) % extents[0]) / extents[0]) + rng.uniform(-20, 20, N)
    Y = np.repeat(np.array(cfg["Y_in"])[:, None], N, 1)
    s = lbfd_lib.Solver(cfg, solid)
    for variant in variants:
        s.variant = variant
        s.set_state(T, Y)
        s.step(100)
        Tg, Yg, _ = s.get_state()
        assert np.isfinite(Tg).all() and np.ptp(Tg) > 100.0
        assert (np.ptp(Yg, axis=1) == 0.0).all(), (variant, np.ptp(Yg, axis=1))
