"""The 3-D tiles with their coded cells against the FP64 oracle where they can
go wrong: extents of one to a few planes and ragged against the 32x4 and 16x8
columns, pieces whose last one is shorter, solids next to every face type, the
convective outlet's cells and the corners that the tiles leave out.
Tolerances are those of the parity tests: FP64 1e-10 relative L2 per field
after 10 steps (rounding order only), mixed T 1e-5 and populations 1e-4 of
their maximum."""
import numpy as np
import pytest

from paper_2304_05657_gb300 import inputs

pytestmark = pytest.mark.gpu

PERIODIC = ["periodic", "periodic"]
FACES = {
    "flow": ["inlet", "outlet_pressure"] + PERIODIC + PERIODIC,
    "eq32": PERIODIC + ["inlet", "outlet"] + PERIODIC,
    "along z": PERIODIC + PERIODIC + ["outlet_pressure", "inlet"],
    "walls": ["inlet", "outlet", "wall_isothermal", "wall_adiabatic"] + PERIODIC,
    "corner": ["inlet", "outlet_pressure", "inlet", "wall_isothermal", "wall_adiabatic", "outlet"],
}


@pytest.mark.parametrize("faces", sorted(FACES))
@pytest.mark.parametrize("nx,ny,nz", [(35, 9, 1), (33, 5, 2), (17, 7, 5), (40, 6, 11), (8, 18, 3)])
def test_columns_and_faces(lbfd_lib, oracle_mod, faces, nx, ny, nz):
    cfg = inputs.base_config(dim=3, nx=nx, ny=ny, nz=nz, bc=FACES[faces], T_wall=[320.0] * 6, T_solid=310.0,
                             solid_isothermal=nx % 2)
    rng = np.random.Generator(np.random.PCG64(nx + nz))
    solid = (rng.random((nz, ny, nx)) < 0.04).astype(np.uint8)
    T, Y = inputs.ignition_fields(cfg, solid, 0, 6, T_hot=900.0)
    g, T, Y = inputs.perturbed_state(cfg, solid, T, Y, seed=nx, T_amp=20.0)
    o = oracle_mod.Sim(cfg, solid)
    o.set_state(T, Y, g)
    o.step(10)
    To, Yo, go = o.get_state()
    for prec in ("fp64", "mixed"):
        for variant in (1, 4, 6):
            s = lbfd_lib.Solver(dict(cfg, precision=prec), solid)
            s.set_state(T, Y, g)
            s.variant = variant
            s.step(10)
            Tg, Yg, gg = s.get_state()
            if prec == "fp64":
                for a, b in [(Tg, To)] + list(zip(Yg, Yo)) + list(zip(gg, go)):
                    assert np.linalg.norm(a - b) <= 1e-10 * max(np.linalg.norm(b), 1e-300)
            else:
                assert np.linalg.norm(Tg - To) <= 1e-5 * np.linalg.norm(To)
                assert np.abs(gg - go).max() <= 1e-4 * np.abs(go).max()
