"""The one-launch form of 2-D steps on small grids (both lane splits) and the
coded boundary cells, in the tiles and over their list, against the FP64
oracle: every face type and corner, extents of one to a few cells and around
the 8x4 and 8x2 tiles, solids next to faces, and grids on both sides of the
rule's lines.  Tolerances are those of the parity tests: FP64 1e-10 relative
L2 per field after 20 steps (rounding order only), mixed T 1e-5 and
populations 1e-4 of their maximum."""
import numpy as np
import pytest

from paper_2304_05657_gb300 import inputs

pytestmark = pytest.mark.gpu

FACES = {
    "flow": ["inlet", "outlet_pressure", "wall_isothermal", "wall_adiabatic"],
    "eq32": ["inlet", "outlet", "wall_adiabatic", "wall_isothermal"],
    "cross": ["wall_isothermal", "wall_adiabatic", "inlet", "outlet_pressure"],
    "closed": ["wall_adiabatic", "wall_isothermal", "wall_isothermal", "wall_adiabatic"],
    "corner": ["inlet", "outlet", "outlet_pressure", "wall_isothermal"],
    "periodic": ["periodic", "periodic", "wall_isothermal", "outlet_pressure"],
}


def state(nx, ny, faces, solids, seed, **over):
    cfg = inputs.base_config(dim=2, nx=nx, ny=ny, bc=FACES[faces] + ["periodic", "periodic"], T_wall=[320.0] * 6,
                             T_solid=310.0, **over)
    rng = np.random.Generator(np.random.PCG64(seed))
    solid = (rng.random((ny, nx)) < 0.04).astype(np.uint8) if solids else np.zeros((ny, nx), np.uint8)
    T, Y = inputs.ignition_fields(cfg, solid, 0, min(6, nx), T_hot=900.0)
    g, T, Y = inputs.perturbed_state(cfg, solid, T, Y, seed=seed, T_amp=20.0)
    return cfg, solid, T, Y, g


def check(lbfd_lib, oracle_mod, cfg, solid, T, Y, g, steps, launches=None, variant=None):
    o = oracle_mod.Sim(cfg, solid)
    o.set_state(T, Y, g)
    o.step(steps)
    To, Yo, go = o.get_state()
    for prec in ("fp64", "mixed"):
        s = lbfd_lib.Solver(dict(cfg, precision=prec), solid)
        s.set_state(T, Y, g)
        if variant is not None:
            s.variant = variant
        if launches is not None:
            assert s.launches_per_step == launches
        s.step(steps)
        Tg, Yg, gg = s.get_state()
        if prec == "fp64":
            for a, b in [(Tg, To)] + list(zip(Yg, Yo)) + list(zip(gg, go)):
                assert np.linalg.norm(a - b) <= 1e-10 * max(np.linalg.norm(b), 1e-300)
        else:
            assert np.linalg.norm(Tg - To) <= 1e-5 * np.linalg.norm(To)
            assert np.abs(gg - go).max() <= 1e-4 * np.abs(go).max()


@pytest.mark.parametrize("faces", sorted(FACES))
@pytest.mark.parametrize("solids", [False, True])
def test_faces_and_corners(lbfd_lib, oracle_mod, faces, solids):
    check(lbfd_lib, oracle_mod, *state(37, 23, faces, solids, seed=5), steps=20)


@pytest.mark.parametrize("nx,ny", [(1, 1), (1, 9), (9, 1), (2, 3), (8, 2), (8, 4), (9, 5), (7, 31), (17, 8)])
def test_tile_edges(lbfd_lib, oracle_mod, nx, ny):
    check(lbfd_lib, oracle_mod, *state(nx, ny, "flow", False, seed=nx + 31 * ny), steps=20, launches=1)


def test_poiseuille_inlet_and_other_omega_hi(lbfd_lib, oracle_mod):
    check(lbfd_lib, oracle_mod, *state(40, 13, "flow", True, seed=2, poiseuille_inlet=True, omega_hi=1.3), steps=20)


# around the rule's lines: two lanes up to 304 warps of 32 cells, one launch
# up to 4 864 (FP32) and 19 456 (FP64) warps
@pytest.mark.parametrize("nx,ny", [(152, 64), (153, 64), (232, 60), (512, 304), (520, 304), (640, 487), (700, 500),
                                   (1216, 513)])
def test_rule_lines(lbfd_lib, oracle_mod, nx, ny):
    check(lbfd_lib, oracle_mod, *state(nx, ny, "flow", True, seed=nx), steps=2)


# an open corner keeps the grid off the one-launch form: the tiles of every
# shape with the coded cells in them (1-4) or over their list (5-12), ragged
# against each tile, the convective outlet's cells and the corner's apart
@pytest.mark.parametrize("variant", range(1, 13))
@pytest.mark.parametrize("isothermal", [0, 1])
def test_tile_variants_with_solids(lbfd_lib, oracle_mod, variant, isothermal):
    case = state(71, 37, "corner", True, seed=variant, solid_isothermal=isothermal)
    check(lbfd_lib, oracle_mod, *case, steps=20, launches=3, variant=variant)
