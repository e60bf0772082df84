"""Which kernels a 2-D variant launches on either side of the small form's
lines (8 warps of 8x4 cells per SM partition in FP32, 32 in FP64; variants 2-4,
where their tiles take every cell, 1): with a convective outlet the small form is
one launch, the tiles and their list two; without, the autotuner times variants
that launch the same kernels once, so that they share a time.  On each grid every
kind of kernel against the general form: FP64 1e-10 relative L2 per field, mixed T
1e-5 and populations 1e-4 of their maximum, the bars of the parity tests."""
import numpy as np
import pytest

from test_gpu_small_grids import state

pytestmark = pytest.mark.gpu


def check(s, prec, case, variants):
    ref = None
    for variant in variants:
        s.variant = variant
        s.set_state(*case)
        s.step(2)
        Tg, Yg, gg = s.get_state()
        if ref is None:
            ref = Tg, Yg, gg
        elif prec == "fp64":
            for a, b in [(Tg, ref[0])] + list(zip(Yg, ref[1])) + list(zip(gg, ref[2])):
                assert np.linalg.norm(a - b) <= 1e-10 * max(np.linalg.norm(b), 1e-300), variant
        else:
            assert np.linalg.norm(Tg - ref[0]) <= 1e-5 * np.linalg.norm(ref[0]), variant
            assert np.abs(gg - ref[2]).max() <= 1e-4 * np.abs(ref[2]).max(), variant


# at each line and one tile column beyond it
@pytest.mark.parametrize("nx,ny", [(256, 76), (264, 76), (1024, 152), (1032, 152), (1024, 608), (1032, 608)])
def test_kernels_on_either_side_of_the_lines(lbfd_lib, nx, ny):
    cfg, solid, T, Y, g = state(nx, ny, "eq32", False, seed=nx)  # (no solid at the outlet)
    for prec in ("fp64", "mixed"):
        s = lbfd_lib.Solver(dict(cfg, precision=prec), solid)
        for variant in (1, 2, 6, 9):
            s.variant = variant
            small = (nx // 8) * (ny // 4) <= 608 * (32 if prec == "fp64" else 8)
            assert s.launches_per_step == (1 if small else 2), (prec, variant)
        check(s, prec, (T, Y, g), (0, 1, 2, 6, 9))


# the variants that are one kernel, and the others
@pytest.mark.parametrize("nx,ny,shared", [(256, 76, range(1, 13)), (264, 76, [1, *range(5, 13)]),
                                          (1024, 152, [1, *range(5, 13)]), (1032, 152, [])])
def test_autotune_times_each_kernel_once(lbfd_lib, nx, ny, shared):
    cfg, solid, T, Y, g = state(nx, ny, "flow", False, seed=1)  # (no cell that the coded tiles leave out)
    s = lbfd_lib.Solver(dict(cfg, precision="mixed"), solid)
    s.set_state(T, Y, g)
    best, ms = s.autotune(reps=3)
    assert np.all(ms > 0) and ms[best] == ms.min() and s.variant == best
    assert len({ms[v] for v in shared}) <= 1
    # the others are timed by themselves (events resolve 32 ns: some tie)
    others = [ms[v] for v in range(13) if v not in shared]
    assert len(others) == 1 or len(set(others)) > 1
    check(s, "mixed", (T, Y, g), (0, 1, 2, 3, 4, 6, 9))
