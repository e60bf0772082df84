"""Which kernels a 2-D variant launches on either side of the small form's
lines (in warps of 8x4 cells per SM partition: FP32 variant 1 3, variants 2-4 1,
others 8; FP64 variants 2-4 1, others 13): the small form is one launch, the tiles
of a grid with a convective outlet are two (tile and list).  On each grid every kind of kernel
against the general form: FP64 1e-10 relative L2 per field, mixed T 1e-5 and
populations 1e-4 of their maximum, the bars of the parity tests.  And the
autotuner: variants that launch the same kernels share one time."""
import numpy as np
import pytest

from test_gpu_small_grids import state

pytestmark = pytest.mark.gpu


LINES = {"fp64": {1: 13, 2: 1, 6: 13, 9: 13}, "mixed": {1: 3, 2: 1, 6: 8, 9: 8}}


# at each line and one tile column beyond it
@pytest.mark.parametrize("nx,ny", [(256, 76), (264, 76), (384, 152), (392, 152), (1024, 152), (1032, 152), (832, 304),
                                   (840, 304)])
def test_kernels_on_either_side_of_the_lines(lbfd_lib, nx, ny):
    cfg, solid, T, Y, g = state(nx, ny, "eq32", False, seed=nx)  # (no solid at the outlet)
    for prec in ("fp64", "mixed"):
        s = lbfd_lib.Solver(dict(cfg, precision=prec), solid)
        ref = None
        for variant in (0, 1, 2, 6, 9):
            s.variant = variant
            if variant:
                small = (nx // 8) * (ny // 4) <= 608 * LINES[prec][variant]
                assert s.launches_per_step == (1 if small else 2), (prec, variant)
            s.set_state(T, Y, g)
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


@pytest.mark.parametrize("nx,ny,shared", [(120, 40, range(1, 13)), (320, 100, [1, *range(5, 13)]),
                                          (800, 100, range(5, 13)), (1100, 160, [])])
def test_autotune_times_each_kernel_once(lbfd_lib, nx, ny, shared):
    cfg, solid, T, Y, g = state(nx, ny, "eq32", False, seed=1)
    s = lbfd_lib.Solver(dict(cfg, precision="mixed"), solid)
    s.set_state(T, Y, g)
    best, ms = s.autotune(reps=3)
    assert np.all(ms > 0) and ms[best] == ms.min() and s.variant == best
    assert len({ms[v] for v in shared}) <= 1
    assert len(set(ms)) >= 13 - len(shared)  # (the others apart, but for a chance tie)
