"""Which kernels a 2-D variant launches on either side of the small form's
lines (one warp of 8x4 cells per SM partition for variants 2.., 3 in FP32 and 13
in FP64 for variant 1): the small form is one launch, the tiles of a grid with a
convective outlet are two (tile and list).  On each grid every kind of kernel
against the general form: FP64 1e-10 relative L2 per field, mixed T 1e-5 and
populations 1e-4 of their maximum, the bars of the parity tests.  And the
autotuner: variants that launch the same kernels share one time."""
import numpy as np
import pytest

from test_gpu_small_grids import state

pytestmark = pytest.mark.gpu


# (nx, ny): at a line and one tile column beyond; which of the variants 1 (FP32,
# FP64) and 2.. are the small form there
@pytest.mark.parametrize("nx,ny,small", [
    (256, 76, (True, True, True)), (264, 76, (True, True, False)),
    (384, 152, (True, True, False)), (392, 152, (False, True, False)),
    (832, 304, (False, True, False)), (840, 304, (False, False, False))])
def test_kernels_on_either_side_of_the_lines(lbfd_lib, nx, ny, small):
    cfg, solid, T, Y, g = state(nx, ny, "eq32", False, seed=nx)  # (no solid at the outlet)
    for prec in ("fp64", "mixed"):
        s = lbfd_lib.Solver(dict(cfg, precision=prec), solid)
        ref = None
        for variant in (0, 1, 2, 6, 9):
            s.variant = variant
            if variant:
                one = small[2] if variant > 1 else small[prec == "fp64"]
                assert s.launches_per_step == (1 if one else 2), (prec, variant)
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


def test_autotune_times_each_kernel_once(lbfd_lib):
    for nx, ny, shared in ((120, 40, range(1, 13)), (320, 100, [])):
        cfg, solid, T, Y, g = state(nx, ny, "eq32", False, seed=1)
        s = lbfd_lib.Solver(dict(cfg, precision="mixed"), solid)
        s.set_state(T, Y, g)
        best, ms = s.autotune(reps=3)
        assert np.all(ms > 0) and ms[best] == ms.min() and s.variant == best
        for v in shared:
            assert ms[v] == ms[1]
        assert shared or len(set(ms[1:])) > 1
