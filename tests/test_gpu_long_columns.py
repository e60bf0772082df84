"""3-D grids so long in z that a launch of the tile kernels holds no more pieces
of the column than a grid's third extent allows (65 535): every fused variant
against the general form, FP64, 1e-12 relative L2 per field after one step
(the same arithmetic, other contractions)."""
import numpy as np
import pytest

from paper_2304_05657_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nz", [262143, 786432, 1048560])
def test_long_columns(lbfd_lib, nz):
    cfg = inputs.base_config(dim=3, nx=1, ny=1, nz=nz, bc=["periodic"] * 6)
    solid = np.zeros((nz, 1, 1), np.uint8)
    rng = np.random.Generator(np.random.PCG64(nz))
    T = 300.0 + 700.0 * rng.random(nz)
    Y = np.array(cfg["Y_in"])[:, None] + 0.01 * rng.random((5, nz))
    Y /= Y.sum(0)
    g = rng.uniform(-1e-3, 1e-3, (27, nz))
    ref = None
    for variant in (0, 1, 2, 3, 6, 7):
        s = lbfd_lib.Solver(cfg, solid)
        s.set_state(T, Y, g)
        s.variant = variant
        s.step(1)
        out = s.get_state()
        s.close()
        if ref is None:
            ref = out
            continue
        for a, b in zip(out, ref):
            assert np.linalg.norm(a - b) <= 1e-12 * np.linalg.norm(b), variant
