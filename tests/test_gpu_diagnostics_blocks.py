"""The diagnostics reduction (block sums joined in block order, the centre line
by a block of its own) against the oracle's where its blocks change: one block,
a cell more, every block one round (608 of 256 cells) and a row more, bands of
rows, and 3-D.  FP64 sums of N terms in another order: 1e-12 relative; counts,
extrema and the centre line's position exact; a second call bit for bit."""
import numpy as np
import pytest

from paper_2304_05657_gb300 import inputs

pytestmark = pytest.mark.gpu

SUMS = ("x_f", "mass", "heat_release", "fuel_consumption")


@pytest.mark.parametrize("extents", [(256, 1), (257, 1), (37, 5), (608, 256), (608, 257), (1100, 190), (64, 50, 40)])
def test_blocks_against_the_oracle(lbfd_lib, oracle_mod, extents):
    dim = len(extents)
    cfg = inputs.base_config(dim=dim, bc=["inlet", "outlet_pressure"] + ["periodic"] * 4,
                             **dict(zip(("nx", "ny", "nz"), extents)))
    rng = np.random.Generator(np.random.PCG64(extents[0]))
    solid = (rng.random(extents[::-1]) < 0.03).astype(np.uint8)
    T, Y = inputs.ignition_fields(cfg, solid, 0, min(20, extents[0]), burnt=False)
    g, T, Y = inputs.perturbed_state(cfg, solid, T, Y, seed=extents[0])
    s = lbfd_lib.Solver(cfg, solid)
    s.set_state(T, Y, g)
    o = oracle_mod.Sim(cfg, solid)
    o.set_state(T, Y, g)
    d, ref = s.diagnostics(), o.diagnostics()
    for k in SUMS:
        assert abs(d[k] - ref[k]) <= 1e-12 * abs(ref[k]), k
    for k in ("T_max", "x_hrr_max", "n_nonfinite", "n_fluid"):
        assert d[k] == ref[k], k
    assert s.diagnostics() == d
    if dim == 2 and extents[1] > 4:  # bands of rows add up
        m = extents[1] // 3
        a, b = s.diagnostics((0, m)), s.diagnostics((m, extents[1]))
        assert a["n_fluid"] + b["n_fluid"] == d["n_fluid"]
        for k in ("mass", "heat_release", "fuel_consumption"):
            assert abs(a[k] + b[k] - d[k]) <= 1e-12 * abs(d[k]), k
