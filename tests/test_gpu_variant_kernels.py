"""Each 2-D variant's own kernels on grids beyond the small form's lines (in
FP32 4 864 warps of 8x4 cells, and 608 for variants 2-4 in both), where the variants
are not one kernel: the packed pairs (9-12) with even nx over 1 000 steps and with odd
nx over 200, every variant over 60, and the persistent step against the variant
whose tiles it runs.  Bars of
the parity tests: mixed T and Y 1e-5 relative L2, populations 1e-4 of their
maximum; FP64 1e-10; persistent against variant 2 1e-13 in FP64, 1e-6 mixed (the
same code in another kernel, contractions aside)."""
import os

import numpy as np
import pytest

from paper_2304_05657_gb300 import inputs

pytestmark = pytest.mark.gpu


def rel(a, b):
    return np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-300)


def channels(length):
    cfg, solid, T, Y, _ = inputs.batched_channels(widths=[16, 40, 64], length=length)
    return cfg, solid, T, Y


def oracle_state(oracle_mod, cfg, solid, T, Y, steps, g=None):
    oracle_mod.set_threads(os.cpu_count() or 1)
    try:
        o = oracle_mod.Sim(cfg, solid)
        o.set_state(T, Y, g) if g is not None else o.set_state(T, Y)
        o.step(steps)
        return o.get_state()
    finally:
        oracle_mod.set_threads(1)


def check_mixed(state, ref, fluid, name):
    assert rel(state[0][fluid], ref[0][fluid]) <= 1e-5, name
    for k in range(5):
        if np.linalg.norm(ref[1][k][fluid]) > 0:
            assert rel(state[1][k][fluid], ref[1][k][fluid]) <= 1e-5, (name, k)
    g, go = state[2][:, fluid], ref[2][:, fluid]
    assert np.abs(g - go).max() <= 1e-4 * np.abs(go).max(), name


@pytest.mark.parametrize("length,steps", [(1280, 1000), (1277, 200)])
def test_packed_pairs(lbfd_lib, oracle_mod, length, steps):
    cfg, solid, T, Y = channels(length)
    ref = oracle_state(oracle_mod, cfg, solid, T, Y, steps)
    s = lbfd_lib.Solver(dict(cfg, precision="mixed"), solid)
    for variant in (9, 10, 11, 12):
        s.variant = variant
        assert s.launches_per_step == 2
        s.set_state(T, Y)
        s.step_graph(steps)
        check_mixed(s.get_state(), ref, solid.ravel() == 0, variant)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_every_variant(lbfd_lib, oracle_mod, precision):
    cfg, solid, T, Y = channels(1280)
    g, T, Y = inputs.perturbed_state(cfg, solid, T, Y, seed=31)
    ref = oracle_state(oracle_mod, cfg, solid, T, Y, 60, g)
    s = lbfd_lib.Solver(dict(cfg, precision=precision), solid)
    seen = []
    for variant in range(2, s.num_variants):
        s.variant = variant
        s.set_state(T, Y, g)
        s.step(60)
        st = s.get_state()
        if precision == "fp64":
            for a, b in [(st[0], ref[0])] + list(zip(st[1], ref[1])) + list(zip(st[2], ref[2])):
                assert rel(a, b) <= 1e-10, variant
        else:
            check_mixed(st, ref, solid.ravel() == 0, variant)
        seen.append(s.launches_per_step)
    # coded cells in the tiles, or over their list (FP64: the small form)
    assert seen == [1, 1, 1] + [2 if precision == "mixed" else 1] * 8


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_persistent_matches_variant_2(lbfd_lib, precision):
    cfg, solid, T, Y = channels(192)
    g, T, Y = inputs.perturbed_state(cfg, solid, T, Y, seed=32)
    s = lbfd_lib.Solver(dict(cfg, precision=precision), solid)
    s.variant = 2
    s.set_state(T, Y, g)
    s.step(41)
    ref = s.get_state()
    s.set_state(T, Y, g)
    s.step_persistent(41)
    st = s.get_state()
    bar = 1e-13 if precision == "fp64" else 1e-6
    assert max(rel(a, b) for a, b in [(st[0], ref[0])] + list(zip(st[1], ref[1])) + list(zip(st[2], ref[2]))) <= bar
