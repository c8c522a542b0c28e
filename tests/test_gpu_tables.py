"""Pass tables under changes of a live handle: a source or a set of decay
classes changes entries in place, allocating nothing but the source itself,
and the passes then see exactly what a handle set up that way at once sees."""
import numpy as np
import pytest

from paper_1211_2205_gb300 import capi
from test_gpu_parity import _random_problem

pytestmark = pytest.mark.gpu

# precision, kernel, schedule, system, cells: every kernel's tables (FP64 by output and streamed)
KINDS = [("fp64", "auto", "merged", "pn2d", (33, 21)), ("fp64", "auto", "literal", "pn2d", (251, 163)),
         ("fp64", "auto", "merged", "slab", (70, 1)), ("fp32", "gather", "merged", "pn2d", (33, 21)),
         ("fp32", "tiled_tall", "merged", "pn2d", (70, 33)), ("fp32", "tiled", "fused", "pn2d", (70, 33))]


def _make(kind):
    precision, kernel, schedule, system, n = kind
    p = _random_problem(6, n, ("periodic", "extrapolation") if system == "pn2d" else ("extrapolation", "periodic"),
                        precision, 640, 3, system=system)
    p.sources = []
    return capi.Stepper.from_problem(p, kernel=kernel, schedule=schedule)


def _source(s, j):
    X, Y = s.grid_coords(s.moment_info(j)["grid"])
    return np.cos(0.7 * j + 3 * X) * np.exp(-Y) / (1 + j % 7)


@pytest.mark.parametrize("kind", KINDS)
def test_a_source_costs_one_allocation(kind):
    s = _make(kind)
    for j in (0, 3, 5):
        q = _source(s, j)
        assert capi.debug_fail_allocation(2) == capi.OK     # the source is the first
        try:
            s.set_source(j, q)
        finally:
            capi.debug_fail_allocation(0)
    s.step(2)
    s.sync()


@pytest.mark.parametrize("kind", KINDS)
def test_changes_on_a_live_handle(kind):
    """Sources set, replaced and removed (the slots behind move up), decay
    classes per order and back, with steps in between."""
    f = [0.7 ** l for l in range(7)]
    a, b = _make(kind), _make(kind)
    start = a.get_state()
    for j in (0, 1, 2, 4, 5):
        a.set_source(j, 2.0 * _source(a, j))
    a.step(2)
    a.set_scattering_factors(f)
    a.step(1)
    a.set_source(1, None)
    a.set_source(4, None)
    a.set_source(6, _source(a, 6))
    for j in (0, 2, 5):
        a.set_source(j, _source(a, j))
    for factors in (f, None):
        a.set_scattering_factors(factors)
        b.set_scattering_factors(factors)
        for j in (0, 2, 5, 6):
            b.set_source(j, _source(b, j))
        a.set_state(start)
        b.set_state(start)
        a.step(3)
        b.step(3)
        assert a.get_state() == b.get_state()
