"""FP64 passes of the 2D system: streamed by order on large grids, output by
output on small ones, both against the FP64 oracle (rel-L2 <= 1e-12, the FP64
bar) and against each other."""
import numpy as np
import pytest

from helpers import assert_parity, gpu_run, oracle_run
from paper_1211_2205_gb300 import capi, inputs
from test_gpu_parity import FP64_TOL, _random_problem

pytestmark = pytest.mark.gpu

BCS = [("periodic", "periodic"), ("extrapolation", "extrapolation"), ("periodic", "extrapolation"),
       ("extrapolation", "periodic")]


@pytest.mark.parametrize("bc", BCS)
@pytest.mark.parametrize("N", [1, 2, 3, 8])
def test_streamed(N, bc):
    """251 x 163 points: above the size from which a pass is streamed, ragged
    blocks, dx != dy; three steps carry the boundary copies back in."""
    p = _random_problem(N, (251, 163), bc, "fp64", 700 + N, 3, aniso=N == 3)
    s, got = gpu_run(p, schedule="merged")
    assert s.kernel == "gather"
    o, ref = oracle_run(p, s)
    assert_parity(got, ref, FP64_TOL, "fp64")


@pytest.mark.parametrize("n", [(1, 1), (2, 1), (1, 3), (5, 129)])
@pytest.mark.parametrize("bc", BCS)
@pytest.mark.parametrize("N", [1, 2, 5])
def test_output_by_output(N, bc, n):
    p = _random_problem(N, n, bc, "fp64", 740 + N, 4, aniso=N == 2)
    s, got = gpu_run(p, schedule="literal")
    o, ref = oracle_run(p, s)
    assert_parity(got, ref, FP64_TOL, "fp64")


@pytest.mark.parametrize("N", [4, 13])
def test_both_give_the_same_values(N):
    """The same operations in the same order: a periodic problem repeated
    four times in x (large enough to be streamed) equals the single one bit
    for bit.  (Dyadic domain: coordinates and spacings agree to the last bit.)"""
    def field(t, x, y):
        return 1.0 + 0.5 * np.sin(2 * np.pi * x) * np.cos(2 * np.pi * y)

    def pulse(t, x, y):
        return np.exp(np.cos(2 * np.pi * x) + np.sin(2 * np.pi * y))

    out = []
    for rep in (1, 4):
        s = capi.Stepper(N=N, ax=(0.0, float(rep), 0.0, 1.0), n=(96 * rep, 96), precision="fp64", schedule="merged")
        for g in range(4):
            X, Y = s.grid_coords(g)
            v = np.tile(field(0, X[:, :96], Y[:, :96]), (1, rep))
            s.set_material(g, 0.3 * v, v)
        X, Y = s.grid_coords(0)
        s.set_source(0, np.tile(pulse(0, X[:, :96], Y[:, :96]), (1, rep)))
        for j in (0, 1, 2):
            X, Y = s.grid_coords(s.moment_info(j)["grid"])
            s.set_moment(j, np.tile(pulse(0, X[:, :96], Y[:, :96]), (1, rep)))
        s.step(5)
        out.append([s.moments(j) for j in range(s.ncomp)])
    for a, b in zip(*out):
        assert np.array_equal(np.tile(a, (1, 4)), b)


@pytest.mark.parametrize("n", [(331, 333), (223, 251)])
@pytest.mark.parametrize("N", [1, 2, 3, 5, 7])
def test_around_the_sizes_of_the_rules(N, n):
    """331 x 333 points: wide output by output (N <= 2) or streamed with the
    passes overlapped; 223 x 251: output by output (N <= 2) or streamed pass
    after pass."""
    p = _random_problem(N, n, ("extrapolation", "periodic"), "fp64", 780 + N, 3)
    s, got = gpu_run(p, schedule="merged")
    o, ref = oracle_run(p, s)
    assert_parity(got, ref, FP64_TOL, "fp64")


@pytest.mark.parametrize("N", [1, 2, 3, 5])
def test_every_kernel_gives_the_same_values(N):
    """As test_both_give_the_same_values, at sizes on both sides of the low
    orders' rules: a row of sixteen copies equals the single one bit for bit."""
    out = []
    for rep in (1, 16):
        s = capi.Stepper(N=N, ax=(0.0, float(rep), 0.0, 1.0), n=(96 * rep, 96), precision="fp64", schedule="merged")
        for g in range(4):
            X, Y = s.grid_coords(g)
            v = np.tile(1.0 + 0.5 * np.sin(2 * np.pi * X[:, :96]) * np.cos(2 * np.pi * Y[:, :96]), (1, rep))
            s.set_material(g, 0.3 * v, v)
        for j in range(s.ncomp):
            X, Y = s.grid_coords(s.moment_info(j)["grid"])
            s.set_moment(j, np.tile(np.exp(np.cos(2 * np.pi * X[:, :96] + j) + np.sin(2 * np.pi * Y[:, :96])), (1, rep)))
        s.set_source(0, np.tile(np.cos(2 * np.pi * s.grid_coords(0)[0][:, :96]), (1, rep)))
        s.step(5)
        out.append([s.moments(j) for j in range(s.ncomp)])
    for a, b in zip(*out):
        assert np.array_equal(np.tile(a, (1, 16)), b)
