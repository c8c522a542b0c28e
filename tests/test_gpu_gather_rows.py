"""The gather kernel by points and by rows of blocks (long rows of large
problems): a row of copies of a periodic problem, long enough for the second,
equals the single one bit for bit, and both match the oracle."""
import numpy as np
import pytest

from helpers import assert_parity, gpu_run, oracle_run
from paper_1211_2205_gb300 import capi
from test_gpu_parity import FP32_TOL, FP64_TOL, _random_problem

pytestmark = pytest.mark.gpu

# system, precision, N, cells of one copy, copies
KINDS = [("pn2d", "fp32", 3, (96, 160), 16), ("pn2d", "fp32", 13, (96, 32), 16), ("slab", "fp64", 31, (96, 1), 128),
         ("slab", "fp32", 63, (96, 1), 256)]


@pytest.mark.parametrize("system,precision,N,n,copies", KINDS)
def test_by_points_and_by_rows(system, precision, N, n, copies):
    out = []
    for rep in (1, copies):
        s = capi.Stepper(N=N, ax=(0.0, float(rep), 0.0, 1.0), n=(n[0] * rep, n[1]), precision=precision, system=system,
                         kernel="gather", schedule="merged")
        for j in range(s.ncomp):
            i = s.moment_info(j)
            X, Y = s.grid_coords(i["grid"])
            X, Y = X[:, :n[0]], Y[:, :n[0]]
            s.set_moment(j, np.tile(np.exp(np.cos(2 * np.pi * X + j) + np.sin(2 * np.pi * Y)), (1, rep)))
            if j % 3 == 0:
                s.set_source(j, np.tile(np.cos(2 * np.pi * X - j), (1, rep)))
        for g in range(4):
            X, Y = s.grid_coords(g)
            if X.size:
                v = np.tile(1.0 + 0.5 * np.sin(2 * np.pi * X[:, :n[0]]) * np.cos(2 * np.pi * Y[:, :n[0]]), (1, rep))
                s.set_material(g, 0.3 * v, v)
        s.step(5)
        out.append([s.moments(j) for j in range(s.ncomp)])
    for a, b in zip(*out):
        assert np.array_equal(np.tile(a, (1, copies)), b)


@pytest.mark.parametrize("bc", [("periodic", "extrapolation"), ("extrapolation", "periodic")])
def test_rows_match_the_oracle(bc):
    """1500 x 80 cells: a ragged last block per row, node and cell axes."""
    p = _random_problem(7, (1500, 80), bc, "fp32", 820, 3, aniso=True)
    s, got = gpu_run(p, kernel="gather", schedule="merged")
    o, ref = oracle_run(p, s)
    assert_parity(got, ref, FP32_TOL, "fp32")


def test_slab_rows_match_the_oracle():
    p = _random_problem(31, (12001, 1), ("extrapolation", "periodic"), "fp64", 821, 3, system="slab")
    s, got = gpu_run(p, schedule="literal")
    o, ref = oracle_run(p, s)
    assert_parity(got, ref, FP64_TOL, "fp64")
