"""The tile shapes of the FP32 kernel give the same values bit for bit: each
point sees the same arithmetic in the same order whatever the tile height, the
rows per warp and the CTAs per SM (the 5-row tiles are held to the oracle in
test_gpu_tiled.py and test_gpu_edge.py)."""
import numpy as np
import pytest

from paper_1211_2205_gb300 import capi
from test_gpu_parity import _random_problem

pytestmark = pytest.mark.gpu

BCS = [("periodic", "periodic"), ("extrapolation", "extrapolation"), ("periodic", "extrapolation"),
       ("extrapolation", "periodic")]


def _state(p, kernel):
    s = capi.Stepper.from_problem(p, kernel=kernel, schedule="merged")
    s.step(p.nsteps)
    return s.get_state()


@pytest.mark.parametrize("bc", BCS)
@pytest.mark.parametrize("N", [1, 2, 5, 15])
def test_five_row_bands(N, bc):
    """641 x 163 cells: 187 tiles of 64 x 10 (more than a GPU has SMs, so the
    five-row bands), one column in the last tile column, three rows in the
    last tile row (the second band empty), an odd width; four steps carry the
    boundary copies back in."""
    p = _random_problem(N, (641, 163), bc, "fp32", 900 + N, 4)
    assert _state(p, "tiled_tall") == _state(p, "tiled_short")


@pytest.mark.parametrize("n", [(64, 10), (65, 11), (63, 9), (2, 30), (3, 5), (130, 47)])
@pytest.mark.parametrize("bc", BCS)
def test_two_row_bands(n, bc):
    """Grids of at most a tile per SM (two-row bands) around the tile's edges."""
    p = _random_problem(6, n, bc, "fp32", 950, 4)
    assert _state(p, "tiled_tall") == _state(p, "tiled_short")


@pytest.mark.parametrize("N", [16, 49, 50, 55])
def test_orders_around_the_table_limits(N):
    """16: two-row bands whatever the grid; 49 / 50: weights kept twice /
    once; 55: the highest order of the 10-row tiles."""
    p = _random_problem(N, (70, 23), ("periodic", "extrapolation"), "fp32", 970, 2)
    assert _state(p, "tiled_tall") == _state(p, "tiled_short")


@pytest.mark.parametrize("bc", BCS)
def test_boundary_copies(bc):
    """After a step every boundary copy, corners included, holds the value it
    copies (periodic: -1 <- n - 1, n <- 0; extrapolation: -1 <- 0, n <- n - 1;
    none on an extrapolation axis of nodes)."""
    import torch
    p = _random_problem(3, (75, 12), bc, "fp32", 980, 1)
    s = capi.Stepper.from_problem(p, kernel="tiled_tall", schedule="merged")
    s.step(1)
    s.sync()

    class View:
        pass

    for j in range(s.ncomp):
        i = s.moment_info(j)
        ptr, pitch, off = s.device_ptr(j)
        v = View()
        v.__cuda_array_interface__ = dict(shape=(i["ny"] + 2, i["nx"] + 2), strides=(pitch * 4, 4), typestr="<f4",
                                          data=(ptr + 4 * (off - pitch - 1), False), version=3)
        a = torch.as_tensor(v, device="cuda").cpu().numpy()
        u = a[1:-1, 1:-1]
        node = (i["grid"] & 1, i["grid"] >> 1)
        copies = [bc[d] == "periodic" or not node[d] for d in range(2)]
        pad = u
        for d, axis in ((0, 1), (1, 0)):
            if copies[d]:
                width = [(0, 0), (0, 0)]
                width[axis] = (1, 1)
                pad = np.pad(pad, width, mode="wrap" if bc[d] == "periodic" else "edge")
        lo = [0 if c else 1 for c in copies]
        got = a[lo[1]:a.shape[0] - lo[1], lo[0]:a.shape[1] - lo[0]]
        assert np.array_equal(got, pad), (j, i)


def test_runs_repeat_bit_for_bit():
    """Nine tiles per block, a state far beyond L2: every run from the same
    initial values ends in the same bits (a ring slot refilled before its last
    value is read shows as a few wrong points in some runs)."""
    p = _random_problem(9, (1501, 1099), ("extrapolation", "periodic"), "fp32", 995, 1)
    s = capi.Stepper.from_problem(p, kernel="tiled_tall", schedule="literal")
    start, ref = s.get_state(), None
    for _ in range(24):
        s.set_state(start)
        s.step(6)
        got = s.get_state()
        assert ref is None or got == ref
        ref = got


def test_sources_in_every_moment():
    """A source in every moment and a decay class per order, on a state that
    L2 does not hold beside its sources (the kernels that load them into L1
    ahead): 10-row and 5-row tiles bit for bit, and the gather kernel at the
    FP32 parity bar."""
    from helpers import assert_parity
    from test_gpu_parity import FP32_TOL
    N, n = 35, (161, 137)
    p = _random_problem(N, n, ("periodic", "extrapolation"), "fp32", 990, 2, aniso=True)
    got = []
    for kernel in ("tiled_tall", "tiled_short", "gather"):
        s = capi.Stepper.from_problem(p, kernel=kernel, schedule="merged")
        for j in range(s.ncomp):
            X, Y = s.grid_coords(s.moment_info(j)["grid"])
            s.set_source(j, np.cos(0.7 * j + 3 * X) * np.exp(-Y) / (1 + j % 7))
        s.step(2)
        got.append([s.moments(j) for j in range(s.ncomp)])
    for a, b in zip(got[0], got[1]):
        assert np.array_equal(a, b)
    assert_parity(got[0], [np.asarray(a, np.float64) for a in got[2]], FP32_TOL, "fp32")


def _with_sources(N, n, kernel, schedule="merged", aniso=True, steps=2):
    p = _random_problem(N, n, ("periodic", "extrapolation"), "fp32", 991 + N, steps, aniso=aniso)
    s = capi.Stepper.from_problem(p, kernel=kernel, schedule=schedule)
    for j in range(s.ncomp):
        X, Y = s.grid_coords(s.moment_info(j)["grid"])
        s.set_source(j, np.cos(0.7 * j + 3 * X) * np.exp(-Y) / (1 + j % 7))
    s.step(steps)
    return [s.moments(j) for j in range(s.ncomp)]


# above half of L2 with its sources: the five-row bands (more tiles than SMs, N <= 15), the two-row bands
# with each weight once (N >= 50) and, with isotropic scattering, twice
WARMED = [(15, (353, 351), True), (15, (353, 351), False), (9, (601, 399), False), (50, (101, 93), True),
          (55, (101, 93), False), (35, (161, 137), False)]


@pytest.mark.parametrize("N,n,aniso", WARMED)
def test_sources_in_every_moment_shapes(N, n, aniso):
    """As test_sources_in_every_moment, for the tile shapes and decay classes
    that it does not reach; ragged in x and y."""
    from helpers import assert_parity
    from test_gpu_parity import FP32_TOL
    tall = _with_sources(N, n, "tiled_tall", aniso=aniso)
    short = _with_sources(N, n, "tiled_short", aniso=aniso)
    for a, b in zip(tall, short):
        assert np.array_equal(a, b)
    gather = _with_sources(N, n, "gather", aniso=aniso)
    assert_parity(tall, [np.asarray(a, np.float64) for a in gather], FP32_TOL, "fp32")


# kernel, N, cells, sources in every moment: two-row bands, the same with each weight once, 5-row tiles, and
# the warming variants of the two-row and five-row bands
REPEATED = [("tiled_tall", 16, (1001, 799), False), ("tiled_tall", 50, (330, 290), False),
            ("tiled_short", 9, (1501, 1099), False), ("tiled_tall", 20, (505, 501), True),
            ("tiled_tall", 9, (701, 699), True)]


@pytest.mark.parametrize("kernel,N,n,sources", REPEATED)
def test_every_shape_repeats_bit_for_bit(kernel, N, n, sources):
    """As test_runs_repeat_bit_for_bit, for the other shapes."""
    p = _random_problem(N, n, ("extrapolation", "periodic"), "fp32", 996, 1)
    s = capi.Stepper.from_problem(p, kernel=kernel, schedule="literal")
    if sources:
        for j in range(s.ncomp):
            X, Y = s.grid_coords(s.moment_info(j)["grid"])
            s.set_source(j, np.cos(0.7 * j + 3 * X) * np.exp(-Y) / (1 + j % 7))
    start, ref = s.get_state(), None
    for _ in range(12):
        s.set_state(start)
        s.step(4)
        got = s.get_state()
        assert ref is None or got == ref
        ref = got


def test_batch_repeats_bit_for_bit():
    """The batched pass, strips of tiles of instances of several orders."""
    probs = [_random_problem(N, n, ("extrapolation", "periodic"), "fp32", 997 + N, 1)
             for N, n in ((9, (701, 499)), (15, (512, 301)), (3, (1024, 1024)), (12, (333, 640)))]
    b = capi.Batch.from_problems(probs, kernel="tiled_tall")
    start, ref = [i.get_state() for i in b.instances], None
    for _ in range(12):
        for i, u in zip(b.instances, start):
            i.set_state(u)
        b.step(4)
        b.sync()
        got = [i.get_state() for i in b.instances]
        assert ref is None or got == ref
        ref = got
    b.close()
