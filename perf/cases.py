"""Performance cases of the StaRMAP stepper: the calls a user's program makes, over the range of
sizes, orders, precisions and options in use.

A case is a dict of plain values; its "what" names the call:

    steps   Stepper.step(n): n time steps from given moments, material and sources
    to_time Stepper.clear(), advance_to(t), output(0), diagnostics(): a whole run from rest
    batch   Batch.step(n): uneven independent instances advanced together
    closed  Stepper.step(n) of P_7 with the learned order-8 closure
    train   Network.train_step over minibatches, then the parameters read back
    grad    Network.loss_grad of one minibatch

prepare() makes the inputs from the seed on the GPU (moments) and the host (material, sources, as
the entry points take them), run() is one call, exact() the same result in plain torch FP64, with
the moment matrices, the staggered grids and the network written out here once more.
"""
import math

import numpy as np
import torch

from paper_1211_2205_gb300 import capi

HIDDEN, INPUTS, OUTPUTS, NMOM = 128, 38, 9, 36


def listed():
    return [
        # the smallest call: one literal FP64 step of a 64^2 pulse, as a program that looks at the
        # solution (or couples other physics) after every step makes it
        dict(name="p5_fp64_64", what="steps", N=5, nx=64, ny=64, bc="pp", precision="fp64", schedule="literal",
             steps=1, medium="uniform", scatter="iso", source="none"),
        # the run of the paper's section 6.3: P_5 checkerboard on 100^2 cells in FP64 to t = 3.2
        dict(name="p5_fp64_100_to_t", what="to_time", N=5, nx=100, ny=100, bc="ee", precision="fp64",
             schedule="merged", t=3.2),
        # an FP64 run of a middle order: reference solutions, convergence studies
        dict(name="p13_fp64_256", what="steps", N=13, nx=256, ny=256, bc="pp", precision="fp64", schedule="merged",
             steps=4, medium="smooth", scatter="iso", source="none"),
        # a small ragged FP32 grid with the default (literal) schedule, mixed boundaries: parameter studies
        dict(name="p4_fp32_70x45", what="steps", N=4, nx=70, ny=45, bc="pe", precision="fp32", schedule="literal",
             steps=10, medium="blocks", scatter="iso", source="point"),
        # the P_13 checkerboard, 512^2, extrapolation, source in R_0^0
        dict(name="p13_fp32_512", what="steps", N=13, nx=512, ny=512, bc="ee", precision="fp32", schedule="merged",
             steps=20, medium="blocks", scatter="iso", source="point"),
        # the largest: P_39 on 1024^2, smooth random medium, periodic
        dict(name="p39_fp32_1024", what="steps", N=39, nx=1024, ny=1024, bc="pp", precision="fp32",
             schedule="merged", steps=4, medium="smooth", scatter="iso", source="none"),
        # a large grid of odd size at a low order, literal schedule (as time-dependent drivers need it)
        dict(name="p9_fp32_1501x1099", what="steps", N=9, nx=1501, ny=1099, bc="ep", precision="fp32",
             schedule="literal", steps=6, medium="blocks", scatter="iso", source="none"),
        # the beam: Henyey-Greenstein scattering (a decay class per order), a source in every moment
        dict(name="p39_fp32_150_beam", what="steps", N=39, nx=150, ny=150, bc="ee", precision="fp32",
             schedule="merged", steps=5, medium="blocks", scatter="hg", source="beam"),
        # a batch of uneven instances (parameter sweeps)
        dict(name="batch_16", what="batch", count=16, nmin=64, nmax=512, schedule="merged", steps=4),
        # the learned closure of P_7 on the closure workload's grid
        dict(name="closed_p7_512", what="closed", nx=512, ny=512, bc="pp", steps=4),
        # closure training: a stretch of the Adam loop between two looks at the network
        dict(name="train_8192", what="train", samples=1 << 18, batch=8192, steps=32, engine="tcgen05"),
        # loss and gradient on a ragged set of samples (validation, another optimiser)
        dict(name="grad_30011", what="grad", samples=1 << 17, batch=30011, engine="tcgen05"),
    ]


def _moments(N):
    return (N + 1) * (N + 2) // 2


# FP64 updates cost this many FP32 ones when the size of a drawn case is capped
_CAP = 1.0e9


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    bc = rng.choice(["pp", "ee", "pe", "ep"])
    what = rng.choice(["steps"] * 6 + ["fp64", "fp64", "to_time", "slab", "batch", "closed", "train", "grad"])
    if what == "steps":
        while True:
            c = dict(what="steps", N=log_int(1, 47), nx=log_int(24, 1600), ny=log_int(24, 1600), bc=bc,
                     precision="fp32", schedule=rng.choice(["literal", "merged", "merged"]), steps=log_int(1, 20),
                     medium=rng.choice(["uniform", "smooth", "blocks"]),
                     scatter=rng.choice(["iso", "iso", "iso", "hg"]),
                     source=rng.choice(["none", "point", "point", "beam"]))
            classes = c["N"] + 1 if c["scatter"] == "hg" else 2
            if (_moments(c["N"]) + 2 * classes) * c["nx"] * c["ny"] * c["steps"] < _CAP:
                return c
    if what == "fp64":
        while True:
            c = dict(what="steps", N=log_int(1, 39), nx=log_int(16, 512), ny=log_int(16, 512), bc=bc,
                     precision="fp64", schedule=rng.choice(["literal", "merged"]), steps=log_int(1, 10),
                     medium=rng.choice(["uniform", "smooth", "blocks"]), scatter=rng.choice(["iso", "iso", "hg"]),
                     source=rng.choice(["none", "point"]))
            if 16 * _moments(c["N"]) * c["nx"] * c["ny"] * c["steps"] < _CAP:
                return c
    if what == "slab":
        return dict(what="steps", N=log_int(3, 63), nx=log_int(100, 10000), ny=1, bc=bc[0] + "p", precision="fp64",
                    schedule=rng.choice(["literal", "merged"]), steps=log_int(1, 20), medium="blocks", scatter="iso",
                    source="point", system="slab")
    if what == "to_time":
        return dict(what="to_time", N=rng.choice([3, 5, 7, 9]), nx=log_int(30, 150), ny=log_int(30, 150), bc=bc,
                    precision=rng.choice(["fp64", "fp32"]), schedule="merged", t=round(rng.uniform(0.8, 3.2), 3))
    if what == "batch":
        return dict(what="batch", count=log_int(3, 16), nmin=64, nmax=rng.choice([128, 256, 512]),
                    schedule=rng.choice(["literal", "merged"]), steps=log_int(1, 4))
    if what == "closed":
        return dict(what="closed", nx=log_int(48, 700), ny=log_int(48, 700), bc=rng.choice(["pp", "ee"]),
                    steps=log_int(1, 6))
    if what == "train":
        return dict(what="train", samples=1 << 17, batch=log_int(256, 16384), steps=log_int(4, 32),
                    engine=rng.choice(["tcgen05", "mma_sync"]))
    return dict(what="grad", samples=1 << 17, batch=log_int(100, 100000),
                engine=rng.choice(["tcgen05", "mma_sync"]))


# ----------------------------------------------------------------------------------- problem data
class _Problem:
    """The inputs of one 2D P_N (or slab) problem, from the seed alone."""

    def __init__(self, N, nx, ny, bc, medium, scatter, source, rng, ax=(-1.0, 1.0, -1.0, 1.0), system="pn2d",
                 checker=False):
        self.N, self.n, self.ax, self.system = N, (nx, ny), ax, system
        self.bc = tuple({"p": "periodic", "e": "extrapolation"}[b] for b in bc)
        self.p = tuple(int(b == "p") for b in bc)
        self.h = ((ax[1] - ax[0]) / nx, (ax[3] - ax[2]) / ny)
        lx, ly = ax[1] - ax[0], ax[3] - ax[2]
        self.factors = [0.85 ** l for l in range(N + 1)] if scatter == "hg" else None
        # material: a value (or a value per block or lattice node) of sigma_a and sigma_s0
        self.medium = medium
        if checker:                             # absorbing and scattering unit blocks of [0, 7]^2
            a = rng.random((7, 7)) < 0.23
            self.sa, self.ss = 10.0 * a, 1.0 * ~a
        elif medium == "uniform":
            self.sa, self.ss = np.zeros((1, 1)), np.full((1, 1), rng.uniform(0.5, 2.0))
        elif medium == "blocks":
            self.sa, self.ss = rng.uniform(0.0, 5.0, (8, 8)), rng.uniform(0.0, 10.0, (8, 8))
        else:
            self.sa, self.ss = np.zeros((1, 1)), rng.uniform(-1.0, 1.0, (32, 32))
        # sources: a Gaussian in R_0^0, in every moment (a beam), or the checkerboard's centre block
        self.source = "checker" if checker else source
        self.src_at = (ax[0] + lx * rng.uniform(0.3, 0.7), ax[2] + ly * rng.uniform(0.3, 0.7))
        self.src_w = 0.05 * lx
        self.src_amp = rng.standard_normal(4096)
        # moments: three pulses, order l damped as scattering damps it
        self.pulse = [(ax[0] + lx * rng.uniform(0.2, 0.8), ax[2] + ly * rng.uniform(0.2, 0.8),
                       lx * rng.uniform(0.05, 0.2), ly * rng.uniform(0.05, 0.2)) for _ in range(3)]
        self.pulse_amp = rng.standard_normal((4096, 3))

    def coords(self, g):
        """x and y of the points of grid g."""
        out = []
        for d, node in enumerate((g & 1, g >> 1)):
            count = self.n[d] + 1 - self.p[d] if node else self.n[d]
            out.append(self.ax[2 * d] + (self.p[d] * self.h[d] if node else 0.5 * self.h[d]) + self.h[d] * np.arange(count))
        return out

    def _lookup(self, v, x, y, smooth):
        k = v.shape[0]
        if k == 1:
            return np.full((y.size, x.size), float(v[0, 0]))
        u = (x - self.ax[0]) / (self.ax[1] - self.ax[0]) * k
        w = (y - self.ax[2]) / (self.ax[3] - self.ax[2]) * k
        if not smooth:
            # block edges moved off the grid points
            i, j = np.floor(u - 0.37031).astype(int) % k, np.floor(w - 0.37031).astype(int) % k
            return v[j[:, None], i[None, :]]
        i, j = np.floor(u).astype(int), np.floor(w).astype(int)
        fu, fw = (u - i)[None, :], (w - j)[:, None]
        i0, i1, j0, j1 = i[None, :] % k, (i[None, :] + 1) % k, j[:, None] % k, (j[:, None] + 1) % k
        return (1 - fw) * ((1 - fu) * v[j0, i0] + fu * v[j0, i1]) + fw * ((1 - fu) * v[j1, i0] + fu * v[j1, i1])

    def material(self, g):
        x, y = self.coords(g)
        sa = self._lookup(self.sa, x, y, False)
        ss = self._lookup(self.ss, x, y, self.medium == "smooth")
        return sa, (10.0 ** ss if self.medium == "smooth" else ss)

    def source_of(self, j, g):
        """Values of component j's source on its grid, or None."""
        if self.source == "none" or (j > 0 and self.source != "beam"):
            return None
        x, y = self.coords(g)
        if self.source == "checker":
            bx, by = np.floor(x / (self.ax[1] / 7) - 0.001), np.floor(y / (self.ax[3] / 7) - 0.001)
            return 1.0 * ((by == 3)[:, None] & (bx == 3)[None, :])
        ex = np.exp(-((x - self.src_at[0]) / self.src_w) ** 2 / 2)
        ey = np.exp(-((y - self.src_at[1]) / self.src_w) ** 2 / 2)
        amp = 1.0 if j == 0 else 0.5 * self.src_amp[j]
        return amp * ey[:, None] * ex[None, :]

    def moments_of(self, comps, g, orders, dtype):
        """The components' initial values on grid g, [components, ny, nx]."""
        x, y = (torch.from_numpy(v).cuda() for v in self.coords(g))
        amp = torch.from_numpy(self.pulse_amp[comps]).cuda()
        l = torch.tensor([float(orders[j]) for j in comps], dtype=torch.float64, device="cuda")
        amp = amp * (0.8 ** l * torch.where(l > 0, 0.3, 1.0))[:, None]
        if 0 in comps:
            amp[list(comps).index(0)] = 1.0
        ex = torch.stack([torch.exp(-((x - a) / s) ** 2 / 2) for a, _, s, _ in self.pulse])
        ey = torch.stack([torch.exp(-((y - b) / s) ** 2 / 2) for _, b, _, s in self.pulse])
        out = torch.empty((len(comps), y.numel(), x.numel()), dtype=dtype, device="cuda")
        for k in range(0, len(comps), 16):
            out[k:k + 16] = torch.einsum("kr,ry,rx->kyx", amp[k:k + 16], ey, ex)
        return out


def _problem(case, seed):
    rng = np.random.default_rng(seed)
    if case["what"] == "to_time":
        return _Problem(case["N"], case["nx"], case["ny"], case["bc"], "blocks", "iso", "none", rng,
                        ax=(0.0, 7.0, 0.0, 7.0 * case["ny"] / case["nx"]), checker=True)
    if case["what"] == "closed":
        return _Problem(8, case["nx"], case["ny"], case["bc"], "smooth", "iso", "none", rng)
    return _Problem(case["N"], case["nx"], case["ny"], case["bc"], case["medium"], case["scatter"], case["source"],
                    rng, system=case.get("system", "pn2d"))


def _batch_problems(case, seed):
    # the shapes stand for the sweep and stay; the media, sources and pulses come from the seed
    shape, rng = np.random.default_rng(24601), np.random.default_rng(seed)
    out = []
    for _ in range(case["count"]):
        n = int(shape.choice(np.arange(case["nmin"], case["nmax"] + 1, 32)))
        N, bc = int(shape.choice([3, 5, 7, 9, 11, 13, 15])), str(shape.choice(["pp", "ee"]))
        out.append(_Problem(N, n, n, bc, "blocks", "iso", "point", rng, ax=(0.0, 1.0, 0.0, 1.0)))
    return out


# ------------------------------------------------------------------------------------- the library
_stream = None


def _work_stream():
    """The program's one stream: a pass begins when the one before it has ended."""
    global _stream
    if _stream is None:
        _stream = torch.cuda.Stream()
    return _stream.cuda_stream


class _Device:
    """Device memory of a library object, which lives as long as the tensors made from it."""

    def __init__(self, owner, **interface):
        self.owner, self.__cuda_array_interface__ = owner, interface


def _grids(s, precision, owner):
    """The state's own device memory, a view [components, ny, nx] per grid, and each grid's components."""
    comps = [[j for j in range(s.ncomp) if s.moment_info(j)["grid"] == g] for g in range(4)]
    size, views = (8 if precision == "fp64" else 4), []
    for g in range(4):
        nx, ny = s.grid_info(g)[:2]
        at = [s.device_ptr(j) for j in comps[g]]
        if not at:
            views.append(None)
            continue
        step = at[1][0] - at[0][0] if len(at) > 1 else at[0][1] * size * (ny + 2)
        assert all(a[0] == at[0][0] + k * step for k, a in enumerate(at))
        views.append(torch.as_tensor(_Device(
            owner, shape=(len(at), ny, nx), strides=(step, at[0][1] * size, size), typestr="<f%d" % size,
            data=(at[0][0] + at[0][2] * size, False), version=3), device="cuda"))
    return views, comps


def _load(s, p, precision, moments=True, comps=None, owner=None):
    """Material, sources (of the first comps components) and, through the state's device memory, the
    moments of a problem; returns the state as tensors, which keep the owner (the stepper, or its
    batch) alive."""
    orders = [s.moment_info(j)["l"] for j in range(s.ncomp)]
    grid = [s.moment_info(j)["grid"] for j in range(s.ncomp)]
    if p.factors is not None:
        s.set_scattering_factors(p.factors)
    for g in range(4):
        s.set_material(g, *p.material(g))
    for j in range(comps or s.ncomp):
        q = p.source_of(j, grid[j])
        if q is not None:
            s.set_source(j, q)
    views, comps = _grids(s, precision, owner or s)
    if moments:
        s.sync()
        for g in range(4):
            if views[g] is not None:
                views[g].copy_(p.moments_of(comps[g], g, orders, views[g].dtype))
        torch.cuda.synchronize()
        s.set_moment(0, s.moments(0))           # an upload: the library refreshes its boundary copies
    return [v for v in views if v is not None]


def _params(rng, scale_out):
    p = {"W1": rng.normal(0, INPUTS ** -0.5, (HIDDEN, INPUTS)), "b1": rng.normal(0, 0.1, HIDDEN),
         "W2": rng.normal(0, HIDDEN ** -0.5, (HIDDEN, HIDDEN)), "b2": rng.normal(0, 0.1, HIDDEN),
         "W3": scale_out * rng.normal(0, HIDDEN ** -0.5, (OUTPUTS, HIDDEN)), "b3": np.zeros(OUTPUTS)}
    return capi.params_from_dict(p)


def _samples(case, seed):
    """Network inputs (normalised moments, log material), targets of a smooth law, minibatch orders."""
    r = torch.Generator(device="cuda").manual_seed(seed)
    X = torch.randn((case["samples"], INPUTS), generator=r, device="cuda")
    X[:, :NMOM] *= math.sqrt(NMOM) / X[:, :NMOM].norm(dim=1, keepdim=True)
    X[:, NMOM:] = torch.rand((case["samples"], 2), generator=r, device="cuda") * 1.5
    A = torch.randn((INPUTS, OUTPUTS), generator=r, device="cuda") / math.sqrt(INPUTS)
    T = 0.3 * torch.tanh(X @ A)
    steps = case.get("steps", 1)
    idx = torch.randint(0, case["samples"], (steps, case["batch"]), generator=r, device="cuda", dtype=torch.int32)
    return X, T, idx


def _learning_rate(k):
    return 2e-3 * 0.98 ** k


def prepare(case, seed):
    what = case["what"]
    if what in ("train", "grad"):
        params = _params(np.random.default_rng(seed), 0.1)
        X, T, idx = _samples(case, seed)
        net = capi.Network(params, stream=_work_stream())
        net.set_engine(case["engine"])
        out = torch.empty(capi.MLP_PARAMS, device="cuda"), torch.empty(1, device="cuda")
        torch.cuda.synchronize()
        return dict(what=what, net=net, X=X, T=T, idx=idx, batch=case["batch"], steps=case.get("steps", 1), out=out)
    if what == "batch":
        ps = _batch_problems(case, seed)
        b = capi.Batch([dict(N=p.N, ax=p.ax, n=p.n, bc=p.bc, precision="fp32", schedule=case["schedule"])
                        for p in ps], stream=_work_stream())
        views = [_load(s, p, "fp32", owner=b) for s, p in zip(b.instances, ps)]
        return dict(what=what, batch=b, steps=case["steps"], views=[v for vs in views for v in vs])
    p = _problem(case, seed)
    if what == "closed":
        s = capi.Stepper(N=7, ax=p.ax, n=p.n, bc=p.bc, precision="fp32", schedule="merged", closure="mlp8",
                         stream=_work_stream())
        s.set_closure(_params(np.random.default_rng(seed + 1), 0.3))
        views = _load(s, p, "fp32", comps=NMOM)
        return dict(what=what, s=s, steps=case["steps"], views=views)
    s = capi.Stepper(N=p.N, ax=p.ax, n=p.n, bc=p.bc, precision=case["precision"], system=p.system,
                     schedule=case["schedule"], stream=_work_stream())
    views = _load(s, p, case["precision"], moments=what == "steps")
    return dict(what=what, s=s, steps=case.get("steps"), t=case.get("t"), views=views)


def run(state):
    what = state["what"]
    if what == "steps" or what == "closed":
        state["s"].step(state["steps"])
        return state["views"]
    if what == "to_time":
        s = state["s"]
        s.clear()
        s.advance_to(state["t"])
        flux = s.output(0)
        mass, l2, _ = s.diagnostics()
        return dict(flux=flux, mass=mass, l2=l2, state=state["views"])
    if what == "batch":
        state["batch"].step(state["steps"])
        return state["views"]
    net, B, grad_loss = state["net"], state["batch"], state["out"]
    if what == "train":
        for k in range(state["steps"]):
            net.train_step(state["X"], state["T"], B, _learning_rate(k), loss=grad_loss[1], idx=state["idx"][k])
        return dict(params=net.params, loss=grad_loss[1])
    net.loss_grad(state["X"], state["T"], B, grad_loss[0], grad_loss[1], idx=state["idx"][0])
    return dict(grad=grad_loss[0], loss=grad_loss[1])


# ---------------------------------------------------------------------------------- what it costs
ON_CHIP = 126e6         # bytes of L2: a state within it need not leave the chip between the steps


def _step_work(K, classes, sources, nx, ny, size, steps):
    state, fixed = K * nx * ny * size, (4 * 2 * classes + sources) * nx * ny * size
    moved = 2 * state + fixed
    return dict(bytes=float(moved * (steps if moved > ON_CHIP else 1)),
                # per value: two differences, about eight weighted sums of them, the decayed update
                flops=float(K * nx * ny * steps * 21))


def work(case):
    what = case["what"]
    if what in ("train", "grad"):
        weights, steps, B = HIDDEN * (INPUTS + HIDDEN + OUTPUTS), case.get("steps", 1), case["batch"]
        return dict(bytes=float(steps * B * 4 * (INPUTS + OUTPUTS + 1) + 4 * 4 * capi.MLP_PARAMS),
                    flops=float(steps * B * (6 * weights - 2 * HIDDEN * INPUTS)))
    if what == "batch":
        each = [_step_work(_moments(p.N), 2, 1, *p.n, 4, 1) for p in _batch_problems(case, 0)]
        total = {k: sum(w[k] for w in each) for k in ("bytes", "flops")}
        many = case["steps"] if total["bytes"] > ON_CHIP else 1
        return dict(bytes=total["bytes"] * many, flops=total["flops"] * case["steps"])
    if what == "closed":
        w = _step_work(45, 2, 0, case["nx"], case["ny"], 4, case["steps"])
        net = 2 * HIDDEN * (INPUTS + HIDDEN + OUTPUTS) * case["nx"] * case["ny"]
        return dict(bytes=w["bytes"], flops=w["flops"] + net * (case["steps"] + 1))
    size = 8 if case["precision"] == "fp64" else 4
    if what == "to_time":
        h = 7.0 / case["nx"]
        steps = math.ceil(case["t"] * _lambda_max(case["N"]) / (0.5 * h))
        return _step_work(_moments(case["N"]), 2, 1, case["nx"], case["ny"], size, steps)
    K = case["N"] + 1 if case.get("system") == "slab" else _moments(case["N"])
    classes = case["N"] + 1 if case["scatter"] == "hg" else 2
    return _step_work(K, classes, {"none": 0, "point": 1, "beam": K}[case["source"]], case["nx"], case["ny"], size,
                      case["steps"])


# ------------------------------------------------------------------------------- in 64 bits, plain
def _lambda_max(N):
    return float(np.polynomial.legendre.leggauss(N + 1)[0][-1])


def _matrices(N, system):
    """Orders of the real moments, and Mx, My as {row: [(column, value)]}: the complex recursion of
    section 3 (Seibold & Frank, arXiv:1211.2205) and its real combinations."""
    if system == "slab":
        Mx = {l: [(l + d, (l + (d > 0)) / (2 * l + 1)) for d in (-1, 1) if 0 <= l + d <= N] for l in range(N + 1)}
        return list(range(N + 1)), Mx, {l: [] for l in range(N + 1)}

    def root(a, b):
        return math.sqrt(a / b) if a > 0 else 0.0

    def up(l, m):           # weight of (l, m) in a row of order l + 1
        return root((l + m + 1) * (l + m + 2), (2 * l + 3) * (2 * l + 1))

    def down(l, m):         # and in a row of order l - 1
        return root((l - m) * (l - m - 1), (2 * l + 1) * (2 * l - 1))

    # row (l, m): (column, x value, y value)
    rows = {}
    for l in range(N + 1):
        for m in range(-l, l + 1, 2):
            r = [((l - 1, m - 1), -0.5 * up(l - 1, m - 1), 0.5j * up(l - 1, m - 1)),
                 ((l + 1, m - 1), 0.5 * down(l + 1, m - 1), -0.5j * down(l + 1, m - 1)),
                 ((l - 1, m + 1), 0.5 * up(l - 1, -m - 1), 0.5j * up(l - 1, -m - 1)),
                 ((l + 1, m + 1), -0.5 * down(l + 1, -m - 1), -0.5j * down(l + 1, -m - 1))]
            rows[l, m] = [(k, a, b) for k, a, b in r if 0 <= k[0] <= N and abs(k[1]) <= k[0]]
    real, orders, used = [], [], {}
    for l in range(N + 1):
        for m in range(l, -1, -2):
            s, q = (-1.0) ** m, math.sqrt(0.5)
            for pair in ([{(l, 0): 1.0}] if m == 0 else
                         [{(l, m): s * q, (l, -m): q}, {(l, m): 1j * s * q, (l, -m): -1j * q}]):
                for k, v in pair.items():
                    used.setdefault(k, []).append((len(real), v))
                real.append(pair)
                orders.append(l)
    out = []
    for axis in (1, 2):
        M = {}
        for r, pair in enumerate(real):
            acc = {}
            for k, v in pair.items():
                for entry in rows[k]:
                    for c, w in used[entry[0]]:
                        acc[c] = acc.get(c, 0.0) + v * entry[axis] * np.conj(w)
            M[r] = [(c, float(np.real(a))) for c, a in sorted(acc.items()) if abs(np.real(a)) > 1e-13]
        out.append(M)
    return orders, out[0], out[1]


class _Exact:
    """The staggered scheme in FP64: one tensor [components, ny, nx] per grid."""

    def __init__(self, p, N, dt=None):
        self.p, self.N = p, N
        self.orders, self.Mx, self.My = _matrices(N, p.system)
        h = p.h[0] if p.system == "slab" else min(p.h)
        self.dt = 0.5 * h / _lambda_max(N)
        grid, todo = {0: 0}, [0]
        while todo:
            i = todo.pop()
            for M, bit in ((self.Mx, 1), (self.My, 2)):
                for c, _ in M[i]:
                    if c not in grid:
                        grid[c] = grid[i] ^ bit
                        todo.append(c)
        self.comps = [[j for j in range(len(self.orders)) if grid[j] == g] for g in range(4)]
        self.grid = grid
        self.local = {j: k for c in self.comps for k, j in enumerate(c)}
        self.size = [tuple(len(v) for v in p.coords(g)) for g in range(4)]
        self.U = [torch.zeros((len(c), n[1], n[0]), dtype=torch.float64, device="cuda")
                  for c, n in zip(self.comps, self.size)]
        self.frozen = 0             # the last components, which the passes leave alone
        self.decay, self.sources = [], [[] for _ in range(4)]
        for g in range(4):
            sa, ss = (torch.from_numpy(np.ascontiguousarray(v)).cuda() for v in p.material(g))
            f = p.factors
            classes = range(N + 1) if f is not None else range(2)
            self.decay.append([sa if c == 0 else sa + ss - (ss * f[c] if f is not None else 0.0) for c in classes])

    def set_sources(self, dtype):
        for j in range(len(self.orders)):
            q = self.p.source_of(j, self.grid[j])
            if q is not None:
                self.sources[self.grid[j]].append((self.local[j], torch.from_numpy(q).cuda().to(dtype).double()))

    def set_moments(self, dtype):
        for g in range(4):
            if self.comps[g]:
                self.U[g] = self.p.moments_of(self.comps[g], g, self.orders, dtype).double()

    def _difference(self, V, axis, target_node):
        """Right minus left neighbour along an axis, on the grid staggered along it."""
        d = 0 if axis == 2 else 1
        per, n = self.p.p[d], V.shape[axis]
        count = self.p.n[d] + 1 - per if target_node else self.p.n[d]
        right = torch.arange(count, device="cuda") + (per if target_node else 1 - per)
        at = [(i % n if per else i.clamp(0, n - 1)) for i in (right, right - 1)]
        return V.index_select(axis, at[0]) - V.index_select(axis, at[1])

    def half(self, odd, tau):
        """One parity's exact solve over tau with the other frozen."""
        new = {}
        for g in ((1, 2) if odd else (0, 3)):
            if not self.comps[g]:
                continue
            W = torch.zeros_like(self.U[g])
            for M, bit, axis in ((self.Mx, 1, 2), (self.My, 2, 1)):
                if not self.comps[g ^ bit]:
                    continue
                D = self._difference(self.U[g ^ bit], axis, bool(g & bit))
                h = self.p.h[0 if bit == 1 else 1]
                most = max(len(M[j]) for j in self.comps[g])
                for k in range(most):
                    rows = [i for i, j in enumerate(self.comps[g]) if len(M[j]) > k]
                    take = torch.tensor([self.local[M[self.comps[g][i]][k][0]] for i in rows], device="cuda")
                    c = torch.tensor([-M[self.comps[g][i]][k][1] / h for i in rows], dtype=torch.float64,
                                     device="cuda")
                    for a in range(0, len(rows), 64):
                        W[torch.tensor(rows[a:a + 64], device="cuda")] += c[a:a + 64, None, None] * D[take[a:a + 64]]
                del D
            for k, q in self.sources[g]:
                W[k] += q
            for cls, c in enumerate(self.decay[g]):
                a = torch.exp(-c * tau)
                b = torch.where(c == 0, torch.full_like(c, tau), -torch.expm1(-c * tau) / torch.where(c == 0, 1.0, c))
                isotropic = len(self.decay[g]) == 2
                for i, j in enumerate(self.comps[g]):
                    l = self.orders[j]
                    if (min(l, 1) if isotropic else l) != cls or j >= len(self.orders) - self.frozen:
                        continue
                    W[i] = a * self.U[g][i] + b * W[i]
            for i, j in enumerate(self.comps[g]):
                if j >= len(self.orders) - self.frozen:
                    W[i] = self.U[g][i]
            new[g] = W
        for g, W in new.items():
            self.U[g] = W

    def steps(self, n, before_odd=None):
        """n steps; consecutive odd halves are one solve over dt, which is the same."""
        for k in range(n + 1):
            if before_odd:
                before_odd()
            self.half(True, self.dt if 0 < k < n else 0.5 * self.dt)
            if k < n:
                self.half(False, self.dt)

    def state(self):
        return [u for u in self.U if u.shape[0]]


def _network(P, X):
    H1 = torch.tanh(X @ P["W1"].T + P["b1"])
    H2 = torch.tanh(H1 @ P["W2"].T + P["b2"])
    return H1, H2, H2 @ P["W3"].T + P["b3"]


def _predict(e, P):
    """The closure: order-8 moments from the local moments of order <= 7 and the material."""
    px, py = e.p.p
    nx, ny = e.p.n

    def to_cells(V, axis, per, n):
        if per:                 # cell i lies between nodes i - 1 and i
            return 0.5 * (V + V.roll(1, axis))
        return 0.5 * (V.narrow(axis, 0, n) + V.narrow(axis, 1, n))

    feats = torch.empty((NMOM, ny, nx), dtype=torch.float64, device="cuda")
    for j in range(NMOM):
        g = e.grid[j]
        v = e.U[g][e.local[j]]
        if g & 1:
            v = to_cells(v, 1, px, nx)
        if g & 2:
            v = to_cells(v, 0, py, ny)
        feats[j] = v
    s = feats.square().mean(0).sqrt()
    X = torch.cat([feats / torch.where(s > 0, s, 1.0), torch.log1p(e.decay[0][0])[None],
                   torch.log1p(e.decay[0][1] - e.decay[0][0])[None]]).reshape(INPUTS, -1).T
    Y = torch.cat([_network(P, x)[2] for x in X.split(1 << 16)])
    Y = (Y.T.reshape(OUTPUTS, ny, nx)) * s

    def to_nodes(V, axis, per):
        if per:                 # node k lies between cells k and k + 1
            return 0.5 * (V + V.roll(-1, axis))
        n = V.shape[axis]
        i = torch.arange(n + 1, device="cuda")
        return 0.5 * (V.index_select(axis, (i - 1).clamp(0)) + V.index_select(axis, i.clamp(max=n - 1)))

    for o in range(OUTPUTS):
        g, v = e.grid[NMOM + o], Y[o]
        if g == 3:
            v = to_nodes(to_nodes(v, 1, px), 0, py)
        e.U[g][e.local[NMOM + o]] = v


def _gradient(P, X, T):
    H1, H2, Y = _network(P, X)
    R = Y - T
    dY = 2.0 * R / R.numel()
    dZ2 = (dY @ P["W3"]) * (1 - H2 * H2)
    dZ1 = (dZ2 @ P["W2"]) * (1 - H1 * H1)
    g = {"W1": dZ1.T @ X, "b1": dZ1.sum(0), "W2": dZ2.T @ H1, "b2": dZ2.sum(0), "W3": dY.T @ H2, "b3": dY.sum(0)}
    return g, R.square().mean()


def _flat(P):
    return torch.cat([P[k].reshape(-1) for k in ("W1", "b1", "W2", "b2", "W3", "b3")])


def _unflat(v):
    out, at = {}, 0
    for k, shape in (("W1", (HIDDEN, INPUTS)), ("b1", (HIDDEN,)), ("W2", (HIDDEN, HIDDEN)), ("b2", (HIDDEN,)),
                     ("W3", (OUTPUTS, HIDDEN)), ("b3", (OUTPUTS,))):
        n = math.prod(shape)
        out[k] = v[at:at + n].reshape(shape)
        at += n
    return out


def _double(params):
    return torch.from_numpy(params.astype(np.float64)).cuda()


def exact(case, seed):
    what = case["what"]
    if what in ("train", "grad"):
        w = _double(_params(np.random.default_rng(seed), 0.1))
        X, T, idx = _samples(case, seed)
        if what == "grad":
            i = idx[0].long()
            g, loss = _gradient(_unflat(w), X[i].double(), T[i].double())
            return dict(grad=_flat(g), loss=loss.reshape(1))
        m, v = torch.zeros_like(w), torch.zeros_like(w)
        for k in range(case["steps"]):
            i = idx[k].long()
            g, loss = _gradient(_unflat(w), X[i].double(), T[i].double())
            g = _flat(g)
            m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
            w = w - _learning_rate(k) * (m / (1 - 0.9 ** (k + 1))) / ((v / (1 - 0.999 ** (k + 1))).sqrt() + 1e-8)
        return dict(params=w, loss=loss.reshape(1))
    if what == "batch":
        out = []
        for p in _batch_problems(case, seed):
            e = _Exact(p, p.N)
            e.set_sources(torch.float32)
            e.set_moments(torch.float32)
            e.steps(case["steps"])
            out += e.state()
        return out
    p = _problem(case, seed)
    e = _Exact(p, p.N)
    if what == "closed":
        P = _unflat(_double(_params(np.random.default_rng(seed + 1), 0.3)))
        e.set_moments(torch.float32)
        e.frozen = OUTPUTS
        e.steps(case["steps"], before_odd=lambda: _predict(e, P))
        return e.state()
    dtype = torch.float64 if case["precision"] == "fp64" else torch.float32
    e.set_sources(dtype)
    if what == "steps":
        e.set_moments(dtype)
        e.steps(case["steps"])
        return e.state()
    n = max(1, math.ceil(case["t"] / e.dt - 1e-9))
    e.steps(n - 1)
    before = e.U[0][0].clone()
    e.steps(1)
    part = case["t"] / e.dt - (n - 1)
    cell = p.h[0] * p.h[1]
    return dict(flux=(1 - part) * before + part * e.U[0][0], mass=float(e.U[0][0].sum() * cell),
                l2=math.sqrt(sum(float(u.square().sum()) for u in e.U) * cell), state=e.state())
