"""Body-force fields, force rates and sources of the problems of a batch.

The batch marches keep a ring of force rows of their own.  FP32: every problem
equals its solo run to the bit, whatever its neighbours carry (fields that vary in
y, rates with planes of their own, sources, constants, nothing) and wherever the
bands end.  16-bit storage: within the N-step bound of the oracle that the unforced
batches have, 5e-7 U0 + 15 N u_r max|n|."""
import math

import numpy as np
import pytest

from oracle.oracle import Oracle
from paper_2306_08216_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2306_08216_gb300 import mdf  # noqa: E402

LID = dict(walls=(True, True), u_wall=(0, 0, 0, 0.1))
CHANNEL = dict(walls=(False, True))
SIZES = [(97, 131), (65, 40), (130, 77), (180, 33), (33, 50), (90, 89), (41, 64)]
FAMILIES = {
    "walls": lambda i, nx, ny: dict(nu=1e-3, **(CHANNEL if i % 2 else LID)),
    "stretched": lambda i, nx, ny: dict(nu=1e-3, grid="separable", x=W.tanh_nodes(nx, 1.5), y=W.tanh_nodes(ny, 1.5), **LID),
    "periodic": lambda i, nx, ny: dict(nu=0.01, lx=2 * math.pi, ly=2 * math.pi * ny / nx),
    "power_law": lambda i, nx, ny: dict(power_law=(1e-3, 0.7, 5e-5, 2e-2), **(CHANNEL if i % 2 else LID)),
    "trapezoid": lambda i, nx, ny: dict(nu=1e-3, grid="curvilinear", x=W.trapezoid_grid(nx, ny)[0],
                                        y=W.trapezoid_grid(nx, ny)[1], **LID),
}


def smooth(nx, ny, amp, seed):
    """A field that varies in x and y, and differs from row to row."""
    g = np.random.default_rng(seed)
    a, b = g.uniform(0, 2 * math.pi, 2)
    x, y = np.arange(nx) / nx, np.arange(ny) / ny
    return (amp * (np.sin(2 * math.pi * x + a)[None, :] + np.cos(4 * math.pi * y + b)[:, None])).astype(np.float32)


def force_up(p, i, nx, ny, source):
    """The forcing of problem i, on a solver, a problem of a batch or the oracle."""
    pair = lambda amp, k: (smooth(nx, ny, amp, 10 * i + k), smooth(nx, ny, amp, 10 * i + k + 1))  # noqa: E731
    if i in (0, 5):
        p.set_force(pair(1e-3, 0))
    if i == 1:
        p.set_force(pair(1e-3, 2))
        p.set_force_rate(pair(1e-2, 4))
    if i == 2:
        p.set_force((1e-3, -5e-4))
    if i == 5 and source:
        p.set_source(smooth(nx, ny, 1e-3, 10 * i + 6))
    if i == 4:
        p.set_force_rate(pair(1e-2, 7))
    if i == 6 and source:
        p.set_source(1e-3)
    # problem 3 has none


@pytest.mark.parametrize("kernel", ["march", "march_rolled", "tile"])
@pytest.mark.parametrize("family", sorted(FAMILIES))
def test_forced_problems_equal_solo_runs_bitwise(family, kernel):
    if family == "trapezoid" and kernel == "march_rolled":
        pytest.skip("the rolled march serves uniform and separable grids")
    if family == "periodic" and kernel != "tile":
        pytest.skip("alone, a periodic Newtonian problem runs the fast path; compared with the oracle below")
    source = family != "power_law"
    batch = mdf.Batch([dict(nx=nx, ny=ny, **FAMILIES[family](i, nx, ny)) for i, (nx, ny) in enumerate(SIZES)])
    batch.set_launch(kernel)
    solos = []
    for i, (nx, ny) in enumerate(SIZES):
        s = mdf.Solver(nx, ny, **FAMILIES[family](i, nx, ny))
        s.set_launch(*((0, 16) if kernel == "tile" else (128, 7)))
        f = W.random_fields(nx, ny, 0.02, seed=i)
        s.init(*f)
        batch.init(i, *f)
        force_up(s, i, nx, ny, source)
        force_up(batch.problem(i), i, nx, ny, source)
        solos.append(s)
    for n in (37, 2):  # graph replays and launches
        batch.step(n)
    for i, s in enumerate(solos):
        s.step(39)
        assert np.isfinite(s.state()).all()
        np.testing.assert_array_equal(batch.problem(i).state(), s.state(), err_msg=str(i))


def feq(u, v, P):
    out = np.zeros((2, 5) + u.shape)
    for a, (ub, fx, fy) in enumerate([(u, u * u + P, u * v), (v, u * v, v * v + P)]):
        out[a, 0] = ub / 5
        out[a, 1], out[a, 3] = ub / 5 + fx / 2, ub / 5 - fx / 2
        out[a, 2], out[a, 4] = ub / 5 + fy / 2, ub / 5 - fy / 2
    return out


@pytest.mark.parametrize("storage", ["fp32", "fp16", "bf16"])
@pytest.mark.parametrize("family", ["walls", "periodic", "power_law"])
def test_forced_batches_against_the_oracle(family, storage):
    steps, U0 = 40, 0.1
    batch = mdf.Batch([dict(nx=nx, ny=ny, storage=storage, **FAMILIES[family](i, nx, ny))
                       for i, (nx, ny) in enumerate(SIZES)])
    batch.set_launch("march_rolled")
    source = storage == "fp32" and family != "power_law"
    for i, (nx, ny) in enumerate(SIZES):
        force_up(batch.problem(i), i, nx, ny, source)
    batch.step(steps)
    for i, (nx, ny) in enumerate(SIZES):
        o = Oracle(nx, ny, **FAMILIES[family](i, nx, ny))
        o.init(*W.zeros(nx, ny))
        force_up(o, i, nx, ny, source)
        o.step(steps)
        st, f = o.state(), o.fields()
        n = float(np.abs(st - feq(f["u"], f["v"], f["P"])).max())
        bound = 1e-5 * U0 if storage == "fp32" else 5e-7 * U0 + steps * 15 * {"fp16": 2.0 ** -11, "bf16": 2.0 ** -8}[storage] * n
        err = float(np.abs(batch.problem(i).state().astype(np.float64) - st).max())
        assert err <= bound, (i, err, bound)
