"""The launch plan a solver picks for itself, for each kind of force.

A march has one kernel without a force, one for a constant force and one for
force fields and sources, and a power-law fluid costs more in motion than at rest;
the plan has to be the better one of the kernel that runs.  The values do not
depend on it."""
import time

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2306_08216_gb300 import mdf  # noqa: E402
from paper_2306_08216_gb300 import workloads as W  # noqa: E402

CHANNEL = dict(walls=(False, True), nu=0.01)
CAVITY = dict(walls=(True, True), u_wall=(0, 0, 0, 0.1), power_law=(1e-3, 0.7, 5e-5, 2e-2))


def make(nx, ny, kw, plan=None):
    s = mdf.Solver(nx, ny, **kw)
    if plan:
        s.set_launch(*plan)
    s.init(*W.random_fields(nx, ny, 0.01, seed=3))
    return s


def us_per_step(s, n=64):
    s.step(n)
    torch.cuda.synchronize()
    best = 1e9
    for _ in range(6):
        t0 = time.perf_counter()
        s.step(n)
        torch.cuda.synchronize()
        best = min(best, time.perf_counter() - t0)
    return best / n * 1e6


@pytest.mark.parametrize("name", ["power_law", "source", "source_field"])
def test_own_plan_is_the_faster_march(name):
    """700 rows of 1200 columns on 152 SMs: one wave of 128 threads (bands of 16
    rows) and one of 256 (12 rows) are close without a force and 6 to 12 % apart
    here."""
    nx, ny = 1200, 700
    out = []
    for plan in (None, (128, 16), (256, 12)):
        s = make(nx, ny, CAVITY if name == "power_law" else CHANNEL, plan)
        if name == "source":
            s.set_source(1e-5)
        elif name == "source_field":
            s.set_source(np.random.default_rng(1).uniform(-1e-5, 1e-5, (ny, nx)).astype(np.float32))
        out.append(us_per_step(s))
    assert out[0] <= 1.05 * min(out[1:]), out


@pytest.mark.parametrize("nx,ny,kw", [(1200, 700, CHANNEL), (700, 600, CHANNEL), (300, 260, dict(nu=0.01)),
                                      (1024, 520, dict(nu=0.01, storage="bf16")), (64, 64, dict(nu=0.01))])
def test_values_do_not_depend_on_the_plan(nx, ny, kw):
    own = make(nx, ny, kw)
    plain = own.launch_info()
    pinned = make(nx, ny, kw, (0, 16) if plain["kernel"] == "tile" else (128, 13))
    field = tuple(np.random.default_rng(2).uniform(-1e-4, 1e-4, (ny, nx)).astype(np.float32) for _ in range(2))
    for k, force in enumerate(((1e-4, 0.0), (2e-4, 1e-4), field, (1e-4, 0.0), None)):
        before = own.launch_info()
        for s in (own, pinned):
            s.set_force(force)
            s.step(35)  # two graph replays and three launches
        now = own.launch_info()
        assert now["kernel"] == plain["kernel"]
        if k == 1:
            assert now == before  # the same kind: the same plan
        if force is None:
            assert now == plain
        np.testing.assert_array_equal(own.state(), pinned.state())
    assert pinned.launch_info()["rows_per_block"] == (16 if plain["kernel"] == "tile" else 13)
