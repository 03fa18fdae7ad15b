"""The march kernels of each kind of body force.

A constant force has a kernel of its own; force fields come from a ring of rows
copied ahead.  A field that holds the constant in every node goes through the
same operations with the same values, so the two give equal bits; a varying
field is compared between the strip widths and band heights of the plans, which
put the ring's first rows, the periodic seam and ragged strips in different
places, again to the bit."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2306_08216_gb300 import mdf  # noqa: E402
from paper_2306_08216_gb300 import workloads as W  # noqa: E402

LID = dict(walls=(True, True), u_wall=(0, 0, 0, 0.1))
KINDS = {
    "periodic": lambda nx, ny: dict(nu=0.01, lx=2 * math.pi, ly=2 * math.pi),
    "periodic_bf16": lambda nx, ny: dict(nu=0.01, lx=2 * math.pi, ly=2 * math.pi, storage="bf16"),
    "periodic_rho0": lambda nx, ny: dict(nu=0.01, lx=2 * math.pi, ly=2 * math.pi, rho0=True),
    "channel": lambda nx, ny: dict(nu=0.01, walls=(False, True)),
    "power_law_cavity": lambda nx, ny: dict(power_law=(1e-3, 0.7, 5e-5, 2e-2), **LID),
    "stretched": lambda nx, ny: dict(nu=1e-3, grid="separable", x=W.tanh_nodes(nx, 1.5), y=W.tanh_nodes(ny, 1.5), **LID),
}


def march(name, nx, ny, plan, force, rate=None):
    s = mdf.Solver(nx, ny, **KINDS[name](nx, ny))
    s.set_launch(*plan)
    s.init(*W.random_fields(nx, ny, 0.02, seed=nx + ny))
    s.set_force(force)
    if rate is not None:
        s.set_force_rate(rate)
    s.step(19)  # one graph replay and three launches
    return s.state()


@pytest.mark.parametrize("name", sorted(KINDS))
@pytest.mark.parametrize("nx,ny", [(9, 7), (121, 40), (250, 131)])
def test_constant_force_equals_constant_field_bitwise(name, nx, ny):
    fx, fy = np.float32(1e-3), np.float32(-2e-4)
    field = (np.full((ny, nx), fx), np.full((ny, nx), fy))
    for plan in [(128, 5)] + ([] if name == "periodic_rho0" else [(256, 64)]):
        const = march(name, nx, ny, plan, (float(fx), float(fy)))
        assert not np.array_equal(const, march(name, nx, ny, plan, None))
        np.testing.assert_array_equal(const, march(name, nx, ny, plan, field))


@pytest.mark.parametrize("rate", [False, True])
@pytest.mark.parametrize("name", sorted(set(KINDS) - {"periodic_rho0"}))
def test_force_fields_are_the_same_on_every_plan_bitwise(name, rate):
    nx, ny = 250, 131
    g = np.random.default_rng(11)
    field = tuple(g.uniform(-1e-3, 1e-3, (ny, nx)).astype(np.float32) for _ in range(2))
    change = tuple(g.uniform(-1e-2, 1e-2, (ny, nx)).astype(np.float32) for _ in range(2)) if rate else None
    ref = march(name, nx, ny, (128, 131), field, change)
    for plan in [(128, 1), (128, 17), (256, 8), (256, 131)]:
        np.testing.assert_array_equal(ref, march(name, nx, ny, plan, field, change))
