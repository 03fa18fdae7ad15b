"""The 8 x 8 tiles of the tile kernel against its 16 x 16 tiles.

Every node goes through the same operations in the same order whatever the
tile, so the states are equal to the bit; the sizes put domain edges, walls and
periodic seams at every place of a tile, down to grids smaller than the region
of one block."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2306_08216_gb300 import mdf  # noqa: E402
from paper_2306_08216_gb300 import workloads as W  # noqa: E402

LID = dict(walls=(True, True), u_wall=(0, 0, 0, 0.1))
PL = dict(nu=1e-3, power_law=(1e-3, 0.7, 5e-5, 2e-2))


def curvi(nx, ny):
    X, Y = W.trapezoid_grid(nx, ny)
    return dict(grid="curvilinear", x=X, y=Y)


CASES = {
    "periodic": lambda nx, ny: dict(nu=0.01, lx=2 * math.pi, ly=2 * math.pi),
    "periodic_forced": lambda nx, ny: dict(nu=0.01, force=(1e-3, -2e-4), force_rate=(1e-4, 0.0), source=1e-3),
    "cavity": lambda nx, ny: dict(nu=1e-3, **LID),
    "power_law_cavity": lambda nx, ny: dict(**LID, **PL),
    "channel": lambda nx, ny: dict(nu=0.01, walls=(False, True), force=(1e-3, 0.0)),
    "stretched": lambda nx, ny: dict(nu=1e-3, grid="separable", x=W.tanh_nodes(nx, 1.5), y=W.tanh_nodes(ny, 1.5), **LID),
    "trapezoid_power_law": lambda nx, ny: dict(**curvi(nx, ny), **LID, **PL),
}


@pytest.mark.parametrize("name", sorted(CASES))
@pytest.mark.parametrize("nx,ny", [(5, 6), (8, 16), (17, 9), (65, 33), (150, 130)])
def test_small_tiles_equal_large_tiles_bitwise(name, nx, ny):
    out = []
    for rows in (16, 8):
        s = mdf.Solver(nx, ny, **CASES[name](nx, ny))
        s.set_launch(0, rows)
        info = s.launch_info()
        assert info["kernel"] == "tile" and info["rows_per_block"] == rows
        s.init(*W.random_fields(nx, ny, 0.02, seed=nx + ny))
        s.step(37)  # two graph replays and five launches
        out.append(s.state())
    np.testing.assert_array_equal(out[0], out[1])
