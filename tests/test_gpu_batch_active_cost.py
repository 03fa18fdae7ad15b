"""Host time of retiring and re-admitting a problem of a batch with a pinned kernel.

It rebuilds the band heights and the table of work items.  Sorting every item, or
playing the blocks' shares through item by item, took 240 us for 48 cavities and
960 us for 128 trapezoids in tiles; without either it was 34 and 121 us before
bands had heights by load, mostly the copies to the device (now 37 and 80).  The
limits are three times the former."""
import time

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2306_08216_gb300 import mdf  # noqa: E402
from paper_2306_08216_gb300 import workloads as W  # noqa: E402

LID = dict(walls=(True, True), u_wall=(0, 0, 0, 0.1), power_law=(1e-3, 0.7, 5e-5, 2e-2))


def trapezoid(n):
    X, Y = W.trapezoid_grid(n, n)
    return dict(grid="curvilinear", x=X, y=Y)


@pytest.mark.parametrize("count,kernel,grid,limit", [
    (48, "march_rolled", lambda n: {}, 100e-6),
    (128, "tile", trapezoid, 360e-6),
])
def test_set_active_is_cheap(count, kernel, grid, limit):
    sides = [(65, 129, 257, 513)[i % 4] for i in range(count)]
    batch = mdf.Batch([dict(nx=n, ny=n, **LID, **grid(n)) for n in sides])
    batch.set_launch(kernel)
    batch.step(2)
    torch.cuda.synchronize()
    best = 1.0
    for k in range(12):
        t0 = time.perf_counter()
        batch.set_active(k // 2, k % 2 == 1)
        best = min(best, time.perf_counter() - t0)
    assert best < limit
