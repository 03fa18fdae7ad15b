"""Batches with more than two work items per block (blocks take the further
items from a queue), with and without a force, against the same problems alone:
equal bits, also on the launches after the first, which find the queue as the
launch before left it."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2306_08216_gb300 import mdf  # noqa: E402
from paper_2306_08216_gb300 import workloads as W  # noqa: E402


def problem(kind, i):
    nx, ny = 1001 - 7 * i, 900 + 11 * i
    kw = dict(nx=nx, ny=ny, walls=(kind != "channel", True))
    if kind == "channel":
        return dict(kw, nu=1e-2)
    return dict(kw, u_wall=(0, 0, 0, 0.1), power_law=(1e-3, 0.6 + 0.05 * i, 5e-5, 2e-2))


@pytest.mark.parametrize("kind,kernel", [("channel", "march"), ("cavity", "march"), ("cavity", "march_rolled")])
def test_queued_items_equal_solo_runs_bitwise(kind, kernel):
    probs = [problem(kind, i) for i in range(22)]
    batch = mdf.Batch(probs)
    batch.set_launch(kernel)
    info = batch.info()
    assert info["work_items"] > 2 * info["blocks"]
    force = [(1e-3 * (i % 3), 0.0) if kind == "channel" else None for i in range(len(probs))]
    for i, f in enumerate(force):
        batch.problem(i).set_force(f)
    batch.step(17)  # one graph replay and a launch
    batch.step(2)
    batch.set_active(7, False)
    batch.step(3)
    for i in (0, 7, 13, 21):
        kw = dict(probs[i])
        nx, ny = kw.pop("nx"), kw.pop("ny")
        solo = mdf.Solver(nx, ny, **kw)
        solo.set_launch(128, 64)
        solo.init(*W.zeros(nx, ny))
        solo.set_force(force[i])
        solo.step(19 if i == 7 else 22)
        np.testing.assert_array_equal(batch.problem(i).state(), solo.state())
