"""Reading the state: four columns per thread where the rows are multiples of
four and the destination is aligned to 16 bytes, one column otherwise; both are
copies, so every value is the same to the bit."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2306_08216_gb300 import mdf  # noqa: E402
from paper_2306_08216_gb300 import workloads as W  # noqa: E402


@pytest.mark.parametrize("walls", [(False, False), (True, True)])
@pytest.mark.parametrize("nx,ny", [(5, 6), (64, 9), (65, 33), (66, 7), (260, 130)])
def test_state_to_any_address(nx, ny, walls):
    s = mdf.Solver(nx, ny, nu=0.01, walls=walls)
    s.init(*W.random_fields(nx, ny, 0.02, seed=nx))
    s.step(3)
    host = s.state()
    n = 10 * nx * ny
    for shift in (0, 1, 2):
        buf = torch.full((n + 8,), 7.0, device="cuda")
        s.state(out=buf[shift:shift + n].view(2, 5, ny, nx))
        s.synchronize()
        got = buf.cpu().numpy()
        np.testing.assert_array_equal(got[shift:shift + n].reshape(2, 5, ny, nx), host)
        assert (got[:shift] == 7.0).all() and (got[shift + n:] == 7.0).all()
    t = mdf.Solver(nx, ny, nu=0.01, walls=walls)
    t.set_state(host)
    np.testing.assert_array_equal(t.state(), host)
