"""launch_info of the tile plans: the shared memory and the resident blocks are
those of the tile that runs.  A block holds five pairs of FP32 of every node of its
tile with a halo of 4 and again with a halo of 2, and two rates of the latter for
a power law."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2306_08216_gb300 import mdf  # noqa: E402


@pytest.mark.parametrize("side,threads", [(8, 256), (16, 288)])
@pytest.mark.parametrize("power_law", [None, (1e-3, 0.7, 5e-5, 2e-2)])
def test_tile_plans(side, threads, power_law):
    s = mdf.Solver(64, 50, nu=1e-3, walls=(True, True), u_wall=(0, 0, 0, 0.1), power_law=power_law)
    s.set_launch(0, side)
    info = s.launch_info()
    smem = 40 * (side + 8) ** 2 + (40 + (8 if power_law else 0)) * (side + 4) ** 2
    assert (info["kernel"], info["threads"], info["rows_per_block"], info["smem_bytes"]) == ("tile", threads, side, smem)
    assert (info["grid_x"], info["grid_y"]) == (-(-64 // side), -(-50 // side))
    props = torch.cuda.get_device_properties(0)
    limit = min(props.max_threads_per_multi_processor // threads, 228 * 1024 // (smem + 1024))
    assert 3 <= info["blocks_per_sm"] <= limit
