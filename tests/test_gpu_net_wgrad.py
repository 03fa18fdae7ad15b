"""The tcgen05 weight- and bias-gradient kernel against the mma.sync kernel.

The forward pass and the input gradients of the two kernels are equal to the
bit, so the parameter gradients differ only by the order in which FP32 adds the
same BF16 products: chains of at most 16 tensor-core steps, each dropping less
than 2^-23 of the partial sum, then rounded additions (2^-24).  A partial sum
of random products stays near the size of the result, so the difference is a
few 1e-7 of it; 2e-6 leaves room for cancellation in small layers, while one
wrong tap, image row or halo pixel shows at 1e-2 and more."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import net_oracle as N  # noqa: E402
from paper_2306_08216_gb300 import warmstart  # noqa: E402
from paper_2306_08216_gb300 import workloads as W  # noqa: E402


@pytest.mark.parametrize("R,batch", [
    (8, 5),    # 8 x 8: four images to a tile, the last tile ragged; 4 x 4 and below on mma.sync
    (16, 1),   # a whole image per tile
    (64, 3),   # tiles of 32 x 8, layers down to 8 x 8 with a ragged tile
    (128, 2),  # 32 x 8 tiles at several columns and rows, fewer tiles than SMs on the small layers
])
def test_weight_gradient_equals_mma_sync(R, batch):
    rng = np.random.default_rng(R + batch)
    p = W.net_init_params(N.layer_shapes(), 3, out_gain=1.0)
    x = rng.standard_normal((batch, W.WARM_IN_PLANES, R, R)).astype(np.float32)
    t = rng.standard_normal((batch, 3, R, R)).astype(np.float32)
    net = warmstart.Net(R, batch)
    net.set_params(p)
    g = {}
    for kind in ("tcgen05", "mma.sync"):
        net.set_conv_kernel(kind)
        g[kind] = net.gradient(x, t)[1].astype(np.float64)
    k = 0
    for name, co, ci in N.layer_shapes():
        for part, n in (("weights", co * 9 * ci), ("bias", co)):
            a, b = g["tcgen05"][k:k + n], g["mma.sync"][k:k + n]
            k += n
            rel = float(np.linalg.norm(a - b) / np.linalg.norm(b))
            assert rel <= 2e-6, (name, part, rel)
