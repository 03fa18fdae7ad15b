"""The order of the sums of the weight and bias gradients.

A weight gradient is a sum of runs of consecutive pixels: one tensor-core chain a
run, one atomic addition a run.  Where the output gradient is nonzero in one or
two neighbouring runs only, the order of the atomics cannot change the result
(0 + a + b = 0 + b + a), so the tcgen05 and the mma.sync kernel are equal to the
bit exactly when they split the pixels alike and sum each run in the same order.
Targets equal to the network's own outputs give an output gradient of zero; the
nonzero pixels are put in by hand."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import net_oracle as N  # noqa: E402
from paper_2306_08216_gb300 import warmstart  # noqa: E402
from paper_2306_08216_gb300 import workloads as W  # noqa: E402

DIV = (1, 1, 2, 2, 4, 4, 8, 8, 4, 4, 2, 2, 1, 1, 1)  # resolution R / DIV of every layer


def run_pixels(P, ci, co):
    """Pixels of a run: enough blocks of 64 x 128 (output, tap x input) channels for four on every SM."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    blocks = -(-9 * max(32, ci) // 128) * -(-max(32, co) // 64)
    splits = min(-(-4 * sms // blocks), -(-P // 32))
    return 32 * -(--(-P // 32) // splits)


def make(R, batch):
    rng = np.random.default_rng(R + batch)
    net = warmstart.Net(R, batch)
    net.set_params(W.net_init_params(N.layer_shapes(), 3, out_gain=1.0))
    x = torch.from_numpy(rng.standard_normal((batch, W.WARM_IN_PLANES, R, R)).astype(np.float32)).cuda()
    o = net.forward(x)
    return net, x, o, rng


def gradients(net, x, t):
    out = {}
    for kind in ("tcgen05", "mma.sync"):
        net.set_conv_kernel(kind)
        g, k, parts = net.gradient(x, t)[1], 0, []
        for _, co, ci in N.layer_shapes():
            parts.append((g[k:k + co * 9 * ci], g[k + co * 9 * ci:k + co * 9 * ci + co]))
            k += co * 9 * ci + co
        out[kind] = parts
    return out["tcgen05"], out["mma.sync"]


@pytest.mark.parametrize("R,batch", [(8, 500), (16, 200), (64, 16), (128, 16), (256, 4), (512, 1)])
def test_runs_of_the_output_layer_are_equal_bitwise(R, batch):
    net, x, o, rng = make(R, batch)
    P = batch * R * R
    run = run_pixels(P, 32, 32)
    runs = -(-P // run)
    for first, last in ((0, run), (runs // 2 * run - run // 2, runs // 2 * run + run // 2 + 5), ((runs - 1) * run, P)):
        d = torch.zeros(P, 3)
        d[first:last] = torch.from_numpy(rng.standard_normal((last - first, 3)).astype(np.float32))
        t = (o - d.view(batch, R, R, 3).permute(0, 3, 1, 2).cuda()).contiguous()
        tc, mma = gradients(net, x, t)
        assert np.count_nonzero(tc[14][0]) >= tc[14][0].size // 3  # a last row alone has no row below it
        np.testing.assert_array_equal(tc[14][0], mma[14][0])
        # the bias: serial sums of 256 pixels, at most two of them nonzero
        lo = first - first % 256 + (256 if first % 256 else 0)
        hi = min(lo + 512, last)
        d[:lo] = 0
        d[hi:] = 0
        t = (o - d.view(batch, R, R, 3).permute(0, 3, 1, 2).cuda()).contiguous()
        dz = (float(np.float32(2.0 * (1.0 / (3.0 * P)))) * (o - t).permute(0, 2, 3, 1).reshape(P, 3)).to(torch.bfloat16)
        dz = dz[lo:hi].to(torch.float32).cpu().numpy()
        want = np.zeros(3, np.float32)
        for k in range(0, hi - lo, 256):
            want += np.cumsum(dz[k:k + 256], axis=0, dtype=np.float32)[-1]
        for g in gradients(net, x, t):
            np.testing.assert_array_equal(g[14][1], want)


@pytest.mark.parametrize("R,batch,y,x0", [(128, 16, 60, 70), (64, 16, 20, 63), (64, 3, 0, 0)])
def test_single_pixel_is_equal_bitwise_down_the_layers(R, batch, y, x0):
    """One pixel of the output, and with it a few rows of every layer on the way
    down: 32 to 256 channels, boxes of several image rows."""
    net, x, o, rng = make(R, batch)
    t = o.clone()
    t[batch // 2, :, y, x0] -= torch.from_numpy(rng.standard_normal(3).astype(np.float32)).cuda()
    tc, mma = gradients(net, x, t)
    checked, lo, hi = [], y, y
    for layer in range(14, 4, -1):
        _, co, ci = N.layer_shapes()[layer]
        r = R // DIV[layer]
        run = run_pixels(batch * r * r, ci, co)
        first, last = (batch // 2 * r + lo) * r // run, ((batch // 2 * r + hi + 1) * r - 1) // run
        if last - first <= 1:
            np.testing.assert_array_equal(tc[layer][0], mma[layer][0], err_msg=str(layer))
            checked.append(layer)
        lo, hi = max(0, lo - 1), min(r - 1, hi + 1)
        if layer in (12, 10, 8):  # through the upsampling
            lo, hi = lo // 2, hi // 2
        if layer == 6:  # layer 5 also receives the skip of layer 8: the whole image
            lo, hi = 0, R // 4 - 1
    assert {14, 13, 12, 7} <= set(checked)
