"""The network at the ends of its sizes and values."""
import math

import numpy as np
import pytest

from gpu_common import require_gpu
from oracle import unet as U

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def test_wide_grid_is_addressed_in_64_bits():
    """A 2D grid of 20 x 8,454,144 voxels with 16 channels: the rows of one
    tile's halo lie more than 2^31 elements apart.  The input is zero but for the
    last 128 columns, so the last 64 of the output (the network sees fewer than
    32 columns to each side) are those of a grid of these 128 columns alone, bit for
    bit."""
    require_gpu()
    from paper_1010_2832_gb300 import stokes
    H, W, w, cin, cout = 20, 8454144, 128, 16, 4
    assert W % 16 == 0 and 16 * W * cin > 2 ** 31
    if torch.cuda.mem_get_info()[0] < 100e9:
        pytest.skip("needs 80 GB of device memory")
    th = U.init_params(2, cin, cout, seed=9)
    g = torch.Generator().manual_seed(9)
    tail = torch.randn(H, w, cin, generator=g).cuda()
    small = stokes.Net(2, cin, cout, H * w)
    small.set_params(small.from_oracle_layout(th))
    want = small.forward(tail.reshape(-1), (1, 1, H, w)).view(H, w, cout)
    small.close()
    net = stokes.Net(2, cin, cout, H * W)
    net.set_params(net.from_oracle_layout(th))
    x = torch.zeros(H, W, cin, dtype=torch.float32, device="cuda")
    x[:, W - w:] = tail
    got = net.forward(x.view(-1), (1, 1, H, W)).view(H, W, cout)
    net.close()
    assert torch.equal(got[:, W - 64:], want[:, w - 64:])
    del x, got
    torch.cuda.empty_cache()


@pytest.mark.parametrize("scale", [1.0, 1e-22, 1e-24, 1e20, 1e30, "mixed"])
@pytest.mark.parametrize("dim,shape", [(2, (2, 1, 12, 20)), (3, (3, 8, 8, 12))])
def test_loss_of_small_and_large_targets(dim, shape, scale):
    """A network of zeros answers 0: the loss is 1 per sample whatever the target's
    scale, 0 for a sample whose target is zero, and of the parameter gradients
    only the output biases' are not 0: the sums over the voxels of
    -2 y / (||y||^2 B) in BF16 (FP32 sums of terms of one sign in chains of fewer than
    100 additions, 6e-6, and one term in 256 whose rounding to BF16 may go the other
    way by the last bit of FP32, 1e-5: 2e-5 together)."""
    require_gpu()
    from paper_1010_2832_gb300 import stokes
    B, D, H, W = shape
    cin, cout, n = 4, 8, D * H * W
    rng = np.random.default_rng(7)
    y = rng.uniform(0.5, 1.5, (B, n, cout))
    y *= np.where(rng.random(y.shape) < 0.5, 1e-30, 1.0) if scale == "mixed" else scale
    y = y.astype(np.float32)
    y[-1] = 0.0
    net = stokes.Net(dim, cin, cout, B * n)
    net.set_params(np.zeros(net.n, dtype=np.float32))
    x = torch.zeros(B * n * cin, dtype=torch.float32, device="cuda")
    loss, g = net.gradient(x, torch.from_numpy(y.reshape(-1)).cuda(), shape)
    assert abs(loss - (B - 1) / B) <= 4 * np.finfo(float).eps
    want = np.zeros(cout)
    for b in range(B - 1):
        den = math.fsum((y[b].astype(np.float64) ** 2).ravel())
        t = torch.from_numpy((-2.0 * y[b].astype(np.float64) / den / B).astype(np.float32)).to(torch.bfloat16)
        want += t.to(torch.float64).sum(0).numpy()
    _, co, _, _, bo = net.layers()[-1]
    assert co == cout
    assert np.all(np.abs(g[bo:bo + co] - want) <= 2e-5 * np.abs(want))
    rest = np.delete(g, np.arange(bo, bo + co))
    assert not rest.any()
    net.close()


def test_loss_is_as_accurate_as_fp64():
    """Random output and target: the loss within the roundings of FP64 sums (the
    two sums and their quotient: fewer than 20 roundings of 2^-53 each)."""
    require_gpu()
    from paper_1010_2832_gb300 import stokes
    shape, cin, cout = (1, 16, 16, 20), 4, 8
    rng = np.random.default_rng(8)
    n = 16 * 16 * 20
    net = stokes.Net(3, cin, cout, n)
    net.set_params(net.from_oracle_layout(U.init_params(3, cin, cout, seed=8)))
    x = torch.from_numpy(rng.normal(size=n * cin).astype(np.float32)).cuda()
    out = net.forward(x, shape).cpu().numpy()
    y = (rng.normal(size=n * cout) * np.exp(3 * rng.normal(size=n * cout))).astype(np.float32)
    loss, _ = net.gradient(x, torch.from_numpy(y).cuda(), shape)
    d = (out - y).astype(np.float64)
    want = math.fsum(d * d) / math.fsum(y.astype(np.float64) ** 2)
    assert abs(loss - want) <= 20 * 2.0 ** -53 * want
    net.close()


def test_infinite_target_is_not_taken_as_a_zero_target():
    """One infinite target value: inf / inf, so loss and gradient are NaN."""
    require_gpu()
    from paper_1010_2832_gb300 import stokes
    shape, cin, cout = (1, 1, 8, 8), 4, 4
    net = stokes.Net(2, cin, cout, 64)
    net.set_params(np.zeros(net.n, dtype=np.float32))
    y = torch.ones(64 * cout, dtype=torch.float32, device="cuda")
    y[5] = float("inf")
    loss, g = net.gradient(torch.zeros(64 * cin, dtype=torch.float32, device="cuda"), y, shape)
    assert math.isnan(loss)
    assert np.isnan(g[net.layers()[-1][4] + 1])
    net.close()
