"""The network at the ends of its sizes and values."""
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
