"""The network's kernels where their tiling can go wrong: one tile, partial
tiles in every direction, more tiles than CTAs fit on the device at once (the
persistent loop with its two halo buffers), inputs off a 16-byte boundary and
every supported channel count.

Forward: a selection network (every output channel copies one tap of one
input channel, sign +-1) on small integers.  Its activations stay
integers over 64 of at most 192, which BF16 and FP32 hold exactly, so the
output must equal the FP64 reference's bit for bit.

Gradient (random weights): against the FP64 reference at the BF16-rounded
weights and stored activations, whose output gradients are not rounded to
BF16 (2^-9 each, independent): a cosine of 1 - 1e-4 or more."""
import numpy as np
import pytest

from gpu_common import require_gpu
from oracle import unet as U
from test_gpu_unet import _bf16_weights, _setup

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

CASES = pytest.mark.parametrize("dim,cin,cout,shape,shift", [
    (3, 12, 8, (1, 4, 4, 4), 0),
    (3, 12, 8, (2, 12, 20, 28), 1),
    (3, 16, 16, (1, 8, 12, 8), 0),
    (3, 4, 12, (1, 8, 8, 8), 0),
    (3, 12, 8, (1, 48, 104, 72), 0),
    (2, 8, 4, (1, 1, 4, 8), 0),
    (2, 16, 12, (3, 1, 36, 20), 1),
    (2, 8, 16, (2, 1, 404, 412), 0),
])


def _up(a, shift):
    """A device copy that starts `shift` floats past an aligned address."""
    t = torch.zeros(a.size + shift, dtype=torch.float32, device="cuda")[shift:]
    return t.copy_(torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32).reshape(-1)))


def _selection(dim, cin, cout, shape):
    """Parameters (oracle layout) and input.  Half the taps are the centre;
    only the first and the last layer have negative signs (a ReLU passes the
    rest of them)."""
    rng = np.random.default_rng(5)
    th = []
    shapes = list(U.layer_shapes(dim, cin, cout))
    for i, (_, co, ci, k) in enumerate(shapes):
        W = np.zeros((co, ci, int(np.prod(k))))
        tap = np.where(rng.random(co) < 0.5, W.shape[2] // 2, rng.integers(0, W.shape[2], co))
        sign = rng.choice([-1, 1], co) if i in (0, len(shapes) - 1) else 1
        W[np.arange(co), rng.integers(0, ci, co), tap] = sign
        th += [W.reshape(-1), np.zeros(co)]
    sp = shape[1:] if dim == 3 else shape[2:]
    return np.concatenate(th), rng.integers(-3, 4, (shape[0],) + sp + (cin,)).astype(np.float32)


@CASES
def test_selection_network_is_exact(dim, cin, cout, shape, shift):
    require_gpu()
    from paper_1010_2832_gb300 import stokes
    th, x = _selection(dim, cin, cout, shape)
    net = stokes.Net(dim, cin, cout, int(np.prod(shape)))
    net.set_params(net.from_oracle_layout(th))
    got = net.forward(_up(x, shift), shape).cpu().numpy().reshape(x.shape[:-1] + (cout,))
    ref = U.predict(th, np.moveaxis(x, -1, 1).astype(np.float64), dim, cin, cout)
    assert np.array_equal(np.moveaxis(got, -1, 1), ref)


@CASES
def test_gradient_over_tiles(dim, cin, cout, shape, shift):
    require_gpu()
    net, th, x, y, to_nc = _setup(dim, cin, cout, shape, 11)
    xb = torch.tensor(x).to(torch.bfloat16).to(torch.float64).numpy()
    th_ref = _bf16_weights(net.to_oracle_layout(net.get_params()), dim, cin, cout)
    L, g = net.gradient(_up(x, shift), _up(y, shift), shape)
    g = net.to_oracle_layout(g)
    L_ref, g_ref = U.loss_and_grad(th_ref, to_nc(xb), to_nc(y), dim, cin, cout, store=U.bf16_store)
    assert abs(L - L_ref) <= 2e-3 * abs(L_ref)
    cos = g @ g_ref / (np.linalg.norm(g) * np.linalg.norm(g_ref))
    assert cos >= 0.9999, cos
    assert abs(np.linalg.norm(g) - np.linalg.norm(g_ref)) <= 1e-2 * np.linalg.norm(g_ref)
