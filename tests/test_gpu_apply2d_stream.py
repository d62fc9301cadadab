"""The streaming 2D apply of large whole grids (strips of 120 columns, one wave of
warps) against the one-slot-per-thread kernel, which vectors off a 16-byte
boundary take: pitches that are a whole number of strips and one tile more, the
last chunk of rows short, single-precision and BF16 coefficients, and a grid large
enough for chunks of more than eight rows.  The kernels may fuse an entry's two
sums of products differently, each within 2^-24 of a term, so the difference stays
below 16 x 2^-24 of the result in norm; non-finite entries spread alike."""
import pytest

from gpu_common import gpu_context, require_gpu
from paper_1010_2832_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n", [(957, 900), (958, 901), (837, 997), (1500, 1450)])
def test_strips_match_the_slot_kernel(n):
    require_gpu()
    ctx = gpu_context(W.random_small(n, seed=sum(n)))[0]
    g = torch.Generator(device="cuda").manual_seed(3)
    x = ctx.new_vector(torch.float32)
    x.copy_(torch.randn(x.shape, device="cuda", generator=g))
    m = x.numel()
    for prec in (1, 2):
        for bad in (None, float("inf"), float("nan")):
            if bad is not None:
                x[m // 2 + 12345] = bad
            xb = torch.zeros(m + 4, dtype=torch.float32, device="cuda")
            yb, y = torch.zeros_like(xb), ctx.new_vector(torch.float32)
            xb[1:m + 1].copy_(x)
            ctx.apply(xb[1:m + 1], yb[1:m + 1], prec)
            ctx.apply(x, y, prec)
            a, b = (ctx.slots_to_fields(v.to(torch.float64)) for v in (y, yb[1:m + 1].contiguous()))
            fin = torch.isfinite(b)
            assert torch.equal(torch.isfinite(a), fin) and torch.equal(torch.isnan(a), torch.isnan(b))
            assert torch.linalg.norm((a - b)[fin]) <= 16 * 2.0 ** -24 * torch.linalg.norm(b[fin])
