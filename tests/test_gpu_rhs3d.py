"""3D right-hand side: slots without an active unknown are left at zero, but a
u* that is not finite anywhere still reaches every row whose stencil holds its
face (0 times NaN is NaN), as in the full evaluation."""
import numpy as np
import pytest

from gpu_common import require_gpu
from paper_1010_2832_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("value", [float("nan"), float("inf"), 1e300])
@pytest.mark.parametrize("where", ["air", "wall"])
def test_non_finite_velocity_reaches_its_rows(value, where):
    require_gpu()
    from paper_1010_2832_gb300 import stokes
    wl = W.random_small((34, 11, 6), seed=2, dim=3)
    ctx, dev = stokes.context_for(wl)
    base = ctx.new_vector()
    ctx.rhs(dev["u_star"], base)
    act = ctx.export(3).cpu().numpy()
    nx, ny, nz = wl.n
    cells = act[:nx * ny * nz].reshape(nz, ny, nx)
    if where == "wall":
        i, j, k = 0, ny // 2, nz // 2
    else:
        # a u face whose cells and their neighbours are all inactive
        ok = [(i, j, k) for k in range(1, nz - 1) for j in range(1, ny - 1) for i in range(2, nx - 1)
              if np.all(cells[k - 1:k + 2, j - 1:j + 2, i - 2:i + 2] == 0)]
        i, j, k = ok[len(ok) // 2]
    us = [t.clone() for t in dev["u_star"]]
    us[0].view(nz, ny, nx + 1)[k, j, i] = value
    b = ctx.new_vector()
    ctx.rhs(us, b)
    lay = ctx.layout
    at = lambda f, i, j, k: f * lay.field_stride + lay.base + ((k + 1) * lay.rows + j + 1) * lay.pitch + i + 1
    # rows that hold u(i, j, k): tau_xx and p of both cells, tau_xy below and above, tau_xz before and behind
    rows = [at(f, ii, j, k) for f in (0, 5) for ii in (i - 1, i) if ii >= 0]
    rows += [at(2, i, j, k), at(2, i, j + 1, k), at(3, i, j, k), at(3, i, j, k + 1)]
    got, ref = b.cpu().numpy(), base.cpu().numpy()
    other = np.ones(got.size, bool)
    other[rows] = False
    assert np.array_equal(got[other], ref[other])
    if not np.isfinite(value):
        assert not np.isfinite(got[rows]).any()
    ctx.close()
