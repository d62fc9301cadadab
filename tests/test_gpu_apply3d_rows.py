"""The 3D apply with FP32 vectors (one thread per staged position) at sizes around
its units: a pitch of exactly one and two tiles, an odd number of tile rows, one
plane past a tile layer, and whole-grid launches of units 4, 8 and 16 planes deep.
Against the oracle's matrix where that is small, else against the FP64 apply
(another kernel)."""
import numpy as np
import pytest

from gpu_common import abs_matvec, gpu_apply_fields, gpu_context, oracle_system, require_gpu
from paper_1010_2832_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

# Norms of the error against that of |A||x|.  FP32: a term is rounded at most 16
# times on its way (staged product, face, gather): 16 x 2^-24 = 9.5e-7.  BF16: three
# coefficients, each within 2^-9: 5.9e-3.
TOL = {1: 9.5e-7, 2: 5.9e-3}


@pytest.mark.parametrize("prec", [1, 2])
@pytest.mark.parametrize("n", [(29, 13, 5), (30, 5, 13), (61, 10, 9), (9, 6, 46), (62, 2, 2)])
def test_small_grids_match_the_matrix(n, prec):
    require_gpu()
    wl = W.random_small(n, seed=sum(n), dim=3)
    S, ctx = oracle_system(wl), gpu_context(wl)[0]
    x = np.random.default_rng(1).normal(size=S.A.shape[0]).astype(np.float32).astype(np.float64)
    y = gpu_apply_fields(ctx, x, prec)
    assert np.linalg.norm(y - S.A @ x) <= TOL[prec] * np.linalg.norm(abs_matvec(S.A, x))


@pytest.mark.parametrize("n", [(62, 41, 33), (93, 93, 121), (94, 90, 297)])
def test_units_of_every_depth_match_fp64(n):
    require_gpu()
    wl = W.random_small(n, seed=sum(n), dim=3)
    ctx = gpu_context(wl)[0]
    N = sum(ctx_field_sizes(n))
    x = np.random.default_rng(2).normal(size=N).astype(np.float32).astype(np.float64)
    y64 = gpu_apply_fields(ctx, x, 0)
    # |A||x| is at least |Ax|; the FP64 apply's own error is far below
    assert np.linalg.norm(gpu_apply_fields(ctx, x, 1) - y64) <= 16 * TOL[1] * np.linalg.norm(y64)


def ctx_field_sizes(n):
    nx, ny, nz = n
    c = nx * ny * nz
    return [c, c, (nx + 1) * (ny + 1) * nz, (nx + 1) * ny * (nz + 1), nx * (ny + 1) * (nz + 1), c]
