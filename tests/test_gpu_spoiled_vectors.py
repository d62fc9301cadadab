"""A solve that ends in infinities leaves them in the context's vectors; a later
geometry with fewer tiles reads some of them as the halo of its own, where their
weights are zero.  The next solves must be those of a fresh context.  Likewise
what a caller's solution array held before the call."""
import numpy as np
import pytest

from gpu_common import require_gpu
from paper_1010_2832_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

N, H = 96, 100.0


def _box(rho, left=0):
    """Liquid from face column `left` on.  At 31 the liquid begins on the edge of a
    column of tiles: the live faces there join cells of both columns, and the left
    ones are inactive.  rho scales the pressure's diagonal, K a^2 = 1e-6 / rho."""
    rng = np.random.default_rng(23)
    L = N * H
    return W.from_functions("box", 2, (N, N), H, 0.01, (0.0, 0.0),
                            lambda X: np.maximum(left * H - X[0], np.abs(X[1] - 0.5 * L) - 0.3 * L) if left
                            else -np.ones(X[0].shape),
                            lambda X: W.box_phi(X, (0.0, 0.0), (L, L)), lambda P: rho, lambda P: 1.0,
                            lambda d, P: 0.0, lambda d, P: rng.uniform(-1.0, 1.0, P[0].shape))


def _build(ctx, wl):
    from paper_1010_2832_gb300 import stokes
    d = stokes.upload_workload(wl)
    ctx.build_weights(d["phi_liquid"], d["phi_solid"], d["rho"], d["mu"], d["u_bc"])
    return d


def _step(ctx, d, **kw):
    from paper_1010_2832_gb300 import stokes
    u = [torch.zeros_like(t) for t in d["u_star"]]
    tau = [torch.zeros(N * N, dtype=torch.float64, device="cuda"),
           torch.zeros((N + 1) ** 2, dtype=torch.float64, device="cuda")]
    p = torch.zeros(N * N, dtype=torch.float64, device="cuda")
    st = ctx.solve_step(d["u_star"], u, tau, p, stokes.default_options(**kw))
    return st, u + tau + [p]


# the inverse of 1e-6 / rho passes the range of FP32, or of FP64
@pytest.mark.parametrize("mode,rho", [(1, 1e36), (0, 1e308)])
@pytest.mark.parametrize("use_graph", [0, 1])
def test_solve_after_a_spoiled_one(mode, rho, use_graph):
    require_gpu()
    from paper_1010_2832_gb300 import stokes
    bad, good = _box(rho), _box(1.0, left=31)
    ctx = stokes.StokesContext(2, bad.n, bad.h, bad.dt, bad.origin)
    kw = dict(mode=mode, tol=1e-10, use_graph=use_graph)
    try:
        st, _ = _step(ctx, _build(ctx, bad), max_iter=50, **kw)
        assert st.precision_used != mode                 # FP32 overflowed and FP64 went on
    except stokes.StokesError as e:
        assert mode == 0 and e.status == -7
    st, out = _step(ctx, _build(ctx, good), **kw)
    fresh = stokes.StokesContext(2, good.n, good.h, good.dt, good.origin)
    st2, out2 = _step(fresh, _build(fresh, good), **kw)
    assert st2.status == 0 and st2.precision_used == mode
    assert (st.status, st.iterations, st.precision_used) == (0, st2.iterations, mode)
    assert all(torch.equal(a, b) for a, b in zip(out, out2))
    ctx.close()
    fresh.close()


@pytest.mark.parametrize("mode", [0, 1])
def test_solution_array_may_hold_anything(mode):
    require_gpu()
    from paper_1010_2832_gb300 import stokes
    wl = _box(1.0, left=31)
    ctx = stokes.StokesContext(2, wl.n, wl.h, wl.dt, wl.origin)
    d = _build(ctx, wl)
    b = ctx.new_vector()
    ctx.rhs(d["u_star"], b)
    want, x = ctx.new_vector(), torch.full_like(b, float("nan"))
    for y in (want, x):
        st = ctx.solve_system(b, y, stokes.default_options(mode=mode, tol=1e-10))
        assert (st.status, st.precision_used) == (0, mode)
    assert torch.equal(x, want)
    ctx.close()
