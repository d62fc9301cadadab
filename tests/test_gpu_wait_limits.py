"""The bounded waits of the one-kernel CG loops and of the batch's grid barrier, run out with the options' test
hook (the CTAs' edge values, or one group of patches' answers, are held back and
the others give up after 1,024 polls): the call returns STOKES_ERR_TIMEOUT,
whichever CTA gave up and whichever held the scalars, and the same context then
solves as a fresh one does.  With few CTAs each forms the totals itself, with more
than 64 the reducer CTA does."""
import numpy as np
import pytest

from gpu_common import require_gpu
from paper_1010_2832_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _sheets(n=256, count=5):
    """Thin vertical liquid sheets, one per column of tiles: many tiles with few
    patches each (155 tiles: 78 tile CTAs of the Schwarz loop and its reducer)."""
    h = 1.0 / n
    xc = [(32 * k + 16) * h for k in range(count)]
    rng = np.random.default_rng(17)

    def phi(X):
        d = np.min([np.abs(X[0] - c) for c in xc], axis=0) - 1.6 * h
        return np.maximum(d, np.abs(X[1] - 0.5) - 0.48)
    return W.from_functions("sheets", 2, (n, n), h, 0.01, (0.0, 0.0), phi,
                            lambda X: W.box_phi(X, (0.0, 0.0), (1.0, 1.0)), lambda P: 1.0, lambda P: 1.0,
                            lambda d, P: 0.0, lambda d, P: rng.uniform(-1.0, 1.0, P[0].shape))


CASES = {
    "disk32": lambda: W.disk_in_box(32),                                # 4 tiles
    "bumps96": lambda: W.bumps_2d(96, seed=21),                         # 22 tiles, FP64: 88 CTAs and the reducer
    "bumps224": lambda: W.bumps_2d(224, seed=5, rho_split=False),       # 85 tiles
    "sheets256": _sheets,
}


def _system(name):
    require_gpu()
    from paper_1010_2832_gb300 import stokes
    ctx, dev = stokes.context_for(CASES[name](), min_face_liquid=0.01)
    b = ctx.new_vector()
    ctx.rhs(dev["u_star"], b)
    return ctx, b


def _solve(ctx, b, **kw):
    from paper_1010_2832_gb300 import stokes
    x = ctx.new_vector()
    st = ctx.solve_system(b, x, stokes.default_options(**kw))
    return st, x


@pytest.mark.parametrize("name,kw", [
    ("disk32", dict(mode=0)), ("disk32", dict(mode=1)), ("bumps96", dict(mode=0)), ("bumps96", dict(mode=2)),
    ("bumps224", dict(mode=0)), ("bumps224", dict(mode=1)),
    ("disk32", dict(mode=1, precond=2)), ("bumps96", dict(mode=1, precond=2)), ("sheets256", dict(mode=1, precond=2)),
    ("bumps96", dict(mode=1, precond=2, use_graph=0)),                  # the separate kernels' copy wait
])
def test_waits_run_out_and_the_context_stays_usable(name, kw):
    from paper_1010_2832_gb300 import stokes
    ctx, b = _system(name)
    for _ in range(3):
        with pytest.raises(stokes.StokesError) as e:
            _solve(ctx, b, wait_test=1, **kw)
        assert e.value.status == -5
    st, x = _solve(ctx, b, tol=1e-9, **kw)
    fresh, b2 = _system(name)
    st2, x2 = _solve(fresh, b2, tol=1e-9, **kw)
    assert (st.status, st.iterations) == (0, st2.iterations)
    assert torch.equal(x, x2)
    ctx.close()
    fresh.close()


def test_schwarz_loop_with_a_reducer_matches_separate_kernels():
    ctx, b = _system("sheets256")
    assert ctx.active_tiles() > 128
    for kw in (dict(tol=1e-10), dict(tol=1e-8, max_iter=5)):
        st, x = _solve(ctx, b, mode=1, precond=2, **kw)
        st2, x2 = _solve(ctx, b, mode=1, precond=2, use_graph=0, check_every=2, **kw)
        assert (st.status, st.iterations, st.outer) == (st2.status, st2.iterations, st2.outer)
        assert torch.equal(x, x2)
    ctx.close()


@pytest.mark.parametrize("precond", [0, 2])
def test_batch_barrier_runs_out(precond):
    """A batch whose barrier misses one arrival: STOKES_ERR_TIMEOUT, and the
    contexts then solve in another batch as fresh ones do."""
    require_gpu()
    from paper_1010_2832_gb300 import stokes
    wls = [W.disk_in_box(32), W.bumps_2d(96, seed=21)]

    def make(ctxs, **kw):
        return stokes.Batch(ctxs, stokes.default_options(mode=0, precond=precond, tol=1e-8, max_iter=3, **kw))

    def run(batch, dev):
        out = [([torch.zeros_like(t) for t in d["u_star"]],
                [torch.zeros(w.n[0] * w.n[1], dtype=torch.float64, device="cuda"),
                 torch.zeros((w.n[0] + 1) * (w.n[1] + 1), dtype=torch.float64, device="cuda")],
                torch.zeros(w.n[0] * w.n[1], dtype=torch.float64, device="cuda")) for w, d in zip(wls, dev)]
        st, _ = batch.solve([d["u_star"] for d in dev], [o[0] for o in out], [o[1] for o in out], [o[2] for o in out])
        return [(s["status"], s["iterations"]) for s in st]
    pairs = [stokes.context_for(w, min_face_liquid=0.01) for w in wls]
    ctxs, dev = [p[0] for p in pairs], [p[1] for p in pairs]
    held = make(ctxs, wait_test=1)
    for _ in range(2):
        with pytest.raises(stokes.StokesError) as e:
            run(held, dev)
        assert e.value.status == -5
    del held
    assert run(make(ctxs), dev) == [(-3, 3), (-3, 3)]
