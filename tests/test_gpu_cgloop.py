"""The one-kernel CG loops of small 2D systems (Jacobi, and Schwarz with its
resident patch factors) against the same solve launched
kernel by kernel (use_graph = 0): the arithmetic and the order of every sum are
the same, so iterates, iteration counts and statuses agree bit for bit.  Sizes:
few CTAs (each forms the totals itself), more than 64 (the reducer CTA), FP64
with two and four rows per CTA, the largest that the loop takes, and one past
it; ragged sides, interfaces, moving solids."""
import numpy as np
import pytest

from gpu_common import require_gpu
from paper_1010_2832_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

CASES = {
    "one_tile": lambda: W.random_small((7, 5), seed=3),
    "disk32": lambda: W.disk_in_box(32),
    "ragged": lambda: W.random_small((61, 45), seed=8),
    "bumps96": lambda: W.bumps_2d(96, seed=21),
    "bumps224": lambda: W.bumps_2d(224, seed=5, rho_split=False),
    "box180": lambda: W.full_box(180, 2),           # 138 tiles
    "box272": lambda: W.full_box(272, 2),           # 315 tiles: past the loop
}
_ctx = {}


def _system(name):
    require_gpu()
    if name not in _ctx:
        from paper_1010_2832_gb300 import stokes
        wl = CASES[name]()
        ctx, dev = stokes.context_for(wl, min_face_liquid=0.01)
        b = ctx.new_vector()
        ctx.rhs(dev["u_star"], b)
        _ctx[name] = (ctx, b)
    return _ctx[name]


def _solve(ctx, b, **kw):
    from paper_1010_2832_gb300 import stokes
    x = ctx.new_vector()
    st = ctx.solve_system(b, x, stokes.default_options(**kw))
    return st, x


@pytest.mark.parametrize("mode", [0, 1, 2])
@pytest.mark.parametrize("name", list(CASES))
def test_loop_matches_separate_kernels(name, mode):
    ctx, b = _system(name)
    for kw in (dict(tol=1e-8), dict(tol=1e-8, max_iter=7)):
        st, x = _solve(ctx, b, mode=mode, **kw)
        st2, x2 = _solve(ctx, b, mode=mode, use_graph=0, check_every=2, **kw)
        assert (st.status, st.iterations, st.outer) == (st2.status, st2.iterations, st2.outer)
        assert st.rel_residual == st2.rel_residual
        assert torch.equal(x, x2)
        st3, x3 = _solve(ctx, b, mode=mode, **kw)               # and again on the same context
        assert torch.equal(x, x3) and st3.iterations == st.iterations


SCHWARZ = dict(CASES,
               bumps160=lambda: W.bumps_2d(160, seed=5, rho_split=False),   # two patches per group
               box96=lambda: W.full_box(96, 2),                             # 625 patches
               box150=lambda: W.full_box(150, 2),                           # 1,444 patches, three per group
               strip=lambda: W.random_small((301, 9), seed=4))


@pytest.mark.parametrize("name", list(SCHWARZ))
def test_schwarz_loop_matches_separate_kernels(name):
    CASES.update(SCHWARZ)
    ctx, b = _system(name)
    for kw in (dict(tol=1e-10), dict(tol=1e-8, max_iter=5), dict(tol=1e-30, max_iter=60, max_outer=1, inner_tol=1e-30)):
        st, x = _solve(ctx, b, mode=1, precond=2, **kw)
        st2, x2 = _solve(ctx, b, mode=1, precond=2, use_graph=0, check_every=2, **kw)
        assert (st.status, st.iterations, st.outer) == (st2.status, st2.iterations, st2.outer)
        assert st.rel_residual == st2.rel_residual
        assert torch.equal(x, x2)


@pytest.mark.parametrize("mode", [0, 1])
def test_loop_rows_of_the_identity(mode):
    """A right-hand side on inactive unknowns of active tiles: their rows are
    the identity, so x = b there."""
    ctx, b0 = _system("ragged")
    act = ctx.export(3)
    b = ctx.fields_to_slots(torch.where(act.bool(), 0.0, 1.0).to(torch.float64)) * 0.25 + b0
    st, x = _solve(ctx, b, mode=mode, tol=1e-10)
    st2, x2 = _solve(ctx, b, mode=mode, tol=1e-10, use_graph=0, check_every=2)
    assert st.status == st2.status and st.iterations == st2.iterations and torch.equal(x, x2)


def test_loop_reports_non_finite_and_stays_usable():
    from paper_1010_2832_gb300 import stokes
    ctx, b = _system("disk32")
    bad = b.clone()
    bad[int(torch.argmax(bad.abs()))] = float("nan")
    for mode in (0, 1):
        x = ctx.new_vector()
        with pytest.raises(stokes.StokesError) as e:
            ctx.solve_system(bad, x, stokes.default_options(mode=mode))
        assert e.value.status == -7
        st, x = _solve(ctx, b, mode=mode, tol=1e-9)
        assert st.status == 0


def test_two_contexts_on_two_streams():
    """Loops of two contexts enqueued on different streams by two threads do
    not disturb each other (each context has its own exchange slots)."""
    import threading
    from paper_1010_2832_gb300 import stokes
    require_gpu()
    wls = [W.disk_in_box(32, seed=1), W.bumps_2d(96, seed=21)]
    sys_ = []
    for wl in wls:
        s = torch.cuda.Stream()
        ctx, dev = stokes.context_for(wl, stream=s, min_face_liquid=0.01)
        torch.cuda.synchronize()
        b = ctx.new_vector()
        torch.cuda.synchronize()
        ctx.rhs(dev["u_star"], b)
        torch.cuda.synchronize()
        x = ctx.new_vector()
        torch.cuda.synchronize()
        ctx.solve_system(b, x, stokes.default_options(mode=1, tol=1e-8))
        sys_.append((ctx, dev, b, x.clone()))
    torch.cuda.synchronize()
    out = [None, None]

    def work(i):
        ctx, dev, b, ref = sys_[i]
        good = True
        for _ in range(5):
            y = torch.empty_like(ref)
            y.zero_()
            torch.cuda.synchronize()
            ctx.solve_system(b, y, stokes.default_options(mode=1, tol=1e-8))
            torch.cuda.synchronize()
            good = good and torch.equal(y, ref)
        out[i] = good
    th = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    [t.start() for t in th]
    [t.join() for t in th]
    assert out == [True, True]
