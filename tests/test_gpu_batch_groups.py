"""The batched kernel's split of a CTA: tiles of 4 rows and Schwarz patches are
taken by halves of a CTA.  The sums' order belongs to the tile height alone, so
with one plan the solution has the same bits for any number of CTAs; it solves
the oracle's systems to the bound the batch's other tests hold it to.  An
instance that breaks down while its neighbours iterate ends alone."""
import numpy as np
import pytest

from gpu_common import gpu_context, oracle_system, require_gpu
from oracle import solve as So
from paper_1010_2832_gb300 import workloads as W
from test_gpu_batched import _outputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _solve(wls, precond, plan, tmp_path, scale=None):
    from paper_1010_2832_gb300 import stokes
    path = tmp_path / "plan.txt"
    ctxs, devs = zip(*[gpu_context(wl) for wl in wls])
    opt = stokes.default_options(mode=0, tol=1e-11, precond=precond)
    stokes.Batch(ctxs, opt, tune_cache=str(path)).close()
    key = path.read_text().splitlines()[-1].split()[0]
    path.write_text(f"{key} {plan[0]} {plan[1]} 1.0\n")
    b = stokes.Batch(ctxs, opt, tune_cache=str(path))
    assert (b.tuning()["tile_rows"], b.tuning()["ctas_per_sm"]) == plan
    if scale:
        for d, s in zip(devs, scale):
            d["u_star"] = [u * s for u in d["u_star"]]
    outs = [_outputs(wl) for wl in wls]
    err = None
    try:
        stats, _ = b.solve([d["u_star"] for d in devs], [o[0] for o in outs], [o[1] for o in outs], [o[2] for o in outs])
        assert [s["status"] for s in stats] == [0] * len(wls), stats
    except stokes.StokesError as e:
        err = e
    b.close()
    return [torch.cat(t + [p]).cpu().numpy() for _, t, p in outs], err


@pytest.mark.parametrize("precond", [0, 2])
@pytest.mark.parametrize("rows", [4, 8, 16])
@pytest.mark.parametrize("sizes", [[17], [24, 90, 33, 127, 64, 17]])
def test_same_bits_for_any_number_of_ctas(sizes, rows, precond, tmp_path):
    require_gpu()
    wls = [W.bumps_2d(n, seed=140 + i, rho_split=False, disk_r=0.05 + 0.02 * i) for i, n in enumerate(sizes)]
    (one, e1), (two, e2) = (_solve(wls, precond, (rows, c), tmp_path) for c in (1, 2))
    assert e1 is None and e2 is None
    for wl, a, b in zip(wls, one, two):
        S = oracle_system(wl)
        assert So.relative_residual(S.A, a, S.b) <= 1e-10
        assert np.array_equal(a, b)


def test_a_breakdown_leaves_the_others_alone(tmp_path):
    """Right-hand sides whose squares underflow: r.r is 0 (nothing to do), or it is
    not and p.Ap is (a breakdown in the apply's phase), whichever the scale gives."""
    require_gpu()
    wls = [W.bumps_2d(24, seed=140, rho_split=False, disk_r=0.05) for _ in range(10)]
    plain, _ = _solve(wls[:1], 0, (4, 1), tmp_path)
    for last in ([], [1.0]):                     # with and without an instance that iterates on
        scale = [10.0 ** -e for e in range(156, 165)] + last
        out, err = _solve(wls[:len(scale)], 0, (4, 1), tmp_path, scale)
        assert err is None or err.status in (-4, -7), err      # breakdown, non-finite
        if last:
            assert np.array_equal(out[-1], plain[0])
