"""The weight build's evaluation of cut control volumes against the oracle's
fractions, bit for bit (both sides round every operation separately and in the
same order).  Level sets: independent random lattice values, so that almost
every control volume is cut, with exact zeros, and values whose products
underflow, sprinkled in; sizes around the 32 x 8 slots of a CTA."""
import numpy as np
import pytest

from gpu_common import require_gpu, to_gpu
from oracle import fractions as Fr

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

OFF = {2: ((2, 2), (1, 1), (1, 2), (2, 1)),
       3: ((2, 2, 2), (1, 2, 2), (2, 1, 2), (2, 2, 1), (1, 1, 2), (1, 2, 1), (2, 1, 1))}


def _level_set(rng, n, kind):
    v = rng.normal(size=tuple(reversed([2 * m + 3 for m in n])))
    pick = rng.random(v.shape)
    if kind == "zeros":
        v[pick < 0.4] = 0.0
    elif kind == "tiny":
        v[pick < 0.3] = 0.0
        v[(pick > 0.3) & (pick < 0.6)] = -1e-120
        v[(pick > 0.6) & (pick < 0.7)] = 1e-90
    elif kind == "one_sign":
        v = np.where(pick < 0.97, -np.abs(v), 0.0)
        v[pick > 0.995] = 1.0
    return v


def _fractions(phi, n):
    out = []
    for off in OFF[len(n)]:
        axes = [2 * np.arange(m + (o == 1)) + o for m, o in zip(n, off)]
        g = np.meshgrid(*reversed(axes), indexing="ij")
        with np.errstate(all="ignore"):
            out.append(Fr.cv_fraction(phi, tuple(reversed(g))).reshape(-1))
    return out


@pytest.mark.parametrize("kind", ["random", "zeros", "tiny", "one_sign"])
@pytest.mark.parametrize("n", [(1, 1), (31, 7), (32, 8), (65, 17), (1, 1, 1), (31, 8, 2), (33, 7, 3), (64, 3, 2)])
def test_fractions_of_random_lattices(n, kind):
    require_gpu()
    from paper_1010_2832_gb300 import stokes
    rng = np.random.default_rng(list(n) + [len(kind)])
    dim = len(n)
    phiL, phiS = _level_set(rng, n, kind), _level_set(rng, n, kind)
    ctx = stokes.StokesContext(dim, n, 0.1, 0.01)
    shp = lambda off: tuple(reversed([m + (o == 1) for m, o in zip(n, off)]))
    faces = OFF[dim][2:] if dim == 2 else OFF[dim][1:4]
    sites = OFF[dim][:2] if dim == 2 else OFF[dim][:1] + OFF[dim][4:]
    one = lambda offs: [to_gpu(np.ones(shp(o))) for o in offs]
    ctx.build_weights(to_gpu(phiL), to_gpu(phiS), one(faces), one(sites), one(faces))
    wl, wf = ctx.export(0).cpu().numpy(), ctx.export(1).cpu().numpy()
    ref_l, ref_s = _fractions(phiL, n), _fractions(phiS, n)
    assert np.array_equal(wl, np.concatenate(ref_l), equal_nan=True)
    assert np.array_equal(wf, np.concatenate([1.0 - f for f in ref_s]), equal_nan=True)
    # a second build on the same context leaves nothing of the first behind
    ctx.build_weights(to_gpu(np.ones_like(phiL)), to_gpu(np.ones_like(phiS)), one(faces), one(sites), one(faces))
    ctx.build_weights(to_gpu(phiL), to_gpu(phiS), one(faces), one(sites), one(faces))
    assert np.array_equal(ctx.export(0).cpu().numpy(), wl, equal_nan=True)
    ctx.close()
