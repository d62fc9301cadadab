"""The Schwarz plan's local factorisation at patch sizes from a few unknowns to
the full 108 (blocks of 16 rows in registers: one block, ragged ones, all seven),
against dense FP64 local solves.  The stored factor is FP16 (each entry within
2^-11) and enters twice; the patches' inverse factors have conditions of tens, so
5e-2 relative (RMS) is the bound, where a misplaced entry gives an error of order
one on grids of so few patches."""
import numpy as np
import pytest

from gpu_common import gpu_context, oracle_system, require_gpu
from oracle import solve as So
from paper_1010_2832_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

CASES = {"one": lambda: W.disk_in_box(6, radius=0.2), "rand5x7": lambda: W.random_small((5, 7), seed=1),
         "rand9x8": lambda: W.random_small((9, 8), seed=2), "rand23x21": lambda: W.random_small((23, 21), seed=3),
         "full13": lambda: W.full_box(13, 2, seed=2)}


@pytest.mark.parametrize("name", list(CASES))
def test_local_solves_match_dense_ones(name):
    require_gpu()
    wl = CASES[name]()
    S = oracle_system(wl)
    ctx = gpu_context(wl)[0]
    r = np.random.default_rng(7).normal(size=S.A.shape[0])
    z_ref = So.additive_schwarz(S, r)
    zs = ctx.new_vector(torch.float32)
    ctx.apply_preconditioner(2, ctx.fields_to_slots(torch.from_numpy(r).cuda()).to(torch.float32), zs)
    z = ctx.slots_to_fields(zs.to(torch.float64)).cpu().numpy()
    act = S.active
    assert act.any()
    assert np.linalg.norm((z - z_ref)[act]) <= 5e-2 * np.linalg.norm(z_ref[act])
