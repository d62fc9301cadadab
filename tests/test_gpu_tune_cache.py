"""The batch tuner's cache file: an entry written for an earlier kernel (a key
without this kernel's revision) is not taken, one written by this build is."""
import pytest

from gpu_common import require_gpu
from paper_1010_2832_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("precond", [0, 2])
def test_entries_of_an_earlier_kernel_are_not_taken(tmp_path, precond):
    require_gpu()
    from paper_1010_2832_gb300 import stokes
    ctxs = [stokes.context_for(w, min_face_liquid=0.01)[0] for w in (W.disk_in_box(32), W.bumps_2d(48, seed=3))]
    slots = 0
    for c in ctxs:
        lay = c.layout
        slots += lay.pitch * lay.rows
    gpu = torch.cuda.get_device_name().replace(" ", "_")
    old = f"batch2d_fp64_{'schwarz_' if precond else ''}n2_slots2^{slots.bit_length() - 1}_{gpu}"
    path = tmp_path / "tune.txt"
    path.write_text(f"{old} 16 1 12345.5\n")
    opt = stokes.default_options(mode=0, precond=precond)
    first = stokes.Batch(ctxs, opt, str(path)).tuning()
    assert first["us_per_iter"] != 12345.5
    lines = path.read_text().splitlines()
    assert len(lines) == 2 and lines[0].startswith(old + " ") and lines[1].startswith(old + "_")
    # this build's entry is taken, with whatever it says
    path.write_text(lines[1].split()[0] + " 8 1 777.25\n")
    again = stokes.Batch(ctxs, opt, str(path)).tuning()
    assert (again["tile_rows"], again["ctas_per_sm"], again["us_per_iter"]) == (8, 1, 777.25)
