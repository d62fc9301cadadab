"""Small systems whose one-kernel loop the device refuses (a cooperative launch
that is too large for the SMs a process may use) or has no memory for: the
separate kernels take the solve, with the same result; and a Schwarz plan without
memory for its room to grow.  The refusals are made on the host, by a library
loaded before the CUDA runtime in a process of its own."""
import os
import subprocess
import sys

import pytest

from gpu_common import require_gpu

pytestmark = pytest.mark.gpu

FAKE = r"""
#define _GNU_SOURCE
#include <dlfcn.h>
#include <stddef.h>
static int launches, mallocs, seen, from, to;
void fake_refuse(int a, int b) { seen = 0; from = a; to = b; }        /* the a-th to the b-1-th allocation from now */
int fake_launches(void) { return launches; }
int fake_mallocs(void) { return mallocs; }
int cudaLaunchCooperativeKernel(const void* f, unsigned long long gxy, unsigned gz, unsigned long long bxy, unsigned bz,
                                void** args, size_t smem, void* stream) {
    (void)f; (void)gxy; (void)gz; (void)bxy; (void)bz; (void)args; (void)smem; (void)stream;
    ++launches;
    return 720;                                    /* cudaErrorCooperativeLaunchTooLarge */
}
int cudaMalloc(void** p, size_t n) {
    static int (*next)(void**, size_t);
    if (!next) next = (int (*)(void**, size_t))dlsym(dlopen("libcudart.so.13", RTLD_LAZY | RTLD_NOLOAD), "cudaMalloc");
    const int k = seen++;
    if (k >= from && k < to) { ++mallocs; return 2; }                  /* cudaErrorMemoryAllocation */
    return next(p, n);
}
"""

RUN = r"""
import ctypes, hashlib, os, sys
import torch
from paper_1010_2832_gb300 import stokes, workloads as W
how = sys.argv[1]
fake = ctypes.CDLL(os.environ["FAKE_CUDA"]) if how != "plain" else None
ctx, dev = stokes.context_for(W.disk_in_box(32), min_face_liquid=0.01)
b = ctx.new_vector()
ctx.rhs(dev["u_star"], b)
for kw in (dict(mode=0), dict(mode=1), dict(mode=1, precond=2)):
    x = ctx.new_vector()
    if how == "malloc":
        if kw.get("precond") == 2:                 # the patch factors' own memory, before the loop's
            z = ctx.new_vector(torch.float32)
            ctx.apply_preconditioner(2, b.to(torch.float32), z)
        fake.fake_refuse(0, 1 << 30)
    if how == "room" and kw.get("precond") == 2:   # the patch grid's buffer, then the factors with room to grow
        fake.fake_refuse(1, 2)
    st = ctx.solve_system(b, x, stokes.default_options(tol=1e-9, **kw))
    if fake:
        fake.fake_refuse(0, 0)
    print(st.status, st.iterations, hashlib.sha1(x.cpu().numpy().tobytes()).hexdigest())
if fake:
    print("refused", fake.fake_mallocs() if how != "launch" else fake.fake_launches(), file=sys.stderr)
"""


def _run(tmp_path, how):
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    src, lib = tmp_path / f"{how}.c", tmp_path / f"lib{how}.so"
    src.write_text(FAKE.replace("cudaLaunchCooperativeKernel", "unused") if how != "launch" else FAKE)
    subprocess.run(["gcc", "-shared", "-fPIC", "-O1", "-o", str(lib), str(src), "-ldl"], check=True)
    env = dict(os.environ, PYTHONPATH=root, FAKE_CUDA=str(lib))
    if how != "plain":
        env["LD_PRELOAD"] = str(lib)
    r = subprocess.run([sys.executable, "-c", RUN, how], cwd=root, capture_output=True, text=True, timeout=300, env=env)
    assert r.returncode == 0, r.stderr
    return r.stdout, int(r.stderr.split("refused")[1].split()[0]) if how != "plain" else 0


@pytest.mark.parametrize("how,least", [("launch", 3), ("malloc", 3), ("room", 1)])
def test_refusals_leave_the_result_as_it_is(tmp_path, how, least):
    """launch: the cooperative launches; malloc: the loops' words; room: the
    Schwarz factors' buffer with its room to grow."""
    require_gpu()
    plain, _ = _run(tmp_path, "plain")
    assert plain.count("\n") == 3 and all(line.startswith("0 ") for line in plain.splitlines())
    out, refused = _run(tmp_path, how)
    assert out == plain
    assert refused >= least
