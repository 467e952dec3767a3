"""A failed build of the matrix sweeps' chunk matrices leaves none behind: the call
returns its error, the next one builds them.  The failure is a runtime call's
error code, from a stand-in for cudaFuncSetAttribute preloaded in a child process
(it refuses the build kernel's shared-memory limit while armed)."""
import os
import shutil
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

STAND_IN = """
#define _GNU_SOURCE
#include <dlfcn.h>
#include <stddef.h>
typedef int (*fn)(const void *, int, int);
static int refused = 0;
void refuse(int bytes) { refused = bytes; }
int cudaFuncSetAttribute(const void *f, int attr, int value) {
    if (refused && value == refused) return 1;   /* cudaErrorInvalidValue */
    void *rt = dlopen("libcudart.so.13", RTLD_LAZY | RTLD_NOLOAD);
    fn real = rt ? (fn)dlsym(rt, "cudaFuncSetAttribute") : NULL;
    return real ? real(f, attr, value) : 1;
}
"""

CHILD = """
import ctypes, sys
import numpy as np
import torch
import synth
from synth.meshes import box_mesh
from paper_2210_04891_gb300 import api, native, PREC_DF, PREC_FP64

stand_in = ctypes.CDLL(sys.argv[1])
m = box_mesh(150 * 8e-6, 20e-6, 10e-6, 150, 2, 1, jitter=0.1, seed=3)
M = api.Mesh.from_synth(m)
L = api.Loops(M, m.ports)
P, Q = (api.Plan(M, L, dict(grid=(16, 8, 8), n_touch=4)) for _ in range(2))
y = torch.from_numpy(synth.complex_gaussian(L.nl, 2, seed=5)).cuda()
om = 2 * np.pi * np.array([1e8, 1e9])
for prec in (PREC_FP64, PREC_DF):
    stand_in.refuse(3 * 32 * 33 * 16)
    try:
        api.pfft_precond_apply(P, y, om, prec=prec)
        raise SystemExit("the refused build went through")
    except native.SieError as e:
        assert e.code == -5, e
    stand_in.refuse(0)
    z = api.pfft_precond_apply(P, y, om, prec=prec)
    ref = api.pfft_precond_apply(Q, y, om, prec=prec)
    assert torch.equal(z, ref), (prec, (z - ref).abs().max().item())
print("ok")
"""


@pytest.mark.skipif(shutil.which("gcc") is None, reason="needs a C compiler")
def test_failed_build_leaves_no_matrices(tmp_path):
    src, lib, child = tmp_path / "stand_in.c", tmp_path / "stand_in.so", tmp_path / "child.py"
    src.write_text(STAND_IN)
    child.write_text(CHILD)
    subprocess.run(["gcc", "-shared", "-fPIC", "-O1", "-o", str(lib), str(src), "-ldl"], check=True)
    env = dict(os.environ, LD_PRELOAD=str(lib), PYTHONPATH=ROOT + os.pathsep + os.environ.get("PYTHONPATH", ""))
    r = subprocess.run([sys.executable, str(child), str(lib)], cwd=ROOT, env=env, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip().endswith("ok"), r.stdout + r.stderr
