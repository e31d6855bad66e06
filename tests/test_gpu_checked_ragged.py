"""The bounds-checked build on the kernels that walk ragged tiles: the Arnoldi step's row tiles
and vector groups, the operator's z chunks over planes that do not divide into blocks, the
packing of one colour, and the three orders of the complex64 restriction -- no index out of
range recorded.  (The checked library runs in a child process, as in test_gpu_checked.py.)"""
import json
import os
import subprocess
import sys

import pytest

from tests.gpu_common import need_gpu

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import ctypes as C, json, sys
import numpy as np, torch
sys.path.insert(0, %(root)r)
import scenes
from tests.gpu_common import problem_for, small_scene, to_dev
import paper_2405_12380_gb300 as hm
from paper_2405_12380_gb300 import _lib
seen = {}
def look(what):
    torch.cuda.synchronize()
    chk, first = C.c_int(0), C.c_ulonglong(0)
    rc = _lib.lib().helm_checked_status(C.byref(chk), C.byref(first))
    seen[what] = [rc, chk.value, first.value >> 8, first.value & 255]
for dim, n in [(2, 9), (2, 33), (2, 71), (3, 5), (3, 13), (3, 22), (3, 31), (3, 45), (3, 66)]:
    s = small_scene(dim, n, cells=1 if n < 9 else 4)
    for prec in ("fp64", "mixed"):
        P = problem_for(s, precision=prec)
        P.don_load(scenes.glorot_mlp(np.random.default_rng(3), [dim, 32, 32, 13]), 13, tau=1e-3)
        b = to_dev(s["b"])
        for dt in (torch.complex128, torch.complex64):
            x = b.to(dt)
            P.apply(x); P.residual(x, x.clone())
            for kind, sweeps in (("rbgs", 1), ("rbgs", 2), ("sor", 1), ("jacobi", 1), ("jacobi", 3)):
                P.relax(kind, x, x.clone(), sweeps=sweeps, omega=0.8)
        look(f"{dim}d {n} {prec} kernels")
        for relax, n_r in (("none", 0), ("rbgs", 1), ("jacobi", 2), ("sor", 1)):
            P.solve(b, None, hm.opts("fgmres", relax, n_r, omega=0.8, tol=1e-14, restart=40, maxit=12 if n > 20 else 45))
            look(f"{dim}d {n} {prec} fgmres {relax}")
        P.close()
print("RESULT " + json.dumps(seen))
"""


def test_no_index_out_of_range():
    need_gpu()
    if not os.path.exists(os.path.join(ROOT, "paper_2405_12380_gb300", "libhelm_checked.so")):
        pytest.fail("libhelm_checked.so not built (__graft_entry__.build builds it)")
    r = subprocess.run([sys.executable, "-c", CHILD % {"root": ROOT}], env=dict(os.environ, HELM_LIBRARY="checked"),
                       capture_output=True, text=True, timeout=600, cwd=ROOT)
    assert r.returncode == 0, r.stderr[-3000:]
    seen = json.loads([ln for ln in r.stdout.splitlines() if ln.startswith("RESULT ")][-1][len("RESULT "):])
    assert seen and all(v == [0, 1, 0, 0] for v in seen.values()), {k: v for k, v in seen.items() if v != [0, 1, 0, 0]}
