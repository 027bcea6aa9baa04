"""The bounds-checked build (-DHOM_DEBUG) on every FP32 path of the solver: the on-chip solver of small 2D grids
(clusters of 1 to 8 CTAs, both schemes, private state on chip and in the workspace), the 2D passes with compiled
and with plan-read radices (a 405 grid keeps a batch off the chip), the 3D ones, the adjoint and the no-allocation
entry point.  No check may fail (that would be an error code), no unwritten shared memory may reach a result (it is
poisoned with NaN), and iteration counts and mean stresses are those of the release build on the same kernels."""
import json
import os
import subprocess
import sys

import numpy as np
import pytest
import torch

from conftest import ROOT

pytestmark = pytest.mark.gpu

hom = pytest.importorskip("paper_1412_3228_gb300")

CODE = r'''
import json, sys
import numpy as np, torch
import paper_1412_3228_gb300 as hom
import hom_inputs as H

if sys.argv[1] == "debug":
    hom.use_debug_library()
    assert hom.lib().hom_build_flags() == 1
torch.cuda.set_device(0)
out = {}
ph = H.two_phases(8.0)
def cell(dim, n):
    kind = H.PRIM_DISK if dim == 2 else H.PRIM_SPHERE
    return H.Cell(dim, n, 0, [H.Primitive(kind, 1, (0.43, 0.51, 0.55), 0.27)], H.RULE_VOIGT if n >= 9 else H.RULE_NONE, 0.9, 6)
def solve(name, sizes, dim, scheme, loads, f=hom.hom_solve, **kw):
    mat = hom.hom_filter_build([cell(dim, n) for n in sizes], ph)
    E = np.eye(3 if dim == 2 else 6)[:loads]
    c0 = H.geometric_lame(ph, dim) if scheme else H.mean_lame(ph)
    kw.update(precision=hom.HOM_FP32, criterion=hom.HOM_CRIT_EN, tol=1e-3, max_iter=60)
    if scheme:
        kw.update(scheme=scheme)
    r = f(mat, E, c0, **kw)
    out[name] = dict(it=r["iterations"].tolist(), ms=r["mean_sigma"].tolist(),
                     nan=bool(torch.isnan(r["eps"]).any() or torch.isnan(r["sigma"]).any()))
    return mat, r, c0
for scheme in (0, 1):
    for i, (sizes, loads) in enumerate([((3, 4, 9, 16), 3), ((30, 45), 2), ((91, 143), 1), ((150, 208), 1), ((208,) * 3, 3)]):
        solve("on chip %d %d" % (scheme, i), sizes, 2, scheme, loads)
    solve("compiled 2D %d" % scheme, (45, 75, 135, 405), 2, scheme, 2)
    solve("plan-read 2D %d" % scheme, (45, 64, 77, 405, 300), 2, scheme, 3)
    solve("compiled 3D %d" % scheme, (27,), 3, scheme, 2)
    solve("plan-read 3D %d" % scheme, (14, 11), 3, scheme, 2)
solve("no allocation", (45, 64), 2, 0, 3, f=hom.hom_solve_noalloc)
solve("no allocation, passes", (405,), 2, 0, 1, f=hom.hom_solve_noalloc)
for dim, sizes in ((2, (405, 50)), (3, (14,))):
    mat, fwd, c0 = solve("forward %dD" % dim, sizes, dim, 0, 3 if dim == 2 else 6)
    b = hom.hom_solve_backward(mat, fwd, c0, dL_dsigma=fwd["sigma"] / 1000.0, precision=hom.HOM_FP32,
                               criterion=hom.HOM_CRIT_EN, tol=0.0, max_iter=6)
    out["adjoint %dD" % dim] = dict(it=[0], ms=np.asarray(b["dphase"]).tolist(), nan=bool(torch.isnan(b["dctilde"]).any()))
print(json.dumps(out))
'''


def _run(kind):
    env = dict(os.environ, PYTHONPATH=ROOT + os.pathsep + os.environ.get("PYTHONPATH", ""))
    r = subprocess.run([sys.executable, "-c", CODE, kind], capture_output=True, text=True, cwd=ROOT, env=env, timeout=600)
    assert r.returncode == 0, r.stderr[-3000:]
    return json.loads(r.stdout.strip().splitlines()[-1])


def test_every_fp32_path_passes_its_checks():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1412_3228_gb300 import _build_lib
    _build_lib.build()
    _build_lib.build(debug=True)
    dbg, rel = _run("debug"), _run("release")
    assert dbg.keys() == rel.keys()
    for k in rel:
        assert not dbg[k]["nan"] and not rel[k]["nan"], k
        # the same operations in the same order; contraction of a x + b may differ between the two builds
        assert np.abs(np.asarray(dbg[k]["it"]) - np.asarray(rel[k]["it"])).max() <= 1, k
        a, b = np.asarray(dbg[k]["ms"]), np.asarray(rel[k]["ms"])
        assert np.abs(a - b).max() <= (2e-3 if dbg[k]["it"] != rel[k]["it"] else 1e-5) * np.abs(b).max(), k
