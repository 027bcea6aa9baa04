"""FP32 passes whose dynamic shared memory lies just below 48 KB: with their static arrays they need more than
the limit a kernel starts with.  Bytes of the row, output, y and Green passes at the sizes below (tile + labels +
twiddles + landing slots, a 16-byte position index of x for the output): 2D row 48288 at 704; output 48448 at
686; Green 48960 at 720, 49152 at 819; 3D row 48864 at 364; output 49072 at 360; y 49152 at 384; Green 48048
at 364.  In a process of its own, so that no larger launch has raised the limit before."""
import subprocess
import sys

import pytest

from conftest import ROOT

pytestmark = pytest.mark.gpu

CODE = """
import numpy as np, torch
import hom_inputs as H
import paper_1412_3228_gb300 as hom
dim, sizes = %d, %r
for n in sizes:
    cell = H.Cell(dim, n, 0, [H.Primitive(H.PRIM_DISK if dim == 2 else H.PRIM_SPHERE, 1, (0.45, 0.5, 0.55), 0.28)],
                  H.RULE_NONE, 1.0, 4)
    ph = H.two_phases(3.0)
    mat = hom.hom_filter_build([cell], ph)
    for scheme in (0, 1):
        kw = dict(precision=hom.HOM_FP32, criterion=hom.HOM_CRIT_EN, tol=0.0, max_iter=2, scheme=scheme)
        c0 = H.geometric_lame(ph, dim)
        E = np.eye(3 if dim == 2 else 6)[:1]
        a = hom.hom_solve(mat, E, c0, **kw)
        b = hom.hom_solve(mat, E, c0, passes=hom.HOM_PASSES_GENERIC, **kw)
        for key in ("eps", "sigma"):
            # in FP32 sums (a norm over 10^8 values): the two evaluations differ by FP32 rounding only
            assert float((a[key] - b[key]).norm() / b[key].norm()) < 5e-6, (n, scheme, key)
print("launched")
"""


@pytest.mark.parametrize("dim,sizes", [(2, (686, 704, 720, 819)), (3, (360, 364, 384))], ids=["2d", "3d"])
def test_every_launch_finds_its_shared_memory(dim, sizes):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1412_3228_gb300 import _build_lib
    _build_lib.build()
    r = subprocess.run([sys.executable, "-c", CODE % (dim, sizes)], cwd=ROOT, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0 and "launched" in r.stdout, r.stderr[-2000:]
