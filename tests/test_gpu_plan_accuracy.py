"""Accuracy of the FP32 passes whose radices are read from a plan, against FP64 iterates.  Their stages read every
twiddle from a table, as the generic passes do, so both round alike: the ratio of their errors is 1 but for the
luck of a size, a few per cent each, and its geometric mean over five sizes stays below 1.1 (twiddles formed as
products of table entries gave 1.21)."""
import numpy as np
import pytest
import torch

import hom_inputs as H

pytestmark = pytest.mark.gpu

hom = pytest.importorskip("paper_1412_3228_gb300")


def _error(mat, dim, loads, ref, **kw):
    s = hom.hom_solve(mat, np.eye(3 if dim == 2 else 6)[:loads], H.mean_lame(H.two_phases(10.0)), precision=hom.HOM_FP32,
                      tol=0.0, max_iter=25, **kw)["sigma"].double()
    return float((s - ref).norm() / ref.norm())


def test_errors_are_those_of_the_generic_passes():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1412_3228_gb300 import _build_lib
    _build_lib.build()
    ratios = []
    for dim, n in ((2, 512), (2, 640), (2, 1024), (3, 64), (3, 128)):
        prim = H.Primitive(H.PRIM_DISK if dim == 2 else H.PRIM_SPHERE, 1, (0.43, 0.51, 0.55), 0.27)
        mat = hom.hom_filter_build([H.Cell(dim, n, 0, [prim], H.RULE_VOIGT, 0.9, 6)], H.two_phases(10.0))
        ref = hom.hom_solve(mat, np.eye(3 if dim == 2 else 6)[:2], H.mean_lame(H.two_phases(10.0)), precision=hom.HOM_FP64,
                            tol=0.0, max_iter=25)["sigma"]
        ratios.append(_error(mat, dim, 2, ref) / _error(mat, dim, 2, ref, passes=hom.HOM_PASSES_GENERIC))
    assert np.exp(np.mean(np.log(ratios))) < 1.1, ratios
