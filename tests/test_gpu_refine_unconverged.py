"""Defect correction that ends above the tolerance: the results are those of the last FP64 check, whatever its
error.  With tol = 0 no load case can pass a check, so every one of them ends that way."""
import numpy as np
import pytest
import torch

import hom_inputs as H

pytestmark = pytest.mark.gpu

hom = pytest.importorskip("paper_1412_3228_gb300")


@pytest.fixture(scope="module", autouse=True)
def _device():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1412_3228_gb300 import _build_lib
    _build_lib.build()


@pytest.mark.parametrize("dim,n,criterion", [(2, 45, 0), (2, 45, 1), (3, 15, 1)])
def test_results_of_an_unconverged_refinement(dim, n, criterion):
    """Mean stress against a converged FP64 solve: the FP32 iteration stalls at e_n near contrast 2^-24 = 6e-6,
    and the fixed point contracts by 1 - 2 / contrast, so the strain is within 50 times that of the solution:
    3e-4, below the bar of 1e-3.  e_n lies between 0 and the same bar, e, which weighs every wave vector xi by
    |xi| <= pi n sqrt(dim) instead of 1, between 0 and that many times the bar.  A second call, after an
    unrelated solve has left its own numbers in the workspace, gives the same values."""
    contrast = 100.0
    nc = 3 if dim == 2 else 6
    kind = H.PRIM_DISK if dim == 2 else H.PRIM_SPHERE
    cell = H.Cell(dim, n, 0, [H.Primitive(kind, 1, (0.45, 0.5, 0.55), 0.28)], H.RULE_VOIGT, 0.9, 6)
    phases = H.two_phases(contrast)
    c0 = H.mean_lame(phases)
    mat = hom.hom_filter_build([cell], phases)
    want = hom.hom_solve(mat, np.eye(nc), c0, precision=hom.HOM_FP64, criterion=hom.HOM_CRIT_EN, tol=1e-9,
                         max_iter=20000, fields=False)
    assert want["code"] == hom.HOM_OK
    kw = dict(precision=hom.HOM_FP32, criterion=criterion, tol=0.0, max_iter=5000, refine=1, refine_inner=1)
    runs = [hom.hom_solve(mat, np.eye(nc), c0, **kw)]
    other = hom.hom_filter_build([H.centred_disk_cell(135)] * 3, H.two_phases(7.0))
    hom.hom_solve(other, np.eye(3), H.mean_lame(H.two_phases(7.0)), precision=hom.HOM_FP64, tol=1e-3, max_iter=50)
    runs.append(hom.hom_solve(mat, np.eye(nc), c0, **kw))
    for r in runs:
        assert r["code"] == hom.HOM_ERR_NOT_CONVERGED and (r["status"] != 0).all()
        assert np.abs(r["mean_sigma"] - want["mean_sigma"]).max() < 1e-3 * np.abs(want["mean_sigma"]).max()
        for key, bar in (("err", 1e-3 * np.pi * n * np.sqrt(dim)), ("err_n", 1e-3)):
            assert (r[key] > 0.0).all() and (r[key] < bar).all(), r[key]
    for key in ("mean_sigma", "err", "err_n", "iterations"):
        np.testing.assert_array_equal(runs[0][key], runs[1][key])
