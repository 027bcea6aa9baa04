"""The autotuner with options that its trial solves must not take over: a warm start (the trials have no initial
field) and defect correction.  Both run on the generic passes, so what is chosen for them is kept apart from the
choice for plain solves of the shape."""
import numpy as np
import pytest
import torch

import hom_inputs as H

pytestmark = pytest.mark.gpu

hom = pytest.importorskip("paper_1412_3228_gb300")
SIZE = 39  # no other test tunes this size


@pytest.fixture(scope="module", autouse=True)
def _device():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1412_3228_gb300 import _build_lib
    _build_lib.build()


def _lines():
    return [ln for ln in hom.hom_autotune_report().splitlines() if ln.split(":")[0].endswith(" %dx1" % SIZE)]


def test_tuned_warm_start_and_refinement():
    """Against the same calls without tuning: other radices, so other FP32 rounding, and at most one iteration
    more or less, a step of about the error 1e-5 at the stop: bar 5e-5 of the field."""
    cell, phases = H.centred_disk_cell(SIZE, rule=H.RULE_TWO_LAYER), H.two_phases(10.0)
    c0, E = H.mean_lame(phases), np.eye(3)
    mat = hom.hom_filter_build([cell], phases)
    kw = dict(precision=hom.HOM_FP32, criterion=hom.HOM_CRIT_EN, max_iter=2000)
    start = hom.hom_solve(mat, E, c0, tol=1e-3, **kw)["eps"]
    for opts in (dict(tol=1e-5, eps0=start), dict(tol=1e-8, refine=4)):
        plain = hom.hom_solve(mat, E, c0, **opts, **kw)
        tuned = hom.hom_solve(mat, E, c0, tune=True, **opts, **kw)
        assert (tuned["status"] == 0).all() and (plain["status"] == 0).all()
        assert float((tuned["eps"] - plain["eps"]).norm() / plain["eps"].norm()) < 5e-5
        assert np.abs(tuned["mean_sigma"] - plain["mean_sigma"]).max() < 5e-5 * np.abs(plain["mean_sigma"]).max()
    assert len(_lines()) == 1 and " generic n " in _lines()[0], _lines()
    assert "specialised" not in _lines()[0].split("->")[1]
    hom.hom_solve(mat, E, c0, tol=1e-5, tune=True, **kw)
    assert len(_lines()) == 2, _lines()
