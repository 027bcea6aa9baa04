"""hom_solve_noalloc at the limit of its fixed 64 MiB of scratch.  What a batch needs is its state, partial sums,
tables and a staged history; what speed costs in scratch (more tasks, split sums, plan-read passes) is given up
where it would not fit.  The histories here are sized to leave less than a page of 256 bytes."""
import re

import numpy as np
import pytest
import torch

import hom_inputs as H

pytestmark = pytest.mark.gpu

hom = pytest.importorskip("paper_1412_3228_gb300")

# As in test_gpu_run_sizes.py: two FP32 evaluations of a few iterations of a contraction (contrast 3)
TOL = 5e-6
SCRATCH = 64 << 20


@pytest.fixture(scope="module", autouse=True)
def _device():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1412_3228_gb300 import _build_lib
    _build_lib.build()


def _need(mat, E, c0, kw):
    """Scratch bytes of a batch without its history (which is staged in the scratch: 8 bytes per pair and entry)."""
    pairs, m = len(mat.cells) * len(E), SCRATCH // 8
    with pytest.raises(hom.HomError) as err:
        hom.hom_solve_noalloc(mat, E, c0, tol=1e-3, max_iter=m, history=True, **kw)
    need = int(re.search(r"needs (\d+) bytes", str(err.value)).group(1))
    return need - (pairs * (m + 1) * 8 + 255) // 256 * 256


def _limit(need, pairs):
    """The largest max_iter whose history still fits beside `need` bytes."""
    return (SCRATCH - need) // 256 * 256 // (8 * pairs) - 1


def test_noalloc_falls_back_to_the_generic_passes():
    """Plan-read passes hold one-byte labels (1 MB here) beside what the generic ones hold: a history that leaves room
    for the generic passes only, to less than a page."""
    phases = H.two_phases(3.0)
    mat = hom.hom_filter_build([H.Cell(2, 1000, 0, [H.Primitive(H.PRIM_DISK, 1, (0.43, 0.51, 0.55), 0.27)], H.RULE_VOIGT, 0.9,
                                       6)], phases)
    E, c0, kw = np.eye(3)[:1], H.mean_lame(phases), dict(precision=hom.HOM_FP32, criterion=hom.HOM_CRIT_EN)
    m = _limit(_need(mat, E, c0, kw), 1)
    got = hom.hom_solve_noalloc(mat, E, c0, tol=1e-3, max_iter=m, history=True, **kw)
    assert got["code"] == hom.HOM_OK
    gen = hom.hom_solve(mat, E, c0, tol=1e-3, max_iter=50, passes=hom.HOM_PASSES_GENERIC, **kw)
    np.testing.assert_array_equal(got["iterations"], gen["iterations"])
    assert np.abs(got["mean_sigma"] - gen["mean_sigma"]).max() < TOL * np.abs(gen["mean_sigma"]).max()
    for key in ("eps", "sigma"):
        x, y = got[key].double(), gen[key].double()
        assert float((x - y).norm() / y.norm()) < TOL, key
    with pytest.raises(hom.HomError) as err:  # 32 entries, a page of 256 bytes, more
        hom.hom_solve_noalloc(mat, E, c0, tol=1e-3, max_iter=m + 32, history=True, **kw)
    assert err.value.code == 2


@pytest.mark.parametrize("dim,sizes,loads,prec,need", [
    (2, (405,), 3, 0, 22481408), (2, (45, 135), 3, 0, 2911488), (3, (27,), 6, 0, 11972864), (3, (45,), 6, 0, 49622784),
    (2, (343,), 3, 0, 15969536), (3, (64,), 2, 0, 55087104), (2, (405,), 3, 1, 44527616), (3, (45,), 2, 1, 32686592),
    (2, (27,) * 8, 3, 1, 1836544), (2, (512,), 2, 1, 47635968)],
    ids=["2d-405-fp32", "2d-small-fp32", "3d-27-fp32", "3d-45-fp32", "2d-343-fp32", "3d-64-fp32", "2d-405-fp64", "3d-45-fp64",
         "2d-many-fp64", "2d-512-fp64"])
def test_noalloc_takes_what_its_scratch_holds(dim, sizes, loads, prec, need):
    """A batch needs its state, partial sums, tables and history, and no more: what speed costs in scratch (more
    tasks, split sums) is given up where it would not fit.  `need`: bytes without history at tasks as large as fit
    on chip."""
    phases = H.two_phases(10.0)
    prim = H.Primitive(H.PRIM_DISK if dim == 2 else H.PRIM_SPHERE, 1, (0.43, 0.51, 0.55), 0.27)
    cells = [H.Cell(dim, n, 0, [prim], H.RULE_NONE, 0.9, 6) for n in sizes]
    mat = hom.hom_filter_build(cells, phases)
    E = np.eye(3 if dim == 2 else 6)[:loads]
    kw = dict(precision=hom.HOM_FP64 if prec else hom.HOM_FP32, criterion=hom.HOM_CRIT_EN, tol=1e-2, fields=True)
    got = hom.hom_solve_noalloc(mat, E, H.mean_lame(phases), max_iter=_limit(need, loads * len(sizes)), history=True, **kw)
    ref = hom.hom_solve(mat, E, H.mean_lame(phases), max_iter=200, passes=hom.HOM_PASSES_GENERIC, **kw)
    assert (got["status"] == 0).all() and np.abs(got["iterations"] - ref["iterations"]).max() <= 1
    if (got["iterations"] == ref["iterations"]).all():
        assert np.abs(got["mean_sigma"] - ref["mean_sigma"]).max() < 1e-5 * np.abs(ref["mean_sigma"]).max()
