"""Results do not depend on how many rows and columns a task of the generic passes takes (small batches take fewer
than fit on chip): batches of one grid size and of several, 2D and 3D, odd and even, one load and all, against the
same cells inside a batch that is large enough for whole tasks."""
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


def _cell(dim, n):
    kind = H.PRIM_DISK if dim == 2 else H.PRIM_SPHERE
    return H.Cell(dim, n, 0, [H.Primitive(kind, 1, (0.43, 0.51, 0.55), 0.27)], H.RULE_VOIGT if n >= 9 else H.RULE_NONE, 0.9, 6)


# (dimension, sizes, loads, copies of the batch that make at least 608 whole tasks in each pass)
BATCHES = [(2, (5, 7), 3, 700), (2, (45,), 1, 320), (2, (64,), 3, 120), (2, (165,), 2, 40), (2, (27, 99, 33), 3, 80),
           (3, (5,), 6, 320), (3, (9, 13), 1, 160), (3, (16,), 6, 40), (3, (26,), 3, 24)]


@pytest.mark.parametrize("precision", [0, 1], ids=["fp32", "fp64"])
@pytest.mark.parametrize("dim,sizes,loads,copies", BATCHES, ids=["%dd-%s-%d" % (b[0], "-".join(map(str, b[1])), b[2]) for b in BATCHES])
def test_small_batches_against_their_copies(dim, sizes, loads, copies, precision):
    """Rows are paired into complex lines task by task, so the two differ by rounding: a few iterations of a
    contraction (contrast 3), as in test_gpu_run_sizes.py: 5e-6 in FP32, 5e-6 x 2^-29 = 1e-14 in FP64, times ten
    there for sums of up to 4e4 values in another order."""
    phases = H.two_phases(3.0)
    E = np.eye(3 if dim == 2 else 6)[:loads]
    kw = dict(precision=precision, criterion=hom.HOM_CRIT_EN, tol=0.0, max_iter=6)
    if precision == hom.HOM_FP32:
        kw["passes"] = hom.HOM_PASSES_GENERIC
    tol = 5e-6 if precision == hom.HOM_FP32 else 1e-13
    cells = [_cell(dim, n) for n in sizes]
    small = hom.hom_solve(hom.hom_filter_build(cells, phases), E, H.mean_lame(phases), **kw)
    many = hom.hom_solve(hom.hom_filter_build(cells * copies, phases), E, H.mean_lame(phases), **kw)
    size = small["eps"].numel()
    for key in ("eps", "sigma"):
        a, b = small[key].double(), many[key][:size].double()
        assert float((a - b).norm() / b.norm()) < tol, key
    assert np.abs(small["mean_sigma"] - many["mean_sigma"][:len(cells)]).max() < tol * np.abs(small["mean_sigma"]).max()
    # e and e_n of the last iterate: residuals far above the rounding after six iterations of factor about 0.5
    np.testing.assert_allclose(small["err_n"], many["err_n"][:len(cells)], rtol=1e-3)
