"""FP32 passes with radices read from a plan, and the on-chip solver of small 2D grids, against the generic
passes: the same fixed number of iterations on the same material, so the fields differ by FP32
rounding only.  Sizes: every register radix in the first and in a later stage, one to four stages, even
grids (padded tiles, Nyquist bins, half spectra of odd and even length), the smallest grids, and the
edges of the on-chip solver's cluster sizes."""
import numpy as np
import pytest
import torch

import hom_inputs as H

pytestmark = pytest.mark.gpu

hom = pytest.importorskip("paper_1412_3228_gb300")

SIZES2 = [3, 4, 5, 6, 7, 8, 9, 11, 13, 14, 15, 16, 22, 26, 30, 32, 33, 35, 39, 45, 48, 49, 63, 64, 65, 75, 77, 84, 88, 90,
          91, 96, 104, 121, 128, 130, 135, 143, 169, 176, 195, 208, 225, 240, 243, 256, 260, 264, 343, 512, 686, 1024, 1080]
SIZES3 = [5, 6, 8, 9, 11, 13, 16, 21, 22, 26, 27, 30, 33, 35, 49]
# Two FP32 evaluations of a contraction (factor about 0.5 at contrast 3) each carry the rounding of the
# last few iterations: a few times 2^-24 sqrt(log2 of the transform's length) relative to the field.
TOL = 5e-6


@pytest.fixture(scope="module", autouse=True)
def _device():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1412_3228_gb300 import _build_lib
    _build_lib.build()


def _cell(dim, n, k=0):
    rule = (H.RULE_VOIGT, H.RULE_TWO_LAYER, H.RULE_REUSS)[(n + k) % 3] if n >= 9 else H.RULE_NONE
    kind = H.PRIM_DISK if dim == 2 else H.PRIM_SPHERE
    return H.Cell(dim, n, 0, [H.Primitive(kind, 1, (0.43 + 0.02 * k, 0.51, 0.55), 0.27 if dim == 2 else 0.3)], rule, 0.9, 6)


def _rel(a, b):
    a, b = a.double(), b.double()
    return float((a - b).norm() / b.norm())


def _compare(cells, phases, dim, loads, scheme, rel=TOL):
    mat = hom.hom_filter_build(cells, phases)
    E = np.eye(3 if dim == 2 else 6)[:loads]
    c0 = H.geometric_lame(phases[:2], dim) if scheme else H.mean_lame(phases[:2])
    kw = dict(precision=hom.HOM_FP32, criterion=hom.HOM_CRIT_EN, tol=0.0, max_iter=9, scheme=scheme, history=True)
    gen = hom.hom_solve(mat, E, c0, passes=hom.HOM_PASSES_GENERIC, **kw)
    by_passes = hom.hom_solve(mat, E, c0, stats=True, **kw)  # statistics keep small grids on the passes
    auto = hom.hom_solve(mat, E, c0, **kw)
    for r in (by_passes, auto):
        assert (r["iterations"] == 9).all() and (r["status"] == gen["status"]).all()
        off = 0
        for c in cells:  # cell by cell: a small cell must not hide behind a large one
            size = loads * E.shape[1] * c.n ** dim
            sl = slice(off, off + size)
            assert _rel(r["eps"][sl], gen["eps"][sl]) < rel and _rel(r["sigma"][sl], gen["sigma"][sl]) < rel, c.n
            off += size
        assert np.abs(r["mean_sigma"] - gen["mean_sigma"]).max() < rel * np.abs(gen["mean_sigma"]).max()
        h, g = r["history"], gen["history"]
        big = g > 1e-3  # above the FP32 floor of the residual
        np.testing.assert_allclose(h[big], g[big], rtol=2e-3)
    return gen, by_passes, auto


@pytest.mark.parametrize("scheme", [0, 1], ids=["basic", "eyre-milton"])
@pytest.mark.parametrize("n", SIZES2)
def test_2d_sizes(n, scheme):
    _compare([_cell(2, n)], H.two_phases(3.0), 2, 3, scheme)


@pytest.mark.parametrize("scheme", [0, 1], ids=["basic", "eyre-milton"])
@pytest.mark.parametrize("n", SIZES3)
def test_3d_sizes(n, scheme):
    _compare([_cell(3, n)], H.two_phases(3.0), 3, 6 if n < 20 else 2, scheme)


@pytest.mark.parametrize("loads", [1, 2, 3])
def test_mixed_batches(loads):
    """Sizes of every path in one batch: on chip (each cluster size) and in passes, odd and even, repeated."""
    cells = [_cell(2, n, k) for k, n in enumerate((45, 63, 405, 16, 300, 130, 225, 45, 97 - 6, 260))]
    _compare(cells, H.two_phases(3.0), 2, loads, 0)


def test_many_small_cells():
    """More pairs than the chip holds clusters at once."""
    cells = [_cell(2, n, k % 5) for k, n in enumerate([45, 30, 64, 75] * 40)]
    _compare(cells, H.two_phases(3.0), 2, 3, 0)


def test_on_chip_stops_as_the_passes_do():
    """Convergence to a tolerance, divergence and stagnation stops, and a graph request, on chip."""
    cells, phases = [_cell(2, n, k) for k, n in enumerate((45, 64, 143))], H.two_phases(10.0)
    mat = hom.hom_filter_build(cells, phases)
    kw = dict(precision=hom.HOM_FP32, criterion=hom.HOM_CRIT_EN)
    c0 = np.array(H.mean_lame(phases))
    for opts in (dict(tol=1e-4, max_iter=400), dict(tol=1e-4, max_iter=400, use_graph=True),
                 dict(tol=1e-9, max_iter=400, stall_window=20), dict(tol=1e-4, max_iter=3), dict(tol=1e9, max_iter=5)):
        a = hom.hom_solve(mat, np.eye(3), c0, **opts, **kw)
        b = hom.hom_solve(mat, np.eye(3), c0, stats=True, **opts, **kw)
        np.testing.assert_array_equal(a["status"], b["status"])
        if "stall_window" not in opts:
            assert np.abs(a["iterations"] - b["iterations"]).max() <= 1
            if (a["iterations"] == b["iterations"]).all():
                assert _rel(a["eps"], b["eps"]) < TOL
    bad = hom.hom_solve(mat, np.eye(3), 0.3 * c0, tol=1e-6, max_iter=4000, diverge_window=20, **kw)
    assert (bad["status"] == 2).all()


def test_adjoint_on_run_sizes():
    """The source term of the adjoint row pass on sizes without compiled radices."""
    for dim, n in ((2, 50), (3, 14)):
        cell, phases = _cell(dim, n), H.two_phases(4.0)
        nc = 3 if dim == 2 else 6
        mat = hom.hom_filter_build([cell], phases)
        c0 = H.mean_lame(phases)
        fwd = hom.hom_solve(mat, np.eye(nc), c0, precision=hom.HOM_FP32, criterion=hom.HOM_CRIT_EN, tol=0.0, max_iter=15)
        S = fwd["sigma"] / n ** dim
        g = [hom.hom_solve_backward(mat, fwd, c0, dL_dsigma=S, precision=hom.HOM_FP32, criterion=hom.HOM_CRIT_EN, tol=0.0,
                                    max_iter=12, passes=p) for p in (hom.HOM_PASSES_AUTO, hom.HOM_PASSES_GENERIC)]
        assert _rel(g[0]["dctilde"], g[1]["dctilde"]) < 2 * TOL
        np.testing.assert_allclose(g[0]["dphase"], g[1]["dphase"], rtol=1e-4, atol=1e-5 * np.abs(g[1]["dphase"]).max())
