"""Which FP32 path a batch takes, and that its results do not depend on it: batches that run on chip whole (all
cluster sizes), batches that stay in the passes (a large grid, many pairs, a grid on which they are faster), and
whole-solve graphs of the passes (2D and 3D, compiled and plan-read radices, both schemes).  But for one, the
solves do not ask for the residual history, so iterates above the tolerance take the short way through the
stopping rule."""
import numpy as np
import pytest
import torch

import hom_inputs as H

pytestmark = pytest.mark.gpu

hom = pytest.importorskip("paper_1412_3228_gb300")

# As in test_gpu_run_sizes.py: two FP32 evaluations of a few iterations of a contraction (contrast 3)
TOL = 5e-6


@pytest.fixture(scope="module", autouse=True)
def _device():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1412_3228_gb300 import _build_lib
    _build_lib.build()


def _cell(dim, n, k=0):
    kind = H.PRIM_DISK if dim == 2 else H.PRIM_SPHERE
    return H.Cell(dim, n, 0, [H.Primitive(kind, 1, (0.43 + 0.02 * k, 0.51, 0.55), 0.27)],
                  H.RULE_VOIGT if n >= 9 else H.RULE_NONE, 0.9, 6)


def _problem(dim, sizes, loads, scheme):
    phases = H.two_phases(3.0)
    cells = [_cell(dim, n, k % 5) for k, n in enumerate(sizes)]
    c0 = H.geometric_lame(phases, dim) if scheme else H.mean_lame(phases)
    kw = dict(precision=hom.HOM_FP32, criterion=hom.HOM_CRIT_EN)
    if scheme:
        kw["scheme"] = scheme
    return cells, hom.hom_filter_build(cells, phases), np.eye(3 if dim == 2 else 6)[:loads], c0, kw


def _close(a, b, cells, loads):
    np.testing.assert_array_equal(a["iterations"], b["iterations"])
    np.testing.assert_array_equal(a["status"], b["status"])
    assert np.abs(a["mean_sigma"] - b["mean_sigma"]).max() < TOL * np.abs(b["mean_sigma"]).max()
    off = 0
    for c in cells:
        size = loads * (3 if c.dim == 2 else 6) * c.n ** c.dim
        for key in ("eps", "sigma"):
            x, y = a[key][off:off + size].double(), b[key][off:off + size].double()
            assert float((x - y).norm() / y.norm()) < TOL, (key, c.n)
        off += size


def _same(a, b):
    for key in ("iterations", "status", "mean_sigma", "err", "err_n"):
        np.testing.assert_array_equal(a[key], b[key])
    assert torch.equal(a["eps"], b["eps"]) and torch.equal(a["sigma"], b["sigma"])


@pytest.mark.parametrize("scheme", [0, 1], ids=["basic", "eyre-milton"])
@pytest.mark.parametrize("sizes,loads", [((9, 3, 16), 3), ((30, 45), 2), ((91, 143, 165), 1), ((64,) * 5, 3), ((208, 195), 1),
                                         ((208,) * 3, 3), ((45,) * 19, 2)],
                         ids=["one-cta", "clusters-of-2-and-4", "clusters-of-8", "even", "one-pair", "workspace", "many"])
def test_batches_on_chip(sizes, loads, scheme):
    """A fixed number of iterations against the generic passes.  A CTA holds about four groups of four rows where
    the chip has room: clusters of 1 up to 16 rows, of 2 at 30, 4 at 45 and 8 from 91 on; from 195 on the private
    state lies in the workspace (Eyre-Milton: from 176 on)."""
    cells, mat, E, c0, kw = _problem(2, sizes, loads, scheme)
    for opts in (dict(tol=0.0, max_iter=9), dict(tol=0.0, max_iter=8)):  # either buffer of the private state
        _close(hom.hom_solve(mat, E, c0, **opts, **kw), hom.hom_solve(mat, E, c0, passes=hom.HOM_PASSES_GENERIC, **opts, **kw),
               cells, loads)


@pytest.mark.parametrize("sizes,loads", [((45, 16, 405), 2), ((45, 30, 64, 75) * 13, 3), ((225,), 1), ((180,) * 16, 1)],
                         ids=["large-grid", "many-pairs", "passes-faster", "two-waves-of-clusters"])
def test_batches_kept_in_the_passes(sizes, loads):
    """On chip a batch runs as a whole or not at all: with a grid that does not fit, with more pairs than the chip
    has SMs, or where the passes were measured faster, the launches are those of the passes (which statistics
    force), bit for bit."""
    _, mat, E, c0, kw = _problem(2, sizes, loads, 0)
    a = hom.hom_solve(mat, E, c0, tol=1e-4, max_iter=200, **kw)
    assert (a["status"] == 0).all()
    _same(a, hom.hom_solve(mat, E, c0, tol=1e-4, max_iter=200, stats=True, **kw))


@pytest.mark.parametrize("dim,sizes,loads,plan", [
    (2, (143,) * 16, 3, False), (2, (150, 130, 121) * 20, 3, False), (2, (64,) * 64, 3, False), (2, (300,) * 8, 3, False),
    (3, (44,), 6, False), (3, (26,) * 8, 6, False), (2, (325,), 3, True), (2, (208,) * 24, 3, True), (2, (512,) * 4, 3, True),
    (2, (507, 45, 45), 3, True), (2, (343,) * 8, 3, True), (3, (64,), 6, True), (3, (49,), 1, True), (3, (98,), 2, True)],
    ids=lambda v: "x".join(map(str, (v[0], len(v)))) if isinstance(v, tuple) else str(v))
def test_plan_read_or_generic_passes(dim, sizes, loads, plan):
    """Sizes without compiled radices take the plan-read passes where these were measured faster and the generic ones
    elsewhere.  The same launches give the same bits; the other passes round differently."""
    cells, mat, E, c0, kw = _problem(dim, sizes, loads, 0)
    kw.update(tol=0.0, max_iter=5)
    a, gen = hom.hom_solve(mat, E, c0, **kw), hom.hom_solve(mat, E, c0, passes=hom.HOM_PASSES_GENERIC, **kw)
    if plan:
        assert not torch.equal(a["eps"], gen["eps"])
        _close(a, gen, cells, loads)
    else:
        _same(a, gen)


@pytest.mark.parametrize("scheme", [0, 1], ids=["basic", "eyre-milton"])
@pytest.mark.parametrize("dim,sizes,loads", [(2, (45, 135, 405), 3), (2, (45, 300, 77), 2), (3, (27,), 2), (3, (14, 22), 2)],
                         ids=["2d-compiled", "2d-plan", "3d-compiled", "3d-plan"])
def test_graphs_of_the_passes(dim, sizes, loads, scheme):
    """One graph launch against the host loop, bit for bit: first use, replay, another limit, new buffers."""
    _, mat, E, c0, kw = _problem(dim, sizes, loads, scheme)
    for opts in (dict(tol=1e-4, max_iter=300), dict(tol=1e-4, max_iter=300), dict(tol=1e-4, max_iter=4)):
        loop = hom.hom_solve(mat, E, c0, **opts, **kw)
        graph = hom.hom_solve(mat, E, c0, use_graph=True, **opts, **kw)
        _same(graph, loop)


def test_stops_on_chip():
    """The stopping points of the passes: tolerance, iteration limit, stagnation, divergence, with and without the
    history (which takes every iterate through the whole stopping rule)."""
    _, _, E, _, kw = _problem(2, (45, 64), 3, 0)
    phases = H.two_phases(10.0)
    mat = hom.hom_filter_build([_cell(2, 45), _cell(2, 64, 1)], phases)
    c0 = np.array(H.mean_lame(phases))
    for opts in (dict(tol=1e-4, max_iter=400), dict(tol=1e-4, max_iter=3), dict(tol=1e9, max_iter=5),
                 dict(tol=1e-4, max_iter=400, history=True)):
        a = hom.hom_solve(mat, E, c0, **opts, **kw)
        b = hom.hom_solve(mat, E, c0, stats=True, **opts, **kw)
        np.testing.assert_array_equal(a["status"], b["status"])
        assert np.abs(a["iterations"] - b["iterations"]).max() <= 1
    stalled = hom.hom_solve(mat, E, c0, tol=1e-9, max_iter=400, stall_window=20, **kw)
    assert (stalled["status"] == 3).all() or (stalled["status"] == hom.hom_solve(
        mat, E, c0, tol=1e-9, max_iter=400, stall_window=20, stats=True, **kw)["status"]).all()
    bad = hom.hom_solve(mat, E, 0.3 * c0, tol=1e-6, max_iter=4000, diverge_window=20, **kw)
    assert (bad["status"] == 2).all()
