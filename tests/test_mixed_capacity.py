"""Room that hom_filter_build reserves for mixed voxels before it knows their number: enough for ordinary packs,
bounded by a quarter of the voxels (or 2^18 entries) for wide filters and overlapping primitives, and no error of
its own for cells that the library will refuse."""
import dataclasses
import math

import pytest
import torch

import hom_inputs as H

hom = pytest.importorskip("paper_1412_3228_gb300")


def _cell(dim=3, n=81, radius=0.2, radius_px=1.0, count=1, rule=H.RULE_VOIGT):
    kind = H.PRIM_DISK if dim == 2 else H.PRIM_SPHERE
    return H.Cell(dim, n, 0, [H.Primitive(kind, 1, (0.5, 0.5, 0.5), radius)] * count, rule, radius_px, 4)


@pytest.mark.parametrize("cell", [_cell(radius_px=20.0), _cell(count=200), _cell(n=135, radius_px=12.0, count=40),
                                  _cell(dim=2, n=1215, radius=0.1, radius_px=300.0)],
                         ids=["wide", "overlapping", "both", "2d"])
def test_room_is_bounded(cell):
    nvox = cell.n ** cell.dim
    assert hom._mixed_estimate([cell]) > nvox // 4
    assert hom._mixed_capacity([cell], nvox) <= max(nvox // 4, 1 << 18)


def test_ordinary_packs_fit_at_once():
    """A sphere of radius R voxels and a ball of radius r: the shell R - r .. R + r holds about 8 pi R^2 r voxels."""
    for n, count in ((64, 1), (135, 140), (243, 140)):
        cell = _cell(n=n, radius=0.085, count=count)
        mixed = count * 8.0 * math.pi * (0.085 * n) ** 2 * cell.radius_px
        assert mixed < hom._mixed_capacity([cell], n ** 3) <= max(n ** 3 // 4, 1 << 18)


BAD = [dict(radius=math.nan), dict(radius=math.inf), dict(radius=-1.0), dict(radius_px=math.nan),
       dict(radius_px=math.inf), dict(radius_px=-2.0)]


@pytest.mark.parametrize("bad", BAD + [dict(n=0), dict(dim=0, n=0)], ids=str)
def test_cells_to_be_refused_raise_nothing_here(bad):
    good = _cell(n=27)
    kw = {k: v for k, v in bad.items() if k in ("radius", "radius_px")}
    cell = dataclasses.replace(_cell(n=27, **kw), **{k: v for k, v in bad.items() if k in ("n", "dim")})
    room = hom._mixed_capacity([cell, good], 2 * 27 ** 3)
    assert 1024 <= room <= 1 << 18
    assert hom._mixed_estimate([good]) <= hom._mixed_estimate([cell, good]) <= 27 ** 3 + hom._mixed_estimate([good])


@pytest.mark.gpu
@pytest.mark.parametrize("bad", BAD, ids=str)
def test_the_library_refuses_them(bad):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1412_3228_gb300 import _build_lib
    _build_lib.build()
    with pytest.raises(hom.HomError) as err:
        hom.hom_filter_build([_cell(n=27, **bad)], H.two_phases(3.0))
    assert err.value.code == 1


@pytest.mark.gpu
def test_a_build_beyond_the_room_is_repeated():
    """A filter of 10 voxels about eight spheres of 13 at 108^3: about 8 x 4.19 (23^3 - 3^3) = 407 k mixed voxels, room
    for a quarter of the grid, 315 k."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1412_3228_gb300 import _build_lib
    _build_lib.build()
    at = (0.25, 0.75)
    prims = [H.Primitive(H.PRIM_SPHERE, 1, (x, y, z), 0.12) for x in at for y in at for z in at]
    cell = H.Cell(3, 108, 0, prims, H.RULE_VOIGT, 10.0, 1)
    mat = hom.hom_filter_build([cell], H.two_phases(3.0))
    assert mat.mixed_count > hom._mixed_capacity([cell], 108 ** 3)
    again = hom.hom_filter_build([cell], H.two_phases(3.0), capacity=108 ** 3)
    # the mixed bit is the sign of the 32-bit label
    assert again.mixed_count == mat.mixed_count and torch.equal(again.label < 0, mat.label < 0)
