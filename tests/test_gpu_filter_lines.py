"""Sample counts of the filter build at the edges of its line-by-line counting: lines longer than one
32-bit mask, lines whose both ends are outside a small primitive, overlapping primitives that share a
line, slabs along and across the lines, and primitives near half the cell, whose lines may wrap.  The
counts are exact integers of a fixed FP64 recipe, so they are compared for equality."""
import numpy as np
import pytest
import torch

import hom_inputs as H
import oracle as O

pytestmark = pytest.mark.gpu

hom = pytest.importorskip("paper_1412_3228_gb300")


def _disk(x, y, r, phase=1):
    return H.Primitive(H.PRIM_DISK, phase, (x, y, 0.0), r)


CASES = {
    # 2 S r = 31, 32, 33, 64, 136 half steps: one mask, just over one, several
    "len31": lambda: H.Cell(2, 15, 0, [_disk(0.5, 0.5, 0.2)], H.RULE_VOIGT, 31 / 32, 16),
    "len32": lambda: H.Cell(2, 15, 0, [_disk(0.41, 0.52, 0.25)], H.RULE_VOIGT, 1.0, 16),
    "len33": lambda: H.Cell(2, 15, 0, [_disk(0.41, 0.52, 0.25)], H.RULE_VOIGT, 33 / 32, 16),
    "len64": lambda: H.Cell(2, 15, 0, [_disk(0.3, 0.7, 0.21)], H.RULE_TWO_LAYER, 1.0, 32),
    "len136": lambda: H.Cell(2, 15, 0, [_disk(0.47, 0.5, 0.13)], H.RULE_REUSS, 1.7, 40),
    # disks much smaller than the ball (runs inside a line), overlapping, of two phases and in both orders
    "small": lambda: H.Cell(2, 27, 0, [_disk(0.31, 0.5, 0.012), _disk(0.5, 0.51, 0.02, 2), _disk(0.515, 0.5, 0.02)],
                            H.RULE_VOIGT, 1.6, 9),
    "nested": lambda: H.Cell(2, 27, 0, [_disk(0.5, 0.5, 0.1, 2), _disk(0.52, 0.5, 0.2), _disk(0.5, 0.5, 0.3, 2)],
                             H.RULE_VOIGT, 1.4, 8),
    # slabs normal to each axis, thinner than the ball; a disk that nearly fills the cell
    "slab-x": lambda: H.laminate_cell(27, 2, 0.03, axis=0, centre=0.513, rule=H.RULE_TWO_LAYER, subgrid=7),
    "slab-z": lambda: H.laminate_cell(9, 3, 0.11, axis=2, centre=0.02, rule=H.RULE_TWO_LAYER, subgrid=5),
    "wide": lambda: H.Cell(2, 45, 0, [_disk(0.93, 0.02, 0.47)], H.RULE_VOIGT, 1.3, 6),
    "sub1": lambda: H.Cell(3, 9, 0, [H.Primitive(H.PRIM_SPHERE, 1, (0.5, 0.4, 0.6), 0.25)], H.RULE_VOIGT, 2.0, 1),
    "sphere": lambda: H.Cell(3, 11, 0, [H.Primitive(H.PRIM_SPHERE, 1, (0.1, 0.4, 0.97), 0.31)], H.RULE_TWO_LAYER, 1.3, 13),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_counts_equal_the_recipe(name):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    cell = CASES[name]()
    phases = H.two_phases(10.0) + [H.lame_from_young(3.0, 0.2)]
    mat = hom.hom_filter_build([cell], phases)
    fb = O.filter_build(cell, phases)
    nm = mat.mixed_count
    assert nm == int(fb["mixed"].sum())
    counts = fb["counts"].reshape(-1, len(phases))
    vox = mat.mixed_voxel[:nm].cpu().numpy()
    ph = mat.mixed_phases[:2 * nm].cpu().numpy().reshape(-1, 2)
    np.testing.assert_array_equal(mat.mixed_frac[:nm].cpu().numpy(), counts[vox, ph[:, 1]] / fb["M"])
    label = mat.label.cpu().numpy().view(np.uint32)
    pure = (label & hom.HOM_MIXED_BIT) == 0
    np.testing.assert_array_equal(np.argmax(counts, axis=1)[pure], label[pure])


def test_small_table_is_rebuilt():
    """A table that is too small reports its size and the rebuilt one holds the same entries."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    cell = CASES["len64"]()
    phases = H.two_phases(10.0)
    a, b = hom.hom_filter_build([cell], phases), hom.hom_filter_build([cell], phases, capacity=3)
    assert a.mixed_count == b.mixed_count > 3
    pa = np.argsort(a.mixed_voxel[:a.mixed_count].cpu().numpy())
    pb = np.argsort(b.mixed_voxel[:b.mixed_count].cpu().numpy())
    ca = a.mixed_c64[:6 * a.mixed_count].cpu().numpy().reshape(-1, 6)[pa]
    cb = b.mixed_c64[:6 * b.mixed_count].cpu().numpy().reshape(-1, 6)[pb]
    np.testing.assert_array_equal(ca, cb)
