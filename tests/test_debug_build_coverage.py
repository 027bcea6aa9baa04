"""The bounds-checked build covers every kernel that takes dynamic shared memory: each declaration of it in the
sources is joined by the poisoning (a read of an element nobody wrote then shows up as NaN) and by a check of the
task or pair the kernel was given."""
import glob
import os

import pytest

from conftest import ROOT

SOURCES = sorted(glob.glob(os.path.join(ROOT, "paper_1412_3228_gb300", "csrc", "*.cu")))


@pytest.mark.parametrize("path", SOURCES, ids=[os.path.basename(p) for p in SOURCES])
def test_kernels_with_dynamic_shared_memory_are_poisoned_and_checked(path):
    body = open(path).read().split("extern __shared__")
    for before, after in zip(body, body[1:]):
        assert "HOM_DBG_POISON();" in before[-200:] + after[:1200], before[-200:]
    if len(body) > 1:
        assert body[-1].count("HOM_CHECK(") >= 1
