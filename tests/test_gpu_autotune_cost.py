"""What a caller waits for in the first tuned solve of a batch shape: ten trial iterations for each of the four
candidate plans, also where the grid runs on chip or in three dimensions."""
import re

import numpy as np
import pytest
import torch

import hom_inputs as H

pytestmark = pytest.mark.gpu

hom = pytest.importorskip("paper_1412_3228_gb300")


@pytest.mark.parametrize("dim,n", [(2, 63), (2, 416), (3, 22)])
def test_trial_iterations_of_a_tuned_solve(dim, n):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1412_3228_gb300 import _build_lib
    _build_lib.build()
    phases = H.two_phases(5.0)
    kind = H.PRIM_DISK if dim == 2 else H.PRIM_SPHERE
    mat = hom.hom_filter_build([H.Cell(dim, n, 0, [H.Primitive(kind, 1, (0.5, 0.5, 0.5), 0.3)], H.RULE_NONE, 1.0, 4)], phases)
    hom.hom_solve(mat, np.eye(3 if dim == 2 else 6), H.mean_lame(phases), precision=hom.HOM_FP32,
                  criterion=hom.HOM_CRIT_EN, tol=1e-3, max_iter=100, tune=True)
    line = [ln for ln in hom.hom_autotune_report().splitlines()
            if ("dim%d " % dim) in ln and ln.split(":")[0].endswith(" %dx1" % n)]
    assert len(line) == 1 and line[0].count(" ms") == 4
    count = re.search(r"\((\d+) trial iterations\)", line[0])
    assert count and int(count.group(1)) <= 4 * 10, line[0]
