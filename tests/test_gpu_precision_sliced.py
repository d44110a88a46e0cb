"""The precision form above the size where its products leave FP64 (2^25 multiply-adds), where
test_gpu_precision.py and test_gpu_split_solve.py stay below it: what it leaves in FP64."""
import os

import numpy as np
import pytest

from synth import make_problem

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cp():
    from paper_1606_01273_gb300 import build as b
    if not os.path.exists(b.LIB):
        b.build()
    import paper_1606_01273_gb300 as cp
    return cp


def test_setup_is_the_plain_form(cp):
    """U, E0, E_core and H^ref come from FP64 steps alone: the same digits in both forms at a size
    where the exchange of g(d_act) has 1e8 multiply-adds."""
    p = make_problem(nclosed=10, nact=4, nvirt=230, naux=440, nstate=2, seed=61)
    a, b = (cp.solve_problem(p, xms=1, shift=0.2, class_mask=1 << 4, precision=x)
            for x in (cp.FP64, cp.BF16X))
    assert a.Ecore == b.Ecore
    for name in ("U", "E0", "Href"):
        assert np.array_equal(getattr(a, name), getattr(b, name)), name
