"""Split-BF16 products above the size where the precision form switches to them (2^25 FMAs), at
ragged edges of their 128 x 64 tiles, with one K chunk and several, against the plain FP64
form: the pair integrals (symmetric result, half of the tiles formed and mirrored), the DF
blocks and the density products."""
import os

import numpy as np
import pytest

from synth import make_problem

pytestmark = pytest.mark.gpu

# (closed, virtual, naux): (c v)^2 naux FMAs of the pair integrals are 67e6, 129e6 and 84e6
SIZES = [(9, 150, 37), (5, 131, 300), (4, 129, 320)]
RTOL = 1e-9        # the bound of the precision-form tests at 7 slices


@pytest.fixture(scope="module")
def cp():
    from paper_1606_01273_gb300 import build as b
    if not os.path.exists(b.LIB):
        b.build()
    import paper_1606_01273_gb300 as cp
    return cp


@pytest.mark.parametrize("c,v,X", SIZES)
def test_precision_form_equals_plain(cp, c, v, X):
    p = make_problem(nclosed=c, nact=2, nvirt=v, naux=X, nstate=2, seed=70 + c, nelact=2)
    a = cp.solve_problem(p, densities=True, xms=1, shift=0.3)
    b = cp.solve_problem(p, densities=True, xms=1, shift=0.3, precision=cp.BF16X, slices=7)
    for cls in "ABCDEFGH":
        for x, y in ((a.e_class[cls], b.e_class[cls]), (a.norm_class[cls], b.norm_class[cls])):
            assert np.abs(x - y).max() <= RTOL * max(1.0, np.abs(x).max()), cls
    for k in ("d1", "d2", "gdf"):
        x, y = getattr(a, k), getattr(b, k)
        assert np.abs(x - y).max() <= RTOL * max(1.0, np.abs(x).max()), k
