"""Sources and their adjoints at every state count the kernels are specialised for (one to four
in registers, five and six through the general variants), with three shared loops in the
groups of classes A and C: class pieces and densities against the RDM-form oracle."""
import os

import numpy as np
import pytest

from synth import make_problem
from oracle import o2_rdm as o2
from oracle import o2_classes as oc

pytestmark = pytest.mark.gpu

# densities: the bound of the density tests (FP64 sums, kept overlap eigenvalues above 1e-4
# of the largest at this cut)
THRESH, RTOL = 1e-4, 1e-9


@pytest.fixture(scope="module")
def cp():
    from paper_1606_01273_gb300 import build as b
    if not os.path.exists(b.LIB):
        b.build()
    import paper_1606_01273_gb300 as cp
    return cp


def expected(n):
    p = make_problem(nclosed=2, nact=4, nvirt=3, naux=40, nstate=n, seed=60 + n)
    st = o2.setup(p, xms=True, kmax=4)
    mom = oc.all_moments(p, st, shift=0.3, thresh=THRESH)
    parts = {k: (-np.einsum("llk->lk", M1), np.diagonal(M2).copy())
             for k, (M1, M2, _) in mom.items()}
    _, _, R = o2.heff(st, parts, 0.3)
    d1, d2, gdf = 0.0, 0.0, 0.0
    for cls in "ABCDEFG":
        x1, xg, x2, _ = oc.class_densities(p, st, cls, 0.3, "msmr", R, 0, thresh=THRESH)
        d1, d2, gdf = d1 + x1, d2 + x2, gdf + xg
    x2, xg, _ = o2.class_h_densities(p, st, R, 0, 0.3, "msmr")
    return p, parts, (d1, d2 + x2, gdf + xg)


@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 6])
def test_state_counts(cp, n):
    p, parts, dens = expected(n)
    r = cp.solve_problem(p, densities=True, xms=1, shift=0.3, ovl_thresh=THRESH)
    for cls, (e, nr) in parts.items():
        assert np.abs(r.e_class[cls] - e).max() <= RTOL * max(1.0, np.abs(e).max()), cls
        assert np.abs(r.norm_class[cls] - nr).max() <= RTOL * max(1.0, np.abs(nr).max()), cls
    for got, ref, what in zip((r.d1, r.d2, r.gdf), dens, ("d1", "d2", "gdf")):
        ref = 0.5 * (ref + np.swapaxes(ref, -1, -2))
        assert np.abs(got - ref).max() <= RTOL * max(1.0, np.abs(ref).max()), what
