"""Overlap cut on the large-matrix eigensolver (more than 96 rows a sector): rank-deficient classes
A and C of 125 rows under SS-SR and 250 under MS-MR, cuts that keep everything but the null space,
that fall inside the spectrum and that keep nothing, against the RDM-form oracle at the same cut."""
import os

import numpy as np
import pytest

from synth import make_problem
from oracle import o2_rdm as o2
from oracle import o2_classes as oc

pytestmark = pytest.mark.gpu

CASE = dict(nclosed=2, nact=5, nvirt=3, naux=24, nstate=2, seed=9, nelact=4)
# rounding of the sector transforms (1e-15) times |S| / smallest kept eigenvalue (16 / 5e-4 where only
# the null space is cut): 5e-11; the cuts lie at least two per cent from an eigenvalue
RTOL = 1e-9


@pytest.fixture(scope="module")
def cp():
    from paper_1606_01273_gb300 import build as b
    if not os.path.exists(b.LIB):
        b.build()
    import paper_1606_01273_gb300 as cp
    return cp


@pytest.mark.parametrize("thresh", [1e-9, 7.5e-3, 0.3, 1e4])
@pytest.mark.parametrize("scheme", ["msmr", "sssr"])
def test_cut_matches_oracle(cp, scheme, thresh):
    p = make_problem(**CASE)
    st = o2.setup(p, xms=True, kmax=4)
    r = cp.solve_problem(p, xms=1, shift=0.3, ovl_thresh=thresh, class_mask=0b101,
                         scheme=cp.MSMR if scheme == "msmr" else cp.SSSR)
    for cls in "AC":
        M1, M2, _ = oc.class_moments(p, st, cls, shift=0.3, scheme=scheme, thresh=thresh)
        e, nr = -np.einsum("llk->lk", M1), np.diagonal(M2)
        if thresh == 1e4:
            assert not r.e_class[cls].any() and not r.norm_class[cls].any()
            continue
        scale = max(np.abs(e).max(), np.abs(nr).max())
        assert np.abs(r.e_class[cls] - e).max() <= RTOL * scale, cls
        assert np.abs(r.norm_class[cls] - nr).max() <= RTOL * scale, cls
