"""Overlap cut of the class solves on the GPU: only the eigenvectors at or above ovl_thresh are
formed.  Cuts that keep everything but the null space, that fall inside the spectrum and that
keep nothing, for sectors on both eigensolver paths (rows up to 32 and above), against the
RDM-form oracle at the same cut."""
import os

import numpy as np
import pytest

from synth import make_problem
from oracle import o2_rdm as o2
from oracle import o2_classes as oc

pytestmark = pytest.mark.gpu

CASES = [dict(nclosed=3, nact=4, nvirt=5, naux=30, nstate=3, seed=34),     # rank-deficient A, C
         dict(nclosed=2, nact=3, nvirt=4, naux=24, nstate=1, seed=7, nelact=2)]
# class pieces in FP64: rounding of the sector transforms (about 1e-15 relative) times the
# conditioning of the kept overlap directions, which the cut bounds by |S| / thresh <= 1e4 for
# the cuts inside the spectrum; at 1e-9 the smallest kept eigenvalues of these cases are above
# 1e-5.  1e-9 leaves two orders of magnitude.
RTOL = 1e-9


@pytest.fixture(scope="module")
def cp():
    from paper_1606_01273_gb300 import build as b
    if not os.path.exists(b.LIB):
        b.build()
    import paper_1606_01273_gb300 as cp
    return cp


@pytest.mark.parametrize("thresh", [1e-9, 3e-3, 0.3, 1e4])
@pytest.mark.parametrize("scheme", ["msmr", "sssr"])
@pytest.mark.parametrize("case", range(len(CASES)))
def test_cut_matches_oracle(cp, case, scheme, thresh):
    p = make_problem(**CASES[case])
    st = o2.setup(p, xms=True, kmax=4)
    ref = oc.all_moments(p, st, shift=0.3, scheme=scheme, thresh=thresh)
    r = cp.solve_problem(p, xms=1, shift=0.3, ovl_thresh=thresh,
                         scheme=cp.MSMR if scheme == "msmr" else cp.SSSR)
    for cls in "ABCDEFG":
        M1, M2, _ = ref[cls]
        e, nr = -np.einsum("llk->lk", M1), np.diagonal(M2)
        if thresh == 1e4:
            assert not r.e_class[cls].any() and not r.norm_class[cls].any()
            continue
        scale = max(np.abs(e).max(), np.abs(nr).max(), 1e-12)
        assert np.abs(r.e_class[cls] - e).max() <= RTOL * scale, cls
        assert np.abs(r.norm_class[cls] - nr).max() <= RTOL * scale, cls
