"""Sector eigenbases of the one-launch solver (sectors of up to 96 rows) and its border with the
large-sector path: row counts 1, 2, 3, 8, 32, 96 (the largest of the one-block solver) and 100
(the first above it), both schemes, against the RDM-form oracle."""
import os

import numpy as np
import pytest

from synth import make_problem
from oracle import o2_rdm as o2
from oracle import o2_classes as oc

pytestmark = pytest.mark.gpu

# rows: D 2 a^2 n, B and F a^2 n, E and G a n (two families where the oracle counts them),
# A and C a^3 n; SS-SR takes n sectors of 1/n of the rows
CASES = {
    "a1n1": dict(nclosed=3, nact=1, nvirt=4, naux=20, nstate=1, seed=3, nelact=2),
    "a2n1": dict(nclosed=1, nact=2, nvirt=3, naux=20, nstate=1, seed=4, nelact=2),
    "a4n2": dict(nclosed=2, nact=4, nvirt=1, naux=24, nstate=2, seed=5),
    "a4n3": dict(nclosed=2, nact=4, nvirt=3, naux=24, nstate=3, seed=6),
    "a5n2": dict(nclosed=2, nact=5, nvirt=2, naux=24, nstate=2, seed=8, nelact=4),
}
# The class pieces carry the FP64 rounding of the sector transforms (1e-15) times |S| / thresh
# (below 1e5 at this cut): 1e-10, and a decade for the sums.
THRESH, RTOL = 1e-4, 1e-9


@pytest.fixture(scope="module")
def cp():
    from paper_1606_01273_gb300 import build as b
    if not os.path.exists(b.LIB):
        b.build()
    import paper_1606_01273_gb300 as cp
    return cp


@pytest.mark.parametrize("scheme", ["msmr", "sssr"])
@pytest.mark.parametrize("name", list(CASES))
def test_sector_sizes_match_oracle(cp, name, scheme):
    p = make_problem(**CASES[name])
    st = o2.setup(p, xms=True, kmax=4)
    ref = oc.all_moments(p, st, shift=0.3, scheme=scheme, thresh=THRESH)
    r = cp.solve_problem(p, xms=1, shift=0.3, ovl_thresh=THRESH,
                         scheme=cp.MSMR if scheme == "msmr" else cp.SSSR)
    for cls in "ABCDEFG":
        M1, M2, _ = ref[cls]
        e, nr = -np.einsum("llk->lk", M1), np.diagonal(M2)
        scale = max(np.abs(e).max(), np.abs(nr).max(), 1e-12)
        assert np.abs(r.e_class[cls] - e).max() <= RTOL * scale, cls
        assert np.abs(r.norm_class[cls] - nr).max() <= RTOL * scale, cls


@pytest.mark.parametrize("size", [dict(nclosed=13, nact=3, nvirt=108, naux=372, seed=5011),
                                  dict(nclosed=2, nact=3, nvirt=3, naux=24, seed=11),
                                  dict(nclosed=2, nact=3, nvirt=3, naux=24, seed=12),
                                  dict(nclosed=2, nact=2, nvirt=3, naux=24, seed=13)])
def test_sectors_without_overlap(cp, size):
    """Two active electrons: the antisymmetric sector of class F has no overlap, its matrix is
    rounding noise of 1e-17 whose reduction passes through elements of 1e-80 and below."""
    p = make_problem(nstate=2, nelact=2, **size)
    st = o2.setup(p, xms=True, kmax=4)
    M1, M2, _ = oc.class_moments(p, st, "F", shift=0.2)
    e, nr = -np.einsum("llk->lk", M1), np.diagonal(M2)
    r = cp.solve_problem(p, xms=1, shift=0.2)
    scale = max(np.abs(e).max(), np.abs(nr).max(), 1e-12)
    assert np.abs(r.e_class["F"] - e).max() <= RTOL * scale
    assert np.abs(r.norm_class["F"] - nr).max() <= RTOL * scale
