"""Class H of the plain form from eight BF16 slices (sizes above 2^26 multiply-adds) against the
oracle: odd and ragged edges, one and several chunks of closed orbitals, nact 0, both schemes, a
closed-orbital range, and a NaN in the closed-virtual factors, which stays an error."""
import os

import numpy as np
import pytest

from synth import make_problem
from oracle import o2_rdm as o2

pytestmark = pytest.mark.gpu

# cv^2 naux: 8.3e7 (one chunk), 7.7e8, 2.6e9 with cv^2 above 2^24 (two chunks)
CASES = {
    "c5v99": dict(nclosed=5, nact=0, nvirt=99, naux=340, nstate=1, seed=31),
    "c13v131a2": dict(nclosed=13, nact=2, nvirt=131, naux=271, nstate=2, seed=32, nelact=2),
    "c33v127": dict(nclosed=33, nact=0, nvirt=127, naux=150, nstate=1, seed=33),
}
# FP64 rounding of the sums (1e-16 sqrt(terms)) and 2^-53 sqrt(naux) of K: below 1e-12
RTOL = 1e-11


@pytest.fixture(scope="module")
def cp():
    from paper_1606_01273_gb300 import build as b
    if not os.path.exists(b.LIB):
        b.build()
    import paper_1606_01273_gb300 as cp
    return cp


@pytest.mark.parametrize("scheme", ["msmr", "sssr"])
@pytest.mark.parametrize("name", list(CASES))
def test_sliced_class_h(cp, name, scheme):
    p = make_problem(**CASES[name])
    st = o2.setup(p, xms=True, kmax=2)
    M1, M2, _ = o2.class_h_moments(p, st, shift=0.2, scheme=scheme)
    e, nr = -np.einsum("llk->lk", M1), np.diagonal(M2)
    opt = dict(xms=1, shift=0.2, class_mask=1 << 7,
               scheme=cp.MSMR if scheme == "msmr" else cp.SSSR)
    r = cp.solve_problem(p, **opt)
    assert np.abs(r.e_class["H"] - e).max() <= RTOL * np.abs(e).max()
    assert np.abs(r.norm_class["H"] - nr).max() <= RTOL * np.abs(nr).max()
    mid = p.nclosed // 2
    parts = [cp.solve_problem(p, closed_begin=x, closed_end=y, **opt)
             for x, y in ((0, mid), (mid, p.nclosed))]
    both = sum(q.e_class["H"] for q in parts)
    assert np.abs(both - e).max() <= RTOL * np.abs(e).max()


def test_nan_stays_an_error(cp):
    p = make_problem(**CASES["c5v99"])
    p.B[7, 2, p.nclosed + 40] = p.B[7, p.nclosed + 40, 2] = np.nan
    with pytest.raises(cp.CASPT2Error):
        cp.solve_problem(p, shift=0.2)
