"""Class H of the plain form where eight slices would hold an element of K to fewer digits than its
FP64 dot product does: factor rows that are graded over P in opposite directions, and a range of
closed orbitals whose own pairs are as small as those elements.  The sums are those of an FP64 dot
product, against extended precision; rows without a common P and zero rows as well."""
import os

import numpy as np
import pytest

from synth import make_problem
from oracle import o2_rdm as o2

pytestmark = pytest.mark.gpu

C, V, X = 5, 99, 340                  # c v^2 X: 8.3e7 multiply-adds, above the switch to slices
# 2^-53 sqrt(X) of an element whose terms are of its own size (2e-15), in a sum of 4e4 elements
RTOL = 1e-13


@pytest.fixture(scope="module")
def cp():
    from paper_1606_01273_gb300 import build as b
    if not os.path.exists(b.LIB):
        b.build()
    import paper_1606_01273_gb300 as cp
    return cp


def _problem(nact, nstate, scale):
    """scale [P][i]: factors of the closed-virtual rows."""
    p = make_problem(nclosed=C, nact=nact, nvirt=V, naux=X, nstate=nstate, seed=31,
                     **(dict(nelact=2) if nact else {}))
    vo = C + nact
    p.B[:, :C, vo:] = (np.random.default_rng(5).standard_normal((X, C, V)) * scale[:, :, None])
    p.B[:, vo:, :C] = p.B[:, :C, vo:].transpose(0, 2, 1)
    return p


def _first_orbital(p, st, shift):
    """Moments of the pairs (0, j >= 0), j > 0 twice, in extended precision."""
    n, vo = p.nstate, C + p.nact
    eps = np.diag(p.f).astype(np.longdouble)
    B = p.B[:, :C, vo:].astype(np.longdouble)
    K = np.einsum("Pa,Pjb->ajb", B[:, 0], B)
    num = K * (2 * K - K.transpose(2, 1, 0))
    num[:, 1:] *= 2
    D = eps[vo:, None, None] + eps[vo:] - eps[0] - eps[:C, None]
    om, W = np.linalg.eigh(0.5 * (st.Ftil + st.Ftil.T))
    M1, M2 = np.zeros((n, n, n)), np.zeros((n, n))
    for L in range(n):
        for nu in range(n):
            d = D + shift + om[nu] - st.E0[L]
            M1[L] += np.outer(W[:, nu], W[:, nu]) * float((num / d).sum())
            M2[L] += W[:, nu] * W[L, nu] * float((num / d ** 2).sum())
    return M1, M2


P = np.arange(X)[:, None] / X
DOWN, UP = P, P[::-1]


def _opposite(decades):
    """Orbital 0 falls over P, the others rise, larger by what the product loses."""
    s = 10.0 ** (-decades * np.concatenate([DOWN] + [UP] * (C - 1), 1))
    s[:, 1:] *= 10.0 ** decades
    return s


def _disjoint():
    s = np.ones((X, C))
    s[X // 2:, 0] = 0.0
    s[:X // 2, 1:] = 0.0
    return s


def _zero_rows():
    s = np.ones((X, C))
    s[:, 2] = 0.0
    return s


SCALES = {"graded_10": _opposite(10), "graded_25": _opposite(25), "disjoint": _disjoint(),
          "zero_rows": _zero_rows(), "even": np.ones((X, C))}


@pytest.mark.parametrize("nact,nstate", [(0, 1), (2, 2), (3, 3)])
@pytest.mark.parametrize("name", list(SCALES))
def test_range_of_small_pairs(cp, name, nact, nstate):
    p = _problem(nact, nstate, SCALES[name])
    st = o2.setup(p, xms=True, kmax=2)
    M1, M2 = _first_orbital(p, st, 0.2)
    r = cp.solve_problem(p, xms=1, shift=0.2, class_mask=1 << 7, closed_begin=0, closed_end=1)
    e, nr = -np.einsum("llk->lk", M1), np.diagonal(M2)
    assert np.abs(r.e_class["H"] - e).max() <= RTOL * np.abs(e).max()
    assert np.abs(r.norm_class["H"] - nr).max() <= RTOL * np.abs(nr).max()
