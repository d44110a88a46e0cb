"""The closed-active, active-virtual and closed-virtual blocks of dE/df: d(1), the derivative through
the one-electron part h = f - g(B, d_sa) alone (an f with those blocks is refused), from
caspt2_densities and from the determinant-space oracle."""
import os

import numpy as np
import pytest

from synth import make_problem
from oracle import o1_determinant as o1

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cp():
    from paper_1606_01273_gb300 import build as b
    if not os.path.exists(b.LIB):
        b.build()
    import paper_1606_01273_gb300 as cp
    return cp


@pytest.mark.parametrize("scheme", ["msmr", "sssr"])
def test_blocks_between_the_spaces(cp, scheme):
    p = make_problem(nclosed=2, nact=4, nvirt=2, naux=24, nstate=2, seed=5)
    c, a = p.nclosed, p.nact
    ctx = cp.Context(c, a, p.nvirt, p.naux, p.nstate, xms=0, shift=0.2,
                     scheme=cp.MSMR if scheme == "msmr" else cp.SSSR)
    try:
        ctx.set_inputs(*cp.problem_inputs(p))
        ctx.solve()
        d1, _, _ = ctx.densities()
        gf, _ = ctx.gradient()
    finally:
        ctx.close()
    between = np.ones_like(gf, dtype=bool)
    between[:c, :c] = between[c:c + a, c:c + a] = between[c + a:, c + a:] = False
    scale = np.abs(gf).max()
    assert np.abs(gf[between]).max() > 1e-3 * scale
    # the same sums, where the sources' adjoint adds with atomics
    assert np.abs((gf - d1)[between]).max() <= 1e-12 * scale
    r = o1.solve_problem(p, xms=False, scheme=scheme, shift=0.2)
    ref = 0.5 * (r.d1 + r.d1.T)
    assert np.abs((gf - ref)[between]).max() <= 1e-9 * scale
