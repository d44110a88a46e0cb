"""Partial solves with an empty closed-orbital range (more partitions than closed orbitals): no pairs
of class H and no tuples of class G, classes A-F where the range starts at 0; the moments of the
partitions add up to those of the whole solve."""
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


# the fused kernel and, above 2^26 multiply-adds, the sliced one
@pytest.mark.parametrize("size", [dict(nclosed=3, nact=2, nvirt=6, naux=24),
                                  dict(nclosed=5, nact=2, nvirt=99, naux=340)])
@pytest.mark.parametrize("precision", [0, 1])
def test_empty_ranges(cp, size, precision):
    p = make_problem(nstate=2, seed=3, nelact=2, **size)
    c = p.nclosed

    def moments(lo, hi):
        ctx = cp.Context(c, p.nact, p.nvirt, p.naux, p.nstate, xms=1, shift=0.2,
                         precision=precision, closed_begin=lo, closed_end=hi)
        try:
            ctx.set_inputs(*cp.problem_inputs(p))
            ctx.solve()
            return ctx.moments()
        finally:
            ctx.close()

    whole = moments(0, -1)
    scale = np.abs(whole).max(axis=1, keepdims=True)
    cuts = [0, 2, 2, c, c]
    parts = {(lo, hi): moments(lo, hi) for lo, hi in zip(cuts, cuts[1:])}
    assert not parts[2, 2].any() and not parts[c, c].any()
    assert (np.abs(sum(parts.values()) - whole) <= 1e-11 * scale).all()
    # an empty range at 0 carries classes A-F alone
    first = moments(0, 0)
    assert not first[6:].any()
    assert (np.abs(first - whole)[:6] <= 1e-11 * scale[:6]).all()
