"""The precision form above the size where its products leave FP64 (2^25 multiply-adds), where
test_gpu_precision.py and test_gpu_split_solve.py stay below it: what it leaves in FP64, the slice
counts and a row-range product."""
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


@pytest.fixture(scope="module")
def reference():
    """c9 a2 v150 X60 n2: the pair integrals have 1.1e8 multiply-adds, the rows of four closed
    orbitals 4.9e7, the virtual Gram products 2.7e8: all above the switch."""
    from test_gpu_precision import _oracle
    p = make_problem(nclosed=9, nact=2, nvirt=150, naux=60, nstate=2, seed=62, nelact=2)
    opt = dict(xms=1, scheme=0, shift=0.2)
    return p, opt, _oracle(p, opt)


@pytest.mark.parametrize("slices,etol,drel", [(7, 1e-9, 1e-9), (5, 1e-8, 1e-6)])
def test_sliced_products_vs_oracle(cp, reference, slices, etol, drel):
    """The bounds of test_gpu_precision.py, at sizes where the slices carry them."""
    p, opt, (parts, w, d1, d2, G) = reference
    r = cp.solve_problem(p, densities=True, precision=cp.BF16X, slices=slices, **opt)
    for cls, (e, nr) in parts.items():
        assert np.abs(r.e_class[cls] - e).max() <= etol * max(1.0, np.abs(e).max()), cls
    assert np.abs(r.Ems - w).max() <= etol * max(1.0, np.abs(w).max())
    for got, ref, name in ((r.d1, d1, "d1"), (r.d2, d2, "d2"), (r.gdf, G, "GDF")):
        assert np.linalg.norm(got - ref) <= drel * np.linalg.norm(ref), name


def test_the_slices_are_used(cp, reference):
    """Five and seven slices differ in class H and in the densities."""
    p, opt, _ = reference
    a, b = (cp.solve_problem(p, densities=True, precision=cp.BF16X, slices=s, **opt) for s in (5, 7))
    assert not np.array_equal(a.e_class["H"], b.e_class["H"])
    assert np.linalg.norm(a.d2 - b.d2) > 1e-14 * np.linalg.norm(b.d2)


@pytest.mark.parametrize("slices", [5, 7])
def test_closed_ranges_of_sliced_products(cp, reference, slices):
    """Partial solves over two closed ranges (row-range products, not symmetric) add up to the whole
    one; an element of K has the same slices in either, so the sums' rounding is all that differs."""
    from paper_1606_01273_gb300.shard import closed_range
    p, opt, _ = reference
    opt = dict(opt, precision=cp.BF16X, slices=slices, class_mask=1 << 7)
    whole = cp.solve_problem(p, **opt)
    parts = []
    for r in range(2):
        lo, hi = closed_range(p.nclosed, r, 2)
        parts.append(cp.solve_problem(p, closed_begin=lo, closed_end=hi, **opt))
    for name in ("e_class", "norm_class"):
        both, one = sum(getattr(q, name)["H"] for q in parts), getattr(whole, name)["H"]
        assert np.abs(both - one).max() <= 1e-12 * np.abs(one).max(), name
