"""FP64 products at the edges of their 32 x 32 tiles (one row or column, 7, 8, 9, 31, 32, 33, 65),
either orientation, K below one chunk and split over a cluster: the densities of small active
spaces run every such product (integral blocks, sector transforms, slot Gram products, the DF
form), compared with the RDM-form oracle."""
import os

import numpy as np
import pytest

from synth import make_problem
from oracle import o2_rdm as o2
from oracle import o2_classes as oc

pytestmark = pytest.mark.gpu

# (closed, virtual, naux)
SIZES = [(1, 1, 5), (1, 33, 3), (7, 8, 300), (8, 9, 16), (9, 31, 130), (2, 65, 257), (31, 7, 33)]
RTOL = 1e-9        # the bound of the density tests: FP64 sums of up to 1e5 terms, well conditioned


@pytest.fixture(scope="module")
def cp():
    from paper_1606_01273_gb300 import build as b
    if not os.path.exists(b.LIB):
        b.build()
    import paper_1606_01273_gb300 as cp
    return cp


@pytest.mark.parametrize("c,v,X", SIZES)
def test_densities_at_tile_edges(cp, c, v, X):
    p = make_problem(nclosed=c, nact=2, nvirt=v, naux=X, nstate=2, seed=50 + c + v, nelact=2)
    st = o2.setup(p, xms=False, kmax=4)
    mom = oc.all_moments(p, st, shift=0.3)
    parts = {k: (-np.einsum("llk->lk", M1), np.diagonal(M2).copy())
             for k, (M1, M2, _) in mom.items()}
    _, _, R = o2.heff(st, parts, 0.3)
    d1, d2, gdf = 0.0, 0.0, 0.0
    for cls in "ABCDEFG":
        x1, xg, x2, _ = oc.class_densities(p, st, cls, 0.3, "msmr", R, 0)
        d1, d2, gdf = d1 + x1, d2 + x2, gdf + xg
    x2, xg, _ = o2.class_h_densities(p, st, R, 0, 0.3, "msmr")
    d2, gdf = d2 + x2, gdf + xg
    r = cp.solve_problem(p, densities=True, xms=0, shift=0.3)
    for got, ref, what in ((r.d1, d1, "d1"), (r.d2, d2, "d2"), (r.gdf, gdf, "gdf")):
        ref = 0.5 * (ref + np.swapaxes(ref, -1, -2))
        assert np.abs(got - ref).max() <= RTOL * max(1.0, np.abs(ref).max()), what
