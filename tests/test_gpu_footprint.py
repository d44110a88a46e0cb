"""Device memory: a server's contexts stay within the smallest budget that it accepts them at, and
a context whose optional class-H workspace does not fit solves without it."""
import gc
import os

import numpy as np
import pytest

from synth import make_problem

pytestmark = pytest.mark.gpu

MB = 1 << 20


@pytest.fixture(scope="module")
def cp():
    from paper_1606_01273_gb300 import build as b
    if not os.path.exists(b.LIB):
        b.build()
    import paper_1606_01273_gb300 as cp
    return cp


def _free():
    import torch
    gc.collect()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.cuda.mem_get_info()[0]


def _serve(cp, p, budget, densities, opt):
    """Bytes held by the idle context of one served request, or None where it is refused."""
    before = _free()
    srv = cp.Server(budget_bytes=budget, slots=1)
    try:
        try:
            t = srv.submit(p, densities=densities, **opt)
        except cp.CASPT2Error as e:
            assert e.status == cp.EINVAL
            return None
        assert srv.wait(t)["status"] >= 0
        return before - _free()
    finally:
        srv.close()


# shapes whose footprint is in the parts that grow apart: slices and chunk of class H, source
# groups of three loops and their G, split products, sectors
SHAPES = {
    "c60a1v200": (dict(nclosed=60, nact=1, nvirt=200, naux=400, nstate=1, seed=3, nelact=2), False,
                  {}),
    "c40a2v300": (dict(nclosed=40, nact=2, nvirt=300, naux=400, nstate=1, seed=4, nelact=2), False,
                  {}),
    "c8a6v60": (dict(nclosed=8, nact=6, nvirt=60, naux=220, nstate=3, seed=5), True, {}),
    "c12a4v100bf16x": (dict(nclosed=12, nact=4, nvirt=100, naux=340, nstate=2, seed=6), True,
                       dict(precision=1, slices=7)),
}


@pytest.mark.parametrize("name", list(SHAPES))
def test_server_stays_within_its_budget(cp, name):
    size, densities, opt = SHAPES[name]
    opt = dict(xms=1, shift=0.2, **opt)
    p = make_problem(**size)
    held = _serve(cp, p, 0, densities, opt)            # modules loaded, nothing refused
    assert held > 0
    lo, hi = held // 8, 8 * held + 256 * MB
    assert _serve(cp, p, hi, densities, opt) is not None
    for _ in range(12):
        mid = (lo + hi) // 2
        used = _serve(cp, p, mid, densities, opt)
        if used is None:
            lo = mid
        else:
            assert used <= mid
            hi = mid


def _fill(leave):
    import torch
    return torch.empty(max(0, _free() - leave), dtype=torch.uint8, device="cuda")


def test_optional_workspace_gives_way(cp):
    """Memory for a context without the sliced class-H workspace (K chunk and slices), then for
    its densities without it: both calls succeed with the results of a whole one."""
    c, v, X = 40, 300, 400
    p = make_problem(nclosed=c, nact=2, nvirt=v, naux=X, nstate=1, seed=4, nelact=2)
    cv = c * v
    optional = 8 * min(cv * cv, max(1 << 24, cv * v)) + 16 * cv * ((X + 31) // 32 * 32)
    opt = dict(xms=1, shift=0.2)

    def solve(dens, fill_create=None, fill_dens=None):
        """Result and the bytes held after the solve and after the densities."""
        gc.collect()
        keep = [_fill(fill_create)] if fill_create else []
        f0 = _free()
        ctx = cp.Context(c, 2, v, X, 1, **opt)
        try:
            ctx.set_inputs(*cp.problem_inputs(p))
            r = ctx.result(ctx.solve())
            f1 = _free()
            if dens:
                keep += [_fill(fill_dens)] if fill_dens else []
                f2 = _free()
                r.d1, r.d2, r.gdf = ctx.densities()
            return r, f0 - f1, (f2 - _free()) if dens else 0
        finally:
            ctx.close()
            keep.clear()
            _free()                                     # gives the filling back

    ref, held, grown = solve(True)
    slack = 48 * MB                                     # rounding of the allocations
    r, _, _ = solve(False, fill_create=held - optional + slack)
    q, _, _ = solve(True, fill_dens=grown - optional + slack)
    for got in (r, q):
        assert np.abs(got.Ems - ref.Ems).max() <= 1e-11 * np.abs(ref.Ems).max()
        assert np.abs(got.e_class["H"] - ref.e_class["H"]).max() <= 1e-11 * np.abs(
            ref.e_class["H"]).max()
    for k in ("d1", "d2", "gdf"):
        a, b = getattr(q, k), getattr(ref, k)
        assert np.linalg.norm(a - b) <= 1e-10 * np.linalg.norm(b), k
