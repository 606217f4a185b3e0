"""GPU tests: optional workspaces (the search-free LU's buffer, FP64's digit workspace) under a tight budget.

They are taken at bm_factor where the budget has room beside the system, yield to a solve that needs the room, and
are taken again at the next bm_factor.  So nothing that fits without them is refused, and a factorisation does not
depend on what the handle solved before: the same bits.
"""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu
N, K, MANY = 300, 4.0, 120


class _Run:
    def __init__(self, bmlib, form, prec, budget=0):
        self.bm, self.rows = bmlib, (3 if form == W.MIXED else 2) * N
        self.h = bmlib.bm_create(0, budget_bytes=budget)
        self.empty = self.held()
        c = W.kite()
        bmlib.bm_assemble(self.h, c.kind, c.params4(), N, K, 1.5 * K, form, bmlib.make_opts(prec))
        self.system = self.held()

    def held(self):
        return self.bm.bm_memory(self.h)[0]

    def factor(self):
        assert self.bm.bm_factor(self.h) == 0
        return self.held()

    def solve(self, ncols):
        B = np.asfortranarray(W.gaussian_full(self.rows, ncols, 3))
        X = np.zeros_like(B, order="F")
        self.bm.bm_solve(self.h, B, X)
        return X

    def close(self):
        self.bm.bm_destroy(self.h)


def _sizes(bmlib, form, prec):
    r = _Run(bmlib, form, prec)
    try:
        optional = r.factor() - r.system
        r.solve(MANY)
        return r.system, optional, r.held() - r.system - optional
    finally:
        r.close()


@pytest.mark.parametrize("form", [W.MIXED, W.ORDINARY])
@pytest.mark.parametrize("prec", [0, 2])
def test_a_factorisation_does_not_depend_on_earlier_solves(bmlib, form, prec):
    system, optional, solve = _sizes(bmlib, form, prec)
    assert optional > 0
    r = _Run(bmlib, form, prec, system + max(optional, solve))
    try:
        first = r.factor()
        assert first == system + optional
        x = r.solve(2)
        r.solve(MANY)  # does not fit beside the optional workspaces
        assert r.held() < system + optional + solve  # some were given back
        r.factor()
        assert np.array_equal(r.solve(2), x)
    finally:
        r.close()


@pytest.mark.parametrize("form", [W.MIXED, W.ORDINARY])
@pytest.mark.parametrize("prec", [0, 2])
@pytest.mark.parametrize("spare", [0, 0.5])
def test_what_fits_without_them_runs(bmlib, form, prec, spare):
    system, optional, solve = _sizes(bmlib, form, prec)
    r = _Run(bmlib, form, prec, system + solve + int(spare * optional) // 256 * 256)
    try:
        r.factor()
        r.solve(MANY)
        r.factor()
    finally:
        r.close()
