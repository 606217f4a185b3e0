"""GPU tests: a handle assembled again with another LU path (block size given or not) factors by that path.

A captured factorisation holds the path it was captured with, and in FP64 the default block size is the one the
pivot search uses, so buffers and sizes alone do not tell the two apart.  Each factorisation of a reused handle
has to give the bits of a fresh handle with the same options; the interchanging system (first interchange in
column 161) leaves a search-free sequence unfinished unless it is continued.
"""
import numpy as np
import pytest

import workloads as W
import oracle as O

pytestmark = pytest.mark.gpu
CASES = {
    "interchanges": (W.ellipse(1.0, 0.6), 400, 5.009682014750906 - 1.281903136008821j),
    "no interchange": (W.circle(), 200, 2.0),
}


def _factor_solve(bmlib, h, case, form, prec, nb, B):
    curve, N, k = CASES[case]
    bmlib.bm_assemble(h, curve.kind, curve.params4(), N, k, 1.5 * k, form, bmlib.make_opts(prec, nb=nb))
    l0 = bmlib.bm_kernel_launches(h)
    assert bmlib.bm_factor(h) == 0
    launches = bmlib.bm_kernel_launches(h) - l0
    X = np.zeros_like(B, order="F")
    bmlib.bm_solve(h, B, X)
    return X, launches


@pytest.mark.parametrize("case", list(CASES))
@pytest.mark.parametrize("form", [W.MIXED, W.ORDINARY])
# the block sizes that equal a default: 64 in FP64, 256 in FP32
@pytest.mark.parametrize("prec,nb", [(0, 64), (2, 256)])
def test_reassembled_with_another_block_size(bmlib, case, form, prec, nb):
    curve, N, k = CASES[case]
    B = np.asfortranarray(W.gaussian_full((3 if form == W.MIXED else 2) * N, 2, 3))
    fresh = {}
    for b in (0, nb):
        h = bmlib.bm_create(0)
        try:
            fresh[b] = _factor_solve(bmlib, h, case, form, prec, b, B)
        finally:
            bmlib.bm_destroy(h)
    g, P = O.nodes(curve, N), O.default_params(k, 1.5 * k)
    eta = (O.backward_error_mixed(O.mixed_blocks(g, P), fresh[0][0], B) if form == W.MIXED
           else O.backward_error_dense(O.ordinary_matrix(g, P), fresh[0][0], B))
    assert eta < (1e-13 if prec == 0 else 1.5e-9)  # the suite's bounds
    for order in ((0, nb, 0), (nb, 0, nb)):
        h = bmlib.bm_create(0)
        try:
            for b in order:
                X, launches = _factor_solve(bmlib, h, case, form, prec, b, B)
                assert np.array_equal(X, fresh[b][0])
                assert launches == fresh[b][1]
        finally:
            bmlib.bm_destroy(h)
