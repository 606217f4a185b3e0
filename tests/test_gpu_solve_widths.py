"""GPU test: refined solves of different widths on one handle.

The iterate's digit planes keep the spacing of the widest solve so far (the tensor maps are made with the
workspace), so a narrower solve after a wide one has to write them with that spacing.
"""
import numpy as np
import pytest

import workloads as W
import oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("resid,tol", [(0, 1e-9), (4, 1e-14)])
def test_narrow_solve_after_a_wide_one(bmlib, handle, resid, tol):
    curve, N = W.star(1.0, 0.3, 5), 150
    bmlib.bm_assemble(handle, curve.kind, curve.params4(), N, 5.0, 7.5, bmlib.BM_MIXED,
                      bmlib.make_opts(bmlib.BM_CF32_3XTF32_IR, refine_tol=tol, residual=resid))
    assert bmlib.bm_factor(handle) == 0
    blocks = O.mixed_blocks(O.nodes(curve, N), O.default_params(5.0, 7.5))
    for nrhs in (70, 3, 40, 70, 1):
        B = np.asfortranarray(W.gaussian_full(3 * N, nrhs, nrhs))
        X = np.zeros_like(B, order="F")
        assert bmlib.bm_solve(handle, B, X).backward_error <= tol
        # 3e-14: the oracle's own FP64 residual at this size
        assert O.backward_error_mixed(blocks, X, B) <= 1.5 * tol + 3e-14
