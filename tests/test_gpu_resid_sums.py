"""GPU test of the digit residuals' sums over chunks of K (csrc/resid_tc.cu): 192 columns with nine digits, 256 with seven.

Sizes put K = N and 2N one below, at and one past a chunk and a block of 64, with one and with several K splits (16 and 48
right-hand sides: one column tile and more).  The refined solution is that of FP64 residuals: both stop at a backward
error of 1e-14 (nine digits), and the condition numbers here are below 1e4, so they agree to 1e-9; a
lost level, chunk or split would leave the residual wrong in its leading digits and the refinement above its target.
With seven digits the target is 1e-12, checked by the oracle's own FP64 residual.
"""
import numpy as np
import pytest

import workloads as W
import oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [95, 96, 97, 127, 128, 129, 192, 193, 257, 520])
@pytest.mark.parametrize("nrhs", [3, 48])
def test_chunk_edges(bmlib, handle, N, nrhs):
    c, k = W.ellipse(1.0, 0.6), 3.0
    B = np.asfortranarray(W.gaussian_full(3 * N, nrhs, N))
    X = {}
    for mode, tol in ((bmlib.BM_RESID_TC_ALL, 1e-14), (bmlib.BM_RESID_FP64_ALL, 1e-14), (bmlib.BM_RESID_TC_UPDATE, 1e-12)):
        bmlib.bm_assemble(handle, c.kind, c.params4(), N, k, 1.5 * k, W.MIXED,
                          bmlib.make_opts(2, refine_tol=tol, residual=mode))
        assert bmlib.bm_factor(handle) == 0
        X[mode] = np.zeros_like(B, order="F")
        assert bmlib.bm_solve(handle, B, X[mode]).backward_error <= tol
    ref = X[bmlib.BM_RESID_FP64_ALL]
    assert np.linalg.norm(X[bmlib.BM_RESID_TC_ALL] - ref) <= 1e-9 * np.linalg.norm(ref)
    blocks = O.mixed_blocks(O.nodes(c, N), O.default_params(k, 1.5 * k))
    assert O.backward_error_mixed(blocks, X[bmlib.BM_RESID_TC_UPDATE], B) <= 1.5e-12
