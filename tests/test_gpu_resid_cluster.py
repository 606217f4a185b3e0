"""GPU test of the nine-digit tensor-core residual over its cluster shapes (csrc/resid_tc.cu).

16 right-hand sides per column tile and one to five tiles per cluster: 1 and 16 columns (one tile), 17
(two), 40 (three), 64 (four), 70 (five), 90 (six tiles in threes), 100 (seven in fours, one of them
empty).  Tolerance: the library stops at a backward error of 1e-14 by a residual exact to 2^-64 of the
scales; the oracle recomputes it in FP64, whose own residual is good to about 300 x 2^-53 = 3e-14 in the
same normalisation.
"""
import numpy as np
import pytest

import workloads as W
import oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("form", [0, 1])
@pytest.mark.parametrize("nrhs", [1, 16, 17, 40, 64, 70, 90, 100])
def test_nine_digit_residual_cluster_shapes(bmlib, handle, form, nrhs):
    curve, N, k0, k1 = W.ellipse(1.0, 0.6), 150, 5.0 - 0.1j, 7.5 - 0.15j
    bmlib.bm_assemble(handle, curve.kind, curve.params4(), N, k0, k1, form,
                      bmlib.make_opts(bmlib.BM_CF32_3XTF32_IR, refine_tol=1e-14, residual=bmlib.BM_RESID_TC_ALL))
    assert bmlib.bm_factor(handle) == 0
    g, P = O.nodes(curve, N), O.default_params(k0, k1)
    B = np.asfortranarray(W.gaussian_full((3 if form == 0 else 2) * N, nrhs, 11))
    X = np.zeros_like(B, order="F")
    info = bmlib.bm_solve(handle, B, X)
    assert info.backward_error <= 1e-14
    eta = (O.backward_error_mixed(O.mixed_blocks(g, P), X, B) if form == 0
           else O.backward_error_dense(O.ordinary_matrix(g, P), X, B))
    assert eta <= 1e-14 + 3e-14
