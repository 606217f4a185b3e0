"""GPU tests: factors of an ordinary system whose block rows differ in size.

beta scales the first block row (D - I/2 + beta N, S + beta (D* + I/2)) against the second, so rows of U12 have two
sizes, the lower rows of L21 are about 1 / beta, and a block of columns where the block rows meet holds both.  The
products take a scale per row, per column and (inner_exponent) per column of L21.

CF32: FP32 factors leave about 1e-6 of the error per correction, so three reach a backward error of 1e-14; a fixed
scale for L21 took seven at beta = 2^30 i / k.  FP64: each component of the solution to 1e-11 of numpy's for the
row-equilibrated matrix (condition numbers below 1e4 leave 1e-12 for either); digits without the inner scale are off by
1e-7.  Sizes: the block rows meet at a block edge of the LU (256, 512) and inside a block; FP64 trailing updates by digits.
"""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nb", [0, 128, 256])
@pytest.mark.parametrize("N", [200, 256, 300])
@pytest.mark.parametrize("scale", [2.0 ** 10, 2.0 ** 20, 2.0 ** 30])
def test_far_beta(bmlib, handle, N, nb, scale):
    c = W.ellipse(1.0, 0.6)
    bmlib.bm_assemble(handle, c.kind, c.params4(), N, 4.0, 6.0, W.ORDINARY,
                      bmlib.make_opts(2, nb=nb, beta=0.25j * scale, refine_tol=1e-14, residual=bmlib.BM_RESID_FP64_ALL))
    assert bmlib.bm_factor(handle) == 0
    B = np.asfortranarray(W.gaussian_full(2 * N, 3, 5))
    info = bmlib.bm_solve(handle, B, np.zeros_like(B, order="F"))
    assert info.backward_error <= 1e-14 and info.iterations <= 3


@pytest.mark.parametrize("N", [450, 512, 600])
@pytest.mark.parametrize("scale", [2.0 ** 20, 2.0 ** 30])
def test_far_beta_fp64(bmlib, handle, N, scale):
    c = W.ellipse(1.0, 0.6)
    bmlib.bm_assemble(handle, c.kind, c.params4(), N, 4.0, 6.0, W.ORDINARY, bmlib.make_opts(0, beta=0.25j * scale))
    assert bmlib.bm_factor(handle) == 0
    B = np.asfortranarray(W.gaussian_full(2 * N, 3, 5))
    X = np.zeros_like(B, order="F")
    bmlib.bm_solve(handle, B, X)
    A = np.zeros((2 * N, 2 * N), dtype=np.complex128, order="F")
    bmlib.bm_copy_block(handle, 0, A)
    r = 1.0 / np.abs(A).max(axis=1)
    ref = np.linalg.solve(A * r[:, None], B * r[:, None])
    for s in (slice(0, N), slice(N, 2 * N)):
        assert np.linalg.norm(X[s] - ref[s]) <= 1e-11 * np.linalg.norm(ref[s])
