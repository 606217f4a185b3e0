"""GPU test: FP64 solutions are as accurate with digit products (csrc/resid_tc.cu) as with FP64 multiply-adds.

Two handles solve the same system, one with room for the digit workspace and one without (its products run on the
CUDA cores).  Their errors are taken against a solution refined in extended precision from the same FP64 blocks.
Digits and level sums are exact to far below FP64's rounding, so the digit products' error has to be no larger;
a factor 2 is left for the factorisation, whose rounding differs between the two (errors of equal size and
independent sign).  Sums held in pairs of FP32 were 3 to 7 times worse at these sizes.
"""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu
DIGITS = "resid_tc_kernel (Schur complement)"


def _solve(bmlib, curve, N, k, budget, B):
    h = bmlib.bm_create(0, budget_bytes=budget)
    try:
        bmlib.bm_assemble(h, curve.kind, curve.params4(), N, k, 1.5 * k, W.MIXED, bmlib.make_opts(0))
        assert bmlib.bm_factor(h) == 0
        held = bmlib.bm_memory(h)[0]
        X = np.zeros_like(B, order="F")
        bmlib.bm_solve(h, B, X)
        blocks = [np.zeros((N, N), dtype=np.complex128, order="F") for _ in range(4)]
        for q, b in enumerate(blocks):
            bmlib.bm_copy_block(h, q, b)
        names = {name for name, _, _ in bmlib.bm_profile(h, B, np.zeros_like(B, order="F"))}
    finally:
        bmlib.bm_destroy(h)
    return X, blocks, held, names


def _refined(blocks, B):
    M13, M23, M31, M32 = blocks
    N = M13.shape[0]
    Ui = np.linalg.inv(-(M31 @ M13) - M32 @ M23)
    m13, m23, m31, m32 = (b.astype(np.clongdouble) for b in blocks)
    b3 = B[2 * N:].astype(np.clongdouble)  # (b1 = b2 = 0)
    z = np.zeros_like(b3)
    for _ in range(3):
        r = b3 + m31 @ (m13 @ z) + m32 @ (m23 @ z)
        z = z + (Ui @ r.astype(np.complex128)).astype(np.clongdouble)
    return np.concatenate([-(m13 @ z), -(m23 @ z), z])


@pytest.mark.parametrize("curve,N,k", [(W.star(1.0, 0.3, 5), 700, 8.0), (W.kite(), 1000, 10.0),
                                       (W.ellipse(1.0, 0.6), 1000, 4.0)])
def test_digits_are_as_accurate_as_fp64(bmlib, curve, N, k):
    B = np.zeros((3 * N, 2), dtype=np.complex128, order="F")
    B[2 * N:] = W.gaussian_full(N, 2, 3)
    Xd, blocks, held, names = _solve(bmlib, curve, N, k, 0, B)
    assert DIGITS in names
    Xc, _, _, names = _solve(bmlib, curve, N, k, held - 1, B)
    assert DIGITS not in names
    ref = _refined(blocks, B)
    for q in range(3):
        s = slice(q * N, (q + 1) * N)
        ed, ec = (np.linalg.norm((X[s] - ref[s]).astype(np.complex128)) for X in (Xd, Xc))
        assert ed <= 2.0 * ec
