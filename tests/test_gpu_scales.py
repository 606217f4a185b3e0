"""GPU tests: scaling the problem by powers of two scales its solution.

Permittivities scaled by 2^j scale M32 by 2^j and M23 by 2^-j and nothing else; every FP64 and FP32 operation commutes
with that (nothing leaves the normal range here), so the products of scaled operands (digit planes, split FP16
packs) have to as well: u and phi keep their bits, q takes 2^-j.  One FP32 correction (refine_maxit = 1) shows the
CF32 factors themselves.  A curve scaled by L = 2^j with wavenumbers divided by L scales M13 and M32 by L, but for the
rounding of the diagonals' logarithms (2^-52 of them): with condition numbers below 1e4, 1e-11 is left
for FP64.  One scale per row of [M31 M32] that takes the blocks as they come loses the smaller block's low bits:
1e-9 at L = 2^-20 in FP64, no convergence at 2^-30 in CF32.  Sizes: CUDA-core and digit products of the FP64
Schur complement, odd and even halves.
"""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def _run(bmlib, N, L, opts):
    h = bmlib.bm_create(0)
    try:
        c = W.ellipse(L, 0.625 * L)
        bmlib.bm_assemble(h, c.kind, c.params4(), N, 3.0 / L, 4.5 / L, W.MIXED, opts)
        blocks = [np.zeros((N, N), dtype=np.complex128, order="F") for _ in range(4)]
        for q, b in enumerate(blocks):
            bmlib.bm_copy_block(h, q, b)
        assert bmlib.bm_factor(h) == 0
        B = np.zeros((3 * N, 3), dtype=np.complex128, order="F")
        B[2 * N:] = W.gaussian_full(N, 3, 7)
        X = np.zeros_like(B, order="F")
        info = bmlib.bm_solve(h, B, X, raise_on_notconv=False)
    finally:
        bmlib.bm_destroy(h)
    return blocks, [X[q * N:(q + 1) * N] for q in range(3)], info


@pytest.mark.parametrize("N", [120, 256, 301])
@pytest.mark.parametrize("prec", [0, 2])
@pytest.mark.parametrize("scale", [2.0 ** 40, 2.0 ** -30, 0.5])
def test_permittivities(bmlib, N, prec, scale):
    def run(eps0):
        return _run(bmlib, N, 1.0, bmlib.make_opts(prec, eps0=eps0, refine_maxit=1, refine_tol=1e-30,
                                                   residual=bmlib.BM_RESID_FP64_ALL))
    b0, x0, _ = run(1.25)
    b1, x1, _ = run(1.25 * scale)
    for a, b, f in zip(b0, b1, (1.0, 1.0 / scale, 1.0, scale)):
        assert np.array_equal(a * f, b)  # the premise
    for a, b, f in zip(x0, x1, (1.0, 1.0 / scale, 1.0)):
        assert np.array_equal(a * f, b)


@pytest.mark.parametrize("N", [120, 256, 301])
@pytest.mark.parametrize("L", [2.0 ** -10, 2.0 ** -20, 2.0 ** -30, 2.0 ** 12])
def test_lengths(bmlib, N, L):
    _, x0, _ = _run(bmlib, N, 1.0, bmlib.make_opts(0))
    _, x1, _ = _run(bmlib, N, L, bmlib.make_opts(0))
    opts = bmlib.make_opts(2, refine_tol=1e-14, residual=bmlib.BM_RESID_FP64_ALL)
    _, xc, info = _run(bmlib, N, L, opts)
    for a, b, f in zip(x0, x1, (1.0, 1.0 / L, 1.0 / L)):
        assert np.abs(a * f - b).max() <= 1e-11 * np.abs(b).max()
    # FP32 factors leave about 1e-6 of the error per correction (test_gpu_split_products)
    assert info.backward_error <= 1e-14 and info.iterations <= 3
