"""GPU tests of the FP32 LU in blocks without a pivot search (csrc/lu_fast.cu).

Every case is a refined solve whose backward error the oracle recomputes with its own FP64 operator.
Tolerance: the library stops at 1e-9 by its own estimate, which differs from the oracle's only by the
FP32 rounding of the norms, hence 1.5e-9 (as in test_gpu_solve).  The profile shows lu_trsm_kernel when
the search-free blocks ran and swap_trsm_kernel when the pivot search did.
"""
import numpy as np
import pytest

import workloads as W
import oracle as O

pytestmark = pytest.mark.gpu
FREE, SEARCH = "lu_trsm_kernel", "swap_trsm_kernel (block row)"


FREE_Z = "lu_trsm_z_kernel"


def _solve(bmlib, curve, N, k0, k1, form, opts, seed=3, ncols=5):
    h = bmlib.bm_create(0)
    try:
        bmlib.bm_assemble(h, curve.kind, curve.params4(), N, k0, k1, form, opts)
        assert bmlib.bm_factor(h) == 0
        nsys = (3 if form == W.MIXED else 2) * N
        B = np.asfortranarray(W.gaussian_full(nsys, ncols, seed))
        X = np.zeros_like(B, order="F")
        info = bmlib.bm_solve(h, B, X)
        kernels = {name for name, _, _ in bmlib.bm_profile(h, B, X)}
    finally:
        bmlib.bm_destroy(h)
    g, P = O.nodes(curve, N), O.default_params(k0, k1)
    eta = (O.backward_error_mixed(O.mixed_blocks(g, P), X, B) if form == W.MIXED
           else O.backward_error_dense(O.ordinary_matrix(g, P), X, B))
    if opts.prec == bmlib.BM_FP64:
        assert info.backward_error < 1e-13 and eta < 1e-13  # the suite's bound for the FP64 path
    else:
        assert info.backward_error <= 1e-9 and eta <= 1.5e-9
    return kernels


# block 128, sub-step 16, chunk 32, 32 or 64 rows per CTA: sizes at and beside each edge; 2N doubles them
@pytest.mark.parametrize("prec", [1, 2])
@pytest.mark.parametrize("form,N", [(0, n) for n in (8, 15, 17, 33, 127, 128, 129, 160, 256, 257, 385, 1100)] +
                                   [(1, n) for n in (8, 64, 65, 97, 320)])
def test_block_edges(bmlib, prec, form, N):
    kernels = _solve(bmlib, W.circle(), N, 2.0, 3.0, form, bmlib.make_opts(prec))
    assert FREE in kernels and SEARCH not in kernels


# FP64: block 32, sub-step 8, outer block 128 (digits above 265 rows), 16 rows per CTA
@pytest.mark.parametrize("form,N", [(0, n) for n in (8, 9, 31, 32, 33, 40, 127, 128, 129, 160, 161, 257, 420)] +
                                   [(1, n) for n in (8, 16, 17, 64, 66, 210)])
def test_fp64_block_edges(bmlib, form, N):
    kernels = _solve(bmlib, W.circle(), N, 2.0, 3.0, form, bmlib.make_opts(0))
    assert FREE_Z in kernels and SEARCH not in kernels


# partial pivoting interchanges rows of these systems, first in the column given: in the first block, in a
# later one, near the end; inside a diagonal block and below it
@pytest.mark.parametrize("curve,N,k0,form", [
    (W.ellipse(1.0, 0.6), 400, 5.2294051420988685 - 1.3485554180016592j, 0),   # column 47
    (W.ellipse(1.0, 0.6), 400, 5.009682014750906 - 1.281903136008821j, 0),     # column 161
    (W.ellipse(1.0, 0.6), 400, 4.901444581998341 - 1.0794051420988682j, 1),    # column 657 of 800
    (W.kite(), 600, 30.0 - 0.6j, 1),                                           # column 790 of 1200
])
@pytest.mark.parametrize("prec", [0, 2])
def test_interchanges_continue_with_the_search(bmlib, curve, N, k0, form, prec):
    kernels = _solve(bmlib, curve, N, k0, 1.5 * k0, form, bmlib.make_opts(prec))
    assert (FREE if prec else FREE_Z) in kernels and SEARCH in kernels


def test_an_explicit_block_size_keeps_the_search(bmlib):
    kernels = _solve(bmlib, W.star(1.0, 0.3, 5), 300, 6.0, 9.0, 0, bmlib.make_opts(2, nb=128))
    assert FREE not in kernels and SEARCH in kernels
