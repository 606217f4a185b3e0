"""GPU tests of the split FP16 products (csrc/gemm_tc.cu) and what feeds them, through refined solves.

Sizes lie at and beside the edges of the packs (32 K), the tiles (128), the persistent updates (more tiles than
SMs are out of reach of the oracle; two tiles per CTA come from a full size in test_gpu_fullsize), and the items of the
triangular solve (64 rows, 8 right-hand sides).  A permittivity far from 1 scales M32 against M31: the
packs have to keep both.  Tolerance: as in test_gpu_lu_fast (the library stops at 1e-9 by its own estimate, the
oracle recomputes it with its own operator).  A product that lost its low parts would need more
corrections: with both parts the first one leaves about 2^-22 K^(1/2) of growth-scaled error, so two suffice.
"""
import numpy as np
import pytest

import workloads as W
import oracle as O

pytestmark = pytest.mark.gpu


def _check(bmlib, N, form, opts, P, ncols, k=(3.0, 4.5)):
    curve = W.ellipse(1.0, 0.6)
    h = bmlib.bm_create(0)
    try:
        bmlib.bm_assemble(h, curve.kind, curve.params4(), N, *k, form, opts)
        assert bmlib.bm_factor(h) == 0
        B = np.asfortranarray(W.gaussian_full((3 if form == 0 else 2) * N, ncols, N))
        X = np.zeros_like(B, order="F")
        info = bmlib.bm_solve(h, B, X)
    finally:
        bmlib.bm_destroy(h)
    g = O.nodes(curve, N)
    eta = (O.backward_error_mixed(O.mixed_blocks(g, P), X, B) if form == 0
           else O.backward_error_dense(O.ordinary_matrix(g, P), X, B))
    assert info.backward_error <= 1e-9 and eta <= 1.5e-9
    return info


@pytest.mark.parametrize("prec", [1, 2])
@pytest.mark.parametrize("nb", [0, 32, 256])
@pytest.mark.parametrize("form,N,ncols", [(0, 31, 1), (0, 33, 8), (0, 64, 9), (0, 200, 17), (0, 385, 65), (1, 65, 7),
                                          (1, 193, 16)])
def test_pack_and_tile_edges(bmlib, prec, nb, form, N, ncols):
    info = _check(bmlib, N, form, bmlib.make_opts(prec, nb=nb), O.default_params(3.0, 4.5), ncols)
    assert info.iterations <= 2


# eps0 scales M32 and 1 / eps1 scales M23: one scale per pack row would cost M31 its low parts
@pytest.mark.parametrize("eps0", [2.0 ** -20, 0.75, 3.0, 1e6])
@pytest.mark.parametrize("N", [65, 129])
def test_far_permittivity(bmlib, eps0, N):
    info = _check(bmlib, N, 0, bmlib.make_opts(2, eps0=eps0), O.default_params(3.0, 4.5, eps0=eps0), 5)
    assert info.iterations <= 2
