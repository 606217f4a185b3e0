"""GPU test: a search-free LU that meets an interchange goes on with the pivot search from that block.

The profile counts the search's outer panels (one row-interchange launch each): from the block that holds the
first interchange on (blocks of 32 columns in FP64, of 128 in FP32), not from the first column.  The block is
restored and, in FP64, the products of its outer block's earlier blocks are applied to the rest before: the solution's
backward error by the oracle's own operator is the suite's.
"""
import numpy as np
import pytest

import workloads as W
import oracle as O

pytestmark = pytest.mark.gpu
SEARCH = "swap_trsm_kernel (block row)"


# partial pivoting interchanges rows first in this column (test_gpu_lu_fast): early and late in an outer block of 128
# columns, at its start (160 is its second block), inside a diagonal block and below it
@pytest.mark.parametrize("curve,N,k0,form,column", [
    (W.ellipse(1.0, 0.6), 400, 5.2294051420988685 - 1.3485554180016592j, W.MIXED, 47),
    (W.ellipse(1.0, 0.6), 400, 5.009682014750906 - 1.281903136008821j, W.MIXED, 161),
    (W.ellipse(1.0, 0.6), 400, 4.901444581998341 - 1.0794051420988682j, W.ORDINARY, 657),
    (W.kite(), 600, 30.0 - 0.6j, W.ORDINARY, 790),
])
@pytest.mark.parametrize("prec,block,panel", [(0, 32, 64), (2, 128, 256)])
def test_the_search_starts_at_the_block(bmlib, handle, curve, N, k0, form, column, prec, block, panel):
    bmlib.bm_assemble(handle, curve.kind, curve.params4(), N, k0, 1.5 * k0, form, bmlib.make_opts(prec))
    assert bmlib.bm_factor(handle) == 0
    n = N if form == W.MIXED else 2 * N
    B = np.asfortranarray(W.gaussian_full((3 if form == W.MIXED else 2) * N, 3, 11))
    X = np.zeros_like(B, order="F")
    bmlib.bm_solve(handle, B, X)
    g, P = O.nodes(curve, N), O.default_params(k0, 1.5 * k0)
    eta = (O.backward_error_mixed(O.mixed_blocks(g, P), X, B) if form == W.MIXED
           else O.backward_error_dense(O.ordinary_matrix(g, P), X, B))
    assert eta < (1e-13 if prec == 0 else 1.5e-9)
    launches = {name: k for name, k, _ in bmlib.bm_profile(handle, B, np.zeros_like(B, order="F"))}
    left = n - (column - 1) // block * block
    assert launches[SEARCH] == -(-left // panel)
