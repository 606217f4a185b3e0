"""GPU tests: an operator with non-finite entries is refused, by every product that forms the factored matrix.

A user curve that repeats a node has a pair of nodes at distance zero, so its blocks hold NaN in two rows and
columns.  Partial pivoting then finds no pivot in the first column a NaN fills (BM_ESINGULAR, that column),
whichever product formed it: FP64 on the CUDA cores (N = 120), FP64 from digits (N = 256), split FP16.  Every
entry of the Schur complement's first column is NaN; the ordinary matrix has a finite first pivot row.
"""
import numpy as np
import pytest

import workloads as W
import oracle as O

pytestmark = pytest.mark.gpu


def _repeated_node(N):
    g = O.nodes(W.circle(), N)
    u = np.concatenate([g.x, g.dx, g.ddx], 1)
    u[0, :2] = u[1, :2]
    return u


@pytest.mark.parametrize("N", [120, 256])
@pytest.mark.parametrize("form,column", [(W.MIXED, 1), (W.ORDINARY, 2)])
@pytest.mark.parametrize("prec", [0, 1, 2])
def test_a_repeated_node_is_singular(bmlib, handle, N, form, column, prec):
    bmlib.bm_assemble(handle, bmlib.BM_CURVE_USER, (0, 0, 0, 0), N, 2.0, 3.0, form, bmlib.make_opts(prec),
                      user=_repeated_node(N))
    assert bmlib.bm_factor(handle) == column


# right-hand sides past FP32's range: the FP32 corrections are NaN, which is no convergence
@pytest.mark.parametrize("residual", ["BM_RESID_TC_UPDATE", "BM_RESID_DF_UPDATE", "BM_RESID_FP64_ALL", "BM_RESID_TC_ALL"])
@pytest.mark.parametrize("form", [W.MIXED, W.ORDINARY])
def test_an_overflowed_correction_does_not_converge(bmlib, handle, residual, form):
    N = 200
    c = W.ellipse(1.0, 0.6)
    bmlib.bm_assemble(handle, c.kind, c.params4(), N, 3.0, 4.5, form,
                      bmlib.make_opts(2, residual=getattr(bmlib, residual), refine_maxit=3))
    assert bmlib.bm_factor(handle) == 0
    B = np.full(((3 if form == W.MIXED else 2) * N, 1), 1e39 + 1e39j, order="F")
    info = bmlib.bm_solve(handle, B, np.zeros_like(B, order="F"), raise_on_notconv=False)
    assert info.backward_error == 1e300 and info.iterations == 3
