"""GPU test of the FP64 precision's digit products (csrc/resid_tc.cu gemm_z64_dg).

The Schur complement enters the FP64 solution; its tolerance against the oracle's FP64 solve is the
suite's 1e-10 for the FP64 path.  Sizes: below the rule's line (CUDA cores), beside tiles of 128 rows, 16
columns and 64 K entries, K splits and none; a budget without room for the workspace takes the CUDA cores
and gives the same solution; one that has room for it only until the solve's buffers gives it back.
"""
import numpy as np
import pytest

import workloads as W
import oracle as O
from oracle.dense import schur_solve

pytestmark = pytest.mark.gpu
DIGITS, CORES = "resid_tc_kernel (Schur complement)", "cgemm_simt_kernel<Z64> (Schur complement)"


def _run(bmlib, N, budget=0, nrhs=2):
    h = bmlib.bm_create(0, budget_bytes=budget)
    try:
        curve = W.kite()
        bmlib.bm_assemble(h, curve.kind, curve.params4(), N, 4.0 - 0.05j, 6.0 - 0.075j, bmlib.BM_MIXED, bmlib.make_opts(0))
        assert bmlib.bm_factor(h) == 0
        B = np.asfortranarray(W.gaussian_full(3 * N, nrhs, 4))
        X = np.zeros_like(B, order="F")
        info = bmlib.bm_solve(h, B, X)
        names = {k for k, _, _ in bmlib.bm_profile(h, B, np.zeros_like(B, order="F"))}
        held, limit = bmlib.bm_memory(h)
    finally:
        bmlib.bm_destroy(h)
    g, P = O.nodes(curve, N), O.default_params(4.0 - 0.05j, 6.0 - 0.075j)
    Xr = schur_solve(O.mixed_blocks(g, P), B)
    assert np.linalg.norm(X - Xr) < 1e-10 * np.linalg.norm(Xr)
    assert info.backward_error < 1e-13
    return names, held


@pytest.mark.parametrize("N,kernel", [(120, CORES), (177, DIGITS), (256, DIGITS), (257, DIGITS), (384, DIGITS),
                                      (500, DIGITS), (700, DIGITS)])
def test_schur_complement_by_digits(bmlib, N, kernel):
    names, _ = _run(bmlib, N)
    assert kernel in names and len({DIGITS, CORES} & names) == 1


def test_tight_budgets_keep_running(bmlib):
    N = 300
    _, held = _run(bmlib, N)
    a, x = 2 * 9 * N * 640 * 2, 27 * 304 * 640 * 2  # digit planes of Mbot and Mtop (K = 600 padded to 640)
    # without the planes' room: the CUDA cores from the start
    names, _ = _run(bmlib, N, budget=held - a - x)
    assert CORES in names and DIGITS not in names
    # room for everything but many right-hand sides: the planes go when the solve needs the room
    names, _ = _run(bmlib, N, budget=held + 4096, nrhs=60)
    assert CORES in names or DIGITS in names
