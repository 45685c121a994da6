"""Blocks of right-hand sides take other projection, interpolation and near-region
kernels than single vectors: past 4,096 triangles times right-hand sides 4 lanes
per triangle and per-triangle coefficients, and the CSR panel's groups of 2, 4 and
8 lanes.  Every column has to be the product of its vector alone, up to the order
of FP64 sums: 1e-13 of the added terms (a few hundred terms of 1.1e-16 each).
"""
import numpy as np
import pytest

from synth import box, cn_vector

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cube(lib, ctx):
    V, T = box((1e-2, 1e-2, 1e-2), (10, 10, 10))  # 1,200 triangles, 1,800 edges
    gm = lib.Mesh(ctx, V, T)
    op = lib.Operator(gm, 3e9, 3.0, 1.0, 0.02, lib.params(dense_pc_max=0))
    assert op.info()[9] == 0.0
    yield gm, op
    op.close()
    gm.close()


@pytest.mark.parametrize("nrhs", [2, 3, 4, 5, 7, 8, 9])
def test_block_columns(lib, cube, nrhs):
    gm, op = cube
    X = cn_vector(gm.ne, 50 + nrhs, nrhs=nrhs)
    for which in (0, 1, 2, 3):
        rp, col, val = op.near_csr(which)
        rows = np.repeat(np.arange(gm.ne), np.diff(rp))
        Y = op.matvec(which, X, nrhs=nrhs)
        for q in range(nrhs):
            y = op.matvec(which, np.ascontiguousarray(X[q]))
            terms = np.linalg.norm(np.bincount(rows, weights=np.abs(val * X[q][col]), minlength=gm.ne))
            assert np.linalg.norm(Y[q] - y) <= 1e-13 * (terms + np.linalg.norm(y))


def test_system_product_sizes(lib, ctx):
    """1,200 (32 lanes) and 4,332 triangles (4 lanes): the FP64 and the complex64
    product agree to FP32 accuracy on both (rounding of the FP32 sums and of the
    cancelling precorrection, below 1e-4 as on the benchmark's coarse spheres)."""
    for n in (10, 19):
        V, T = box((1e-2, 1e-2, 1e-2), (n, n, n))
        gm = lib.Mesh(ctx, V, T)
        op = lib.Operator(gm, 3e9, 1.0, 1.0, 1e5, lib.params(dense_pc_max=0, interior_model=1, tol_inner=1e-10))
        x = cn_vector(gm.ne + gm.nt, 3)
        y = op.matvec(lib.SIE_OP_SYS, x)
        again = op.matvec(lib.SIE_OP_SYS, x)
        assert np.array_equal(y, again)  # gather projection, two addends per edge: replays are equal
        op.set_solver(precision=lib.SIE_MIXED, tol_inner=1e-10)
        z = op.matvec(lib.SIE_OP_SYS, x)
        assert np.linalg.norm(z[:gm.ne] - y[:gm.ne]) <= 1e-4 * np.linalg.norm(y[:gm.ne])
        op.close()
        gm.close()
