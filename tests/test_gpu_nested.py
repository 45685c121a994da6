"""The resident nested solves (interior impedance) at the sizes where their form
changes: one right-hand side per cluster of 8 CTAs (up to 1,024 rows) and of 16
(up to 2,048), a cooperative grid beyond; fewer rows than CTAs; several
right-hand sides side by side (lockstep solves).

Cubes with n cells per side have 18 n^2 edges.  Reference: a dense solve with
the oracle's matrices (SIBC: RWG Gram matrix and I_x) or with the exported
near-region matrices (GIBC).  The nested FGMRES runs to 1e-12, so 1e-9 of the
result leaves room for the conditioning of the Gram matrix and of L_i,NR.
"""
import numpy as np
import pytest

from oracle import system
from oracle.rwg import Mesh
from oracle import mom
from synth import box, cn_vector

pytestmark = pytest.mark.gpu


def _dense(rp, col, val, n):
    A = np.zeros((n, n), complex)
    A[np.repeat(np.arange(n), np.diff(rp)), col] = val
    return A


@pytest.mark.parametrize("n,model", [(1, 1), (2, 1), (7, 1), (8, 1), (10, 1), (11, 1), (1, 0), (7, 0), (8, 0), (11, 0)])
def test_interior_impedance(lib, ctx, n, model):
    f, sigma = 10e9, 1e5
    V, T = box((1e-3, 1e-3, 1e-3), (n, n, n))
    m = Mesh(V, T)
    gm = lib.Mesh(ctx, V, T)
    op = lib.Operator(gm, f, 1.0, 1.0, sigma, lib.params(interior_model=model, tol_inner=1e-12, dense_pc_max=0,
                                                         grid_n=24))
    assert op.info()[9] == 1.0
    H = cn_vector(m.ne, 5, nrhs=2)
    Ix = system.Ix_sparse(m)
    if model == 1:
        want = system.eta_medium(f, 1.0, sigma) / system.ETA0 * np.linalg.solve(mom.gram(m), (Ix @ H.T)).T
    else:
        L, K = _dense(*op.near_csr(2), m.ne), _dense(*op.near_csr(3), m.ne)
        want = -np.linalg.solve(L, K @ H.T - 0.5 * (Ix @ H.T)).T / system.zscale(f, 1.0, sigma)
    got = op.matvec(lib.SIE_OP_ZI, H, nrhs=2)
    for q in range(2):
        assert np.linalg.norm(got[q] - want[q]) <= 1e-9 * np.linalg.norm(want[q])
    # inside the captured system product
    x = np.concatenate([H[0], cn_vector(m.nt, 6)])
    y = op.matvec(lib.SIE_OP_SYS, x)
    assert np.isfinite(y).all() and int(op.info()[16]) == 1
    assert op.stats()["inner_relres_max"] < 1e-12
    op.close()
    gm.close()


@pytest.mark.parametrize("n,nrhs", [(3, 3), (8, 2), (11, 3)])
def test_lockstep_panels(lib, ctx, n, nrhs):
    V, T = box((1e-3, 1e-3, 1e-3), (n, n, n))
    gm = lib.Mesh(ctx, V, T)
    op = lib.Operator(gm, 10e9, 1.0, 1.0, 1e5, lib.params(interior_model=1, tol_inner=1e-11, tol_outer=1e-8, grid_n=24,
                                                         restart=200))
    r = np.random.default_rng(4)
    k = r.standard_normal((nrhs, 3))
    k /= np.linalg.norm(k, axis=1, keepdims=True)
    e = np.cross(k, r.standard_normal((nrhs, 3)))
    b = op.rhs_planewave(k, e / np.linalg.norm(e, axis=1, keepdims=True))
    x, _, rr = op.solve(b, nrhs=nrhs)
    assert (rr < 1e-8).all()
    xs, _, _ = op.solve(b, nrhs=nrhs, sequential=True)
    for q in range(nrhs):  # both residuals below 1e-8, amplified by the conditioning
        assert np.linalg.norm(x[q] - xs[q]) <= 1e-5 * np.linalg.norm(xs[q])
    op.close()
    gm.close()
