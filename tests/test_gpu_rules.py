"""Quadrature rules and solver controls that take the less travelled branches.

* More than 8 angular points (exponentials evaluated instead of tabulated) and panels so
  short that a point's edges have hundreds (several lists per point): the default rule's
  angular error is about rho^-16 = 5e-11, rho = 4.4 for panels of 1.5 and poles at
  +-i pi / 2, so both agree with it to 1e-9.
* More units than fit the list at 32 outer points each (2^18): units of 64 points.  Two
  neighbouring, far finer outer rules on either side of that line agree to 1e-8.
* Restarted constraint solves (constraint_restart 1 and 2): the outer solution is the
  same to the outer tolerance.
* A tetrahedron (6 edges, 4 triangles): fewer rows than CTAs in every resident kernel.
"""
import numpy as np
import pytest

from oracle import mom, system
from oracle.rwg import Mesh
from synth import cn_vector, icosphere

pytestmark = pytest.mark.gpu


def _entries(lib, ctx, sigma, **rule):
    mesh = lib.Mesh(ctx, *icosphere(1, 0.01))
    op = lib.Operator(mesh, 3e9, 4.0, 1.0, sigma, lib.params(dense_pc_max=0, **rule))
    assert op.info()[9] == 0.0
    v = [op.near_csr(w)[2] for w in range(4)]
    op.close()
    mesh.close()
    return v


@pytest.mark.parametrize("rule", [{"q_ang": 9}, {"q_ang": 12}, {"q_alen": 0.05}])
@pytest.mark.parametrize("sigma", [0.0, 0.1])
def test_angular_rules(lib, ctx, sigma, rule):
    for a, b in zip(_entries(lib, ctx, sigma, **rule), _entries(lib, ctx, sigma)):
        assert np.abs(a - b).max() <= 1e-9 * np.abs(b).max()


def test_long_units(lib, ctx):
    T = icosphere(1, 0.01)[1]
    shared = (T[:, None, :, None] == T[None, :, None, :]).sum(axis=(2, 3))

    def units(q):  # runs of 32 outer points of every pair, as if all were close
        ge = q["q_opan"] * q["q_olam"] * 2 * q["q_emupan"] * q["q_emu"]
        points = {0: 25, 1: q["q_opan"] * q["q_olam"] * 6, 2: ge, 3: 3 * ge}
        return sum(int((shared == n).sum()) * -(-p // 32) for n, p in points.items())

    a, b = ({"q_opan": 14, "q_olam": 10, "q_emupan": 6, "q_emu": n} for n in (9, 12))
    assert units(a) < 2**18 < units(b) - 10000  # fewer pairs than that are far
    for u, v in zip(_entries(lib, ctx, 0.0, **a), _entries(lib, ctx, 0.0, **b)):
        assert np.abs(u - v).max() <= 1e-8 * np.abs(v).max()


@pytest.mark.parametrize("restart", [1, 2])
def test_restarted_constraint_solve(lib, ctx, restart):
    mesh = lib.Mesh(ctx, *icosphere(1, 0.01, equal_volume=True))
    op = lib.Operator(mesh, 3e9, 4.0, 1.0, 0.0, lib.params(tol_outer=1e-8, tol_inner=1e-10))
    b = op.rhs_planewave([0, 0, -1.0], [1.0, 0, 0])
    want, _, _ = op.solve(b)
    # three iterations to 1e-13
    op.set_solver(tol_outer=1e-8, tol_inner=1e-10, tol_constraint=1e-13, constraint_restart=restart, constraint_maxit=40)
    got, _, rr = op.solve(b)
    assert op.stats()["constraint_iters_max"] > restart and rr < 1e-8
    assert np.linalg.norm(got - want) <= 1e-5 * np.linalg.norm(want)
    op.close()
    mesh.close()


@pytest.mark.parametrize("model", [0, 1])
def test_tetrahedron(lib, ctx, model):
    V = 1e-3 * np.array([[1, 1, 1], [1, -1, -1], [-1, 1, -1], [-1, -1, 1]], float)
    T = np.array([[0, 1, 2], [0, 2, 3], [0, 3, 1], [1, 3, 2]], np.int32)
    n = np.cross(V[T[:, 1]] - V[T[:, 0]], V[T[:, 2]] - V[T[:, 0]])
    assert ((n * V[T].mean(axis=1)).sum(axis=1) > 0).all()
    m = Mesh(V, T)
    mesh = lib.Mesh(ctx, V, T)
    f, sigma = 10e9, 1e5
    op = lib.Operator(mesh, f, 1.0, 1.0, sigma, lib.params(interior_model=model, tol_inner=1e-12, tol_outer=1e-9))
    assert op.info()[9] == 1.0
    H = cn_vector(m.ne, 5)
    Ix = system.Ix_sparse(m)

    def dense(w):
        rp, col, val = op.near_csr(w)
        A = np.zeros((m.ne, m.ne), complex)
        A[np.repeat(np.arange(m.ne), np.diff(rp)), col] = val
        return A

    if model == 1:
        want = system.eta_medium(f, 1.0, sigma) / system.ETA0 * np.linalg.solve(mom.gram(m), Ix @ H)
    else:
        want = -np.linalg.solve(dense(2), dense(3) @ H - 0.5 * (Ix @ H)) / system.zscale(f, 1.0, sigma)
    got = op.matvec(lib.SIE_OP_ZI, H)
    assert np.linalg.norm(got - want) <= 1e-9 * np.linalg.norm(want)
    k, e = np.array([[0, 0, -1.0], [0, 1.0, 0]]), np.array([[1.0, 0, 0], [0, 0, 1.0]])
    b = op.rhs_planewave(k, e)
    x, _, rr = op.solve(b, nrhs=2)
    xs, _, rs = op.solve(b, nrhs=2, sequential=True)
    assert (rr < 1e-9).all() and (rs < 1e-9).all()
    assert np.linalg.norm(x - xs) <= 1e-5 * np.linalg.norm(xs)
    op.close()
    mesh.close()
