"""Grid products at every FFT length and axis order, and the block exponents.

The L and K products of small meshes on grids whose lengths run from 16 to 512
against the oracle's AIM product (numpy FFTs of length 2 N).  A grid much finer
than the mesh makes the grid part and the precorrected near part cancel (80
triangles on 63 nodes per axis: by 2e6), so both sides' FP64 rounding counts
relative to the terms that are added: 1e-13 of |near x| + |y|.  The complex128
transforms run in block fixed point, so scaling the input by a power of two must
scale the result exactly up to the order of the projection's atomic additions
(1e-14 of the same terms), and a NaN must reach the result.
"""
import numpy as np
import pytest

from oracle import aim
from oracle.rwg import Mesh
from synth import box, cn_vector, icosphere

pytestmark = pytest.mark.gpu

C0 = 299792458.0


def _mesh(kind, n):
    if kind == "sphere":
        return icosphere(1, 1e-2)
    d = {"x": (n, 1, 1), "y": (1, n, 1), "z": (1, 1, n)}[kind]
    return box([1e-3 * v for v in d], d)


@pytest.mark.parametrize("kind,n", [("sphere", 0), ("sphere", 17), ("sphere", 20), ("sphere", 24), ("sphere", 33),
                                    ("sphere", 40), ("sphere", 48), ("sphere", 64), ("sphere", 65), ("sphere", 81),
                                    ("sphere", 96), ("x", 2), ("x", 5), ("x", 60), ("z", 2), ("z", 5), ("z", 60),
                                    ("x", 3), ("x", 30), ("x", 80), ("y", 45), ("z", 22), ("z", 45), ("z", 80)])
def test_grid_products_match_oracle(lib, ctx, kind, n):
    V, T = _mesh(kind, n)
    m = Mesh(V, T)
    gm = lib.Mesh(ctx, V, T)
    f = 3e9
    op = lib.Operator(gm, f, 2.0, 1.0, 0.0, lib.params(dense_pc_max=0, grid_n=n if kind == "sphere" else 0,
                                                       interior_model=lib.SIE_SIBC))
    g = aim.grid_params(m, M=2, h=op.grid()[1])
    assert np.array_equal(op.grid()[2], g.N)
    ref = aim.AIM(m, 2 * np.pi * f / C0, g)
    X = cn_vector(m.ne, 17, nrhs=3)
    for which, mul in ((0, ref.L), (1, ref.K)):
        want = np.stack([mul(x) for x in X])
        rp, col, val = op.near_csr(which)
        rows = np.repeat(np.arange(m.ne), np.diff(rp))
        near = np.zeros((3, m.ne), complex)
        for r in range(3):
            np.add.at(near[r], rows, val * X[r][col])
        terms = np.linalg.norm(near, axis=1) + np.linalg.norm(want, axis=1)
        y1 = op.matvec(which, np.ascontiguousarray(X[0]))
        assert np.linalg.norm(y1 - want[0]) <= 1e-13 * terms[0]
        Y = op.matvec(which, X, nrhs=3)
        assert (np.linalg.norm(Y - want, axis=1) <= 1e-13 * terms).all()
        for e in (-700, 300):
            ys = op.matvec(which, X[0] * 2.0 ** e)
            assert np.linalg.norm(ys * 2.0 ** -e - y1) <= 1e-14 * terms[0]
        x = X[0].copy()
        x[5] = np.nan
        assert not np.isfinite(op.matvec(which, x)).any()
    op.close()
    gm.close()
