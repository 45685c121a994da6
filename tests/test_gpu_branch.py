"""Block products whose near part runs on a branch beside the grid part (from
2 M near entries x right-hand sides) against one vector at a time, on either
side of that line.  Both forms add the same terms in another order: about 500
near entries a row and a tenfold cancellation with the grid part bound the
difference by 500 x 10 x 1.1e-16 = 5.5e-13 of |y|; asked: 1e-12."""
import numpy as np
import pytest

from synth import cn_vector, icosphere

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sphere(lib, ctx):
    V, T = icosphere(3, 0.01)
    gm = lib.Mesh(ctx, V, T)
    op = lib.Operator(gm, 3e9, 4.0, 1.0, 0.0)
    yield op
    op.close()
    gm.close()


@pytest.mark.parametrize("which", [0, 1, 3])
@pytest.mark.parametrize("R", [2, 5, 8])
def test_branch_matches_one_vector(sphere, which, R):
    op = sphere
    assert op.info()[8] * 8 >= 2e6  # eight vectors take the branch
    X = cn_vector(op.mesh.ne, 700 + which, nrhs=R)
    Y = op.matvec(which, X, nrhs=R)
    for r in range(R):
        one = op.matvec(which, np.ascontiguousarray(X[r]))
        assert np.linalg.norm(Y[r] - one) <= 1e-12 * np.linalg.norm(one)
