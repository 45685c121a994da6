"""Grid products of vectors near the bottom of the FP64 range: intermediate results below
the normal range round to a multiple of 2^-1074, as FP64 arithmetic does, instead of to
zero.  Scaling by a power of two then costs at most the rounding of those multiples: a
product whose result is around 1e-304 keeps 1e-12 of its norm (a few hundred thousand
roundings of 5e-324 in grids that are at most 1e6 below or above the result).
"""
import numpy as np
import pytest

from synth import cn_vector, icosphere

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("which", [0, 1])
def test_scaled_down_products(lib, ctx, which):
    mesh = lib.Mesh(ctx, *icosphere(1, 1e-2))
    op = lib.Operator(mesh, 3e9, 4.0, 1.0, 0.0, lib.params(dense_pc_max=0))
    x = cn_vector(mesh.ne, 8)
    y = op.matvec(which, x)
    # x itself stays normal: the products' scale decides how far down it may go
    k = -int(np.floor(np.log2(1e-304 / np.linalg.norm(y))))
    small = op.matvec(which, np.ldexp(x.real, -k) + 1j * np.ldexp(x.imag, -k))
    back = np.ldexp(small.real, k) + 1j * np.ldexp(small.imag, k)
    assert np.linalg.norm(back - y) <= 1e-12 * np.linalg.norm(y)
    op.close()
    mesh.close()
