"""Near-region matrices in every branch of the close-pair integration kernel.

Small icosphere (80 triangles: self, edge, vertex and plain close pairs, far
pairs), exterior and interior wavenumbers that take each radial rule: real and
complex Taylor orders (|k| R <= 1), graded radial Gauss and the coplanar closed
forms with real and complex k beyond it.  Both sides evaluate the same FP64
quadrature rule, so they agree to the rounding of its sums amplified by the
precorrection (exact minus grid): 1e-10 of the largest entry, as in
test_gpu_aim.py.
"""
import numpy as np
import pytest

from oracle import aim
from oracle.rwg import Mesh
from synth import icosphere

from test_gpu_aim import C0, _csr_dense, k_medium

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("freq,eps_r,sigma", [(3e9, 4.0, 0.0), (3e9, 4.0, 0.1), (20e9, 4.0, 0.0), (20e9, 4.0, 5.0),
                                              (0.3e9, 2.0, 0.01)])
def test_near_rules_match_oracle(lib, ctx, freq, eps_r, sigma):
    V, T = icosphere(1, 0.01)
    m = Mesh(V, T)
    gm = lib.Mesh(ctx, V, T)
    op = lib.Operator(gm, freq, eps_r, 1.0, sigma, lib.params(dense_pc_max=0))
    assert op.info()[9] == 0.0
    g = aim.grid_params(m, M=2)
    for k, which in ((2 * np.pi * freq / C0, 0), (k_medium(freq, eps_r, sigma), 2)):
        ref = aim.AIM(m, k, g)
        for w, a in ((which, "NL"), (which + 1, "NK")):
            got = _csr_dense(*op.near_csr(w), m.ne)
            want = getattr(ref, a).toarray()
            assert np.abs(got - want).max() <= 1e-10 * np.abs(want).max()
    op.close()
    gm.close()
