"""Lockstep solutions of conductors, number by number.

A lockstep solve stops at tol_outer and its preconditioner rounds to complex64, so any
other rounding in the entries, the block product or the preconditioner gives another
(equally valid) solution: 1e-16 in b moves x of the bar by 2.5e-3, and its x is 5 to 7%
from the exact solution of the system.  What programs have must stay what it is, so
these are compared with solutions kept from before the transforms were made in integer
arithmetic.  Nothing in the path depends on timing and every run repeats to the bit;
1e-9 is what remains for another compiler's library functions.
"""
import os

import numpy as np
import pytest

from synth import box

pytestmark = pytest.mark.gpu

GOLDEN = os.path.join(os.path.dirname(__file__), "golden", "lockstep_solutions.txt")
CASES = {  # box sizes and cells, frequency, interior model (0 GIBC, 1 SIBC), right-hand sides, grid_n
    "bar": ((40e-6, 4e-6, 4e-6), (20, 2, 2), 100e9, 0, 8, 0),
    "sibc": ((5e-3, 1e-3, 1e-3), (10, 2, 2), 5e9, 1, 3, 0),
}


def solve(lib, ctx, name):
    size, div, f, model, nrhs, grid_n = CASES[name]
    mesh = lib.Mesh(ctx, *box(size, div))
    op = lib.Operator(mesh, f, 1.0, 1.0, 5.8e7, lib.params(interior_model=model, grid_n=grid_n))
    th, ph = 0.3 + 0.35 * np.arange(nrhs), 0.2 + 0.9 * np.arange(nrhs)
    k = np.stack([np.sin(th) * np.cos(ph), np.sin(th) * np.sin(ph), np.cos(th)], axis=1)
    e = np.stack([np.cos(th) * np.cos(ph), np.cos(th) * np.sin(ph), -np.sin(th)], axis=1)
    x, it, rr = op.solve(op.rhs_planewave(k, e), nrhs=nrhs)
    op.close()
    mesh.close()
    assert (rr < 1e-4).all()
    return x[:, ::13]


def kept(name):
    rows = [line.split() for line in open(GOLDEN) if line.startswith(name + " ")]
    n = max(int(r[1]) for r in rows) + 1
    v = np.array([float.fromhex(r[2]) + 1j * float.fromhex(r[3]) for r in rows])
    return v.reshape(n, -1)


@pytest.mark.parametrize("name", sorted(CASES))
def test_solutions_are_what_they_were(lib, ctx, name):
    want, got = kept(name), solve(lib, ctx, name)
    assert got.shape == want.shape
    for q in range(len(want)):
        assert np.linalg.norm(got[q] - want[q]) <= 1e-9 * np.linalg.norm(want[q])


def test_bar_to_a_tight_tolerance(lib, ctx):
    """At tol_outer 1e-8 the method's own noise no longer decides: eight right-hand sides in
    lockstep and one after another (another arithmetic, another preconditioner path) agree
    to the two residuals times the condition of the row-weighted system, 2e4."""
    size, div, f, model, nrhs, grid_n = CASES["bar"]
    mesh = lib.Mesh(ctx, *box(size, div))
    op = lib.Operator(mesh, f, 1.0, 1.0, 5.8e7, lib.params(interior_model=model, grid_n=grid_n, tol_outer=1e-8,
                                                         tol_inner=1e-11, restart=400))
    th, ph = 0.3 + 0.35 * np.arange(nrhs), 0.2 + 0.9 * np.arange(nrhs)
    k = np.stack([np.sin(th) * np.cos(ph), np.sin(th) * np.sin(ph), np.cos(th)], axis=1)
    e = np.stack([np.cos(th) * np.cos(ph), np.cos(th) * np.sin(ph), -np.sin(th)], axis=1)
    b = op.rhs_planewave(k, e)
    x, _, rr = op.solve(b, nrhs=nrhs)
    xs, _, rs = op.solve(b, nrhs=nrhs, sequential=True)
    assert (rr < 1e-8).all() and (rs < 1e-8).all()
    for q in range(nrhs):
        assert np.linalg.norm(x[q] - xs[q]) <= 4e-4 * np.linalg.norm(xs[q])
    op.close()
    mesh.close()
