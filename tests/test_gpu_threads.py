"""Contexts in threads of their own, with operators of different sizes, as the serving
slots run them: the resident kernels of all sizes share their functions' limits, and no
launch may fail or fall back because another thread asked for less.
"""
import threading

import numpy as np
import pytest

from synth import box, cn_vector

pytestmark = pytest.mark.gpu


def test_two_sizes_at_once(lib):
    sizes = {2: [], 10: []}
    errors = []
    start = threading.Barrier(len(sizes))

    def work(n):
        try:
            ctx = lib.Context(0)
            mesh = lib.Mesh(ctx, *box((1e-3, 1e-3, 1e-3), (n, n, n)))
            op = lib.Operator(mesh, 10e9, 1.0, 1.0, 1e5, lib.params(interior_model=1, dense_pc_max=0, grid_n=24))
            H = cn_vector(mesh.ne, n)
            start.wait()
            for _ in range(400):
                sizes[n].append(op.matvec(lib.SIE_OP_ZI, H))
            op.close()
            mesh.close()
            ctx.close()
        except Exception as e:  # noqa: BLE001 - reported by the main thread
            errors.append((n, repr(e)))

    th = [threading.Thread(target=work, args=(n,)) for n in sizes]
    for t in th:
        t.start()
    for t in th:
        t.join()
    assert not errors
    for n, ys in sizes.items():  # the same kernel every time: the same bits
        assert all(np.array_equal(y, ys[0]) for y in ys)
