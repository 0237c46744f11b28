"""Results brought to the host in one copy: every subset of an evaluation's four result arrays, on grids
of one cell and of more values than a block gathers, from the evaluation and from an iteration."""

import numpy as np
import pytest

from test_gpu_parity import L, _grid, _pool  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,cols", [(1, 1), (4, 16)])
def test_every_subset_of_results(L, rows, cols):  # noqa: F811
    C = rows * cols
    pool = _pool(2, 200, 64)
    g = _grid(L, rows, cols, 5, pool, precision="bf16", batch=16, x_dim=64)
    full = g.eval(pairs=True)
    names, shapes = ("fG", "fD", "LG", "LD"), ((C, 5), (C, 5), (C, 5, 5), (C, 5, 5))
    for mask in range(1, 16):
        out = [np.full(s, np.nan, np.float32) if mask >> i & 1 else None
               for i, s in enumerate(shapes)]
        L.lipz_eval_neighborhoods(g.h, *out)
        for n, o in zip(names, out):
            assert o is None or np.array_equal(o, full[n]), (mask, n)
    x = np.ascontiguousarray(g.batch()[0])
    fg, fd = (np.full((C, 5), np.nan, np.float32) for _ in range(2))
    L.lipz_iterate_batch(g.h, x, fg, fd)
    assert np.array_equal(fg, full["fG"]) and np.array_equal(fd, full["fD"])
    g.close()
