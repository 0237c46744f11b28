"""The forward by CTA pairs: grids whose generator pairs divide their output blocks among idle
clusters (one to four blocks, last blocks of 16 to 256 columns, parts of different lengths) and grids just
too large for it, and first layers whose last K chunk holds one to four steps; against the oracle."""

import pytest

from test_gpu_parity import L, _grid, _one_iteration_check, _pool  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,cols,batch,x", [
    (1, 1, 100, 80), (1, 1, 33, 256), (1, 2, 100, 272), (1, 1, 256, 1024), (2, 3, 150, 528),
    (3, 3, 100, 784), (4, 5, 100, 784), (3, 4, 64, 112), (5, 8, 60, 96)])
def test_one_iteration_against_the_oracle(L, rows, cols, batch, x):  # noqa: F811
    """Evaluation, gradients, Adam and weights by the rules of the one-iteration checks."""
    pool = _pool(11, 300, x)
    g = _grid(L, rows, cols, 31, pool, precision="bf16", batch=batch, x_dim=x, keep_grads=1)
    _one_iteration_check(L, g, pool, 2e-2, label="pairs x=%d" % x)
