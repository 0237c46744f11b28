"""The CUDA-core grouped GEMM and the gathered training inputs: sizes at the edges of the output
tiles (32, 64, 128) and of the 16-wide k-slices, rows that allow and forbid four-element loads, in
both precisions (bf16 with force_simt, which keeps it off the tensor cores), and grids on both sides of
the tile-shape rule; one iteration against the oracle.
"""

import pytest

from test_gpu_parity import L, _grid, _one_iteration_check, _pool  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,rows,cols,batch,z,hidden,x", [
    ("fp32", 1, 1, 1, 1, 1, 1), ("fp32", 1, 2, 5, 3, 9, 33), ("fp32", 2, 2, 32, 16, 64, 128),
    ("fp32", 2, 3, 33, 50, 66, 130), ("fp32", 1, 3, 127, 4, 132, 60),
    ("fp32", 4, 5, 21, 20, 128, 64), ("bf16", 1, 2, 37, 50, 200, 500), ("bf16", 1, 1, 16, 6, 31, 17),
    ("bf16", 2, 2, 65, 24, 136, 72)])
def test_one_iteration_against_the_oracle(L, precision, rows, cols, batch, z, hidden, x):  # noqa: F811
    """Evaluation, gradients, Adam and weights by the rules of the one-iteration checks."""
    pool = _pool(5, 500, x)
    g = _grid(L, rows, cols, 23, pool, precision=precision, batch=batch, z_dim=z, hidden=hidden,
              x_dim=x, keep_grads=1, force_simt=int(precision == "bf16"))
    _one_iteration_check(L, g, pool, 1e-4 if precision == "fp32" else 2e-2,
                         label="CUDA-core %s h=%d" % (precision, hidden))
