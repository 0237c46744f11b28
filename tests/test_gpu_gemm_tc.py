"""The tensor-core grouped GEMM (bf16 networks that the chained kernels do not take): widths and
batches at the edges of its 128 x 64 and 128 x 128 tiles, of the 64-wide chunks and of the last MMA
step of 16, rows whose starts allow copies of 16, 8, 4 and 2 bytes, both operand orders (the
backward's transposed products), later minibatch steps, and the stored Gram matrix of a batch that is
too long for the Gram kernel; against the oracle, or the CUDA-core kernels."""

import numpy as np
import pytest

from test_gpu_parity import L, _grid, _one_iteration_check, _pool  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,cols,batch,z,hidden,x", [
    (1, 1, 1, 1, 1, 1), (1, 2, 3, 5, 17, 33), (1, 2, 21, 16, 64, 63), (2, 2, 22, 50, 66, 130),
    (1, 3, 64, 15, 128, 65), (1, 2, 43, 100, 129, 127), (2, 3, 37, 48, 200, 500),
    (3, 3, 130, 66, 300, 1000), (4, 5, 24, 36, 257, 196), (1, 2, 65, 20, 512, 64)])
def test_one_iteration_against_the_oracle(L, rows, cols, batch, z, hidden, x):  # noqa: F811
    """Evaluation, gradients, Adam and weights by the rules of the one-iteration checks. (Nine cells
    at the largest size: the rules bound the median cell, and one cell with an activation that rounds
    the other way than the oracle's is off by 0.8 to 1.2 times 1e-2 on either route.)"""
    pool = _pool(7, 400, x)
    g = _grid(L, rows, cols, 29, pool, precision="bf16", batch=batch, z_dim=z, hidden=hidden,
              x_dim=x, keep_grads=1)
    _one_iteration_check(L, g, pool, 2e-2, label="bf16 h=%d" % hidden)


@pytest.mark.parametrize("batch,hidden,x,steps", [(30, 40, 50, 3), (1400, 24, 72, 1)])
def test_equals_the_cuda_core_kernels(L, batch, hidden, x, steps):  # noqa: F811
    """An iteration (several minibatch steps; a mixture on a stored Gram matrix) and the next
    evaluation on both routes. The fp32 sums differ in their order only, which moves a bf16 activation
    by at most one unit in the last place (2^-8); fitnesses and block means are means over many."""
    out = []
    for simt in (0, 1):
        g = L.Grid(1, 2, seed=3, precision="bf16", batch=batch, z_dim=10, hidden=hidden, x_dim=x,
                   train_steps=steps, mixture=1, force_simt=simt)
        g.set_data(_pool(4, 500, x))
        g.iterate(1)
        ev = g.eval()
        out.append((ev["fG"], ev["fD"], g.mixture(blocks=True)[1]))
        g.close()
    for a, b in zip(*out):
        assert np.max(np.abs(a - b)) <= 2.0 ** -7 * np.max(np.abs(b))
