"""The tensor-core Gram kernel's tiles: batches at the edges of its 32-row groups, 128-row tiles,
256-column blocks and of its range (32 to 1360), against the oracle, and at the largest batch
against the CUDA-core path."""

import numpy as np
import pytest

from test_gpu_mixture import L, _check_mixture, _pool  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,cols,batch", [(1, 1, 32), (1, 2, 33), (1, 1, 64), (1, 2, 128),
                                             (2, 2, 250), (1, 1, 251), (1, 2, 256)])
def test_block_means_against_the_oracle(L, rows, cols, batch):  # noqa: F811
    pool = _pool(3, 2000, 784)
    g = L.Grid(rows, cols, seed=9, precision="bf16", batch=batch, mixture=1, mix_sigma=0.05)
    g.set_data(pool)
    _check_mixture(g, pool)


@pytest.mark.parametrize("batch", [1360, 1361])
def test_largest_batches_against_the_cuda_core_path(L, batch):  # noqa: F811
    """1361 is the first batch that the Gram kernel leaves to the CUDA-core path. The two paths'
    fakes differ by bf16 rounding (their sums' order), so the block means get the bf16 tolerance
    of the oracle checks (2e-2); they agree to 1e-4 and better."""
    pool = _pool(4, 3000, 64)
    means = []
    for simt in (0, 1):
        g = L.Grid(1, 1, seed=2, precision="bf16", batch=batch, x_dim=64, mixture=1, force_simt=simt)
        g.set_data(pool)
        g.eval()
        means.append(g.mixture(blocks=True)[1])
    assert np.max(np.abs(means[0] - means[1])) < 2e-2 * np.max(np.abs(means[1]))
