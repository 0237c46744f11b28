"""The tensor-core Gram kernel's tiles: batches at the edges of its 32-row groups, 128-row tiles,
256-column blocks and of its range (32 to 1360), against the oracle, and at the largest batch
against the CUDA-core path; and its sums' own error."""

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


@pytest.mark.parametrize("x,batch", [(784, 256), (1024, 256), (1024, 300)])
def test_products_are_as_exact_as_a_stored_fp32_matrix(L, x, batch):  # noqa: F811
    """The block mean of the real rows with themselves, known exactly, for batches above 250: the mean
    of its error over 24 cells. A result's own rounding is at most 2^-24 and the exponentials' mean error
    (1 / x and the argument rounded) about as much; tensor memory's truncation, if all of a product's
    terms were summed there, would add 1e-7 (784) to 1.7e-7 (1024)."""
    pool = _pool(6, 3000, x)
    errs = []
    for seed in range(6):
        g = L.Grid(2, 2, seed=seed, precision="bf16", batch=batch, x_dim=x, mixture=1)
        g.set_data(pool)
        g.eval()
        X = g.batch()[0].astype(np.float64)
        S = g.mixture(blocks=True)[1]
        for c in range(4):
            n = (X[c] ** 2).sum(1)
            ref = np.exp(-(n[:, None] + n - 2.0 * X[c] @ X[c].T) / x).mean()
            errs.append((S[c][0, 0] - ref) / ref)
        g.close()
    assert abs(np.mean(errs)) < 1.5 * 2.0 ** -24, np.mean(errs)
