"""The minibatch draw: rows that are copied in 16, 8, 4 and 2-byte vectors and in parts of a lane's
eight, last groups of fewer than four rows, and noise whose count is no multiple of four or of a
block, against the oracle's draw; and the fitness of a batch around its groups of 128 logits."""

import numpy as np
import pytest

from oracle import lipz_oracle as O
from test_gpu_parity import L, _grid, _pool  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,batch,x,z", [
    ("bf16", 1, 8, 1), ("bf16", 3, 97, 7), ("bf16", 33, 98, 5), ("bf16", 37, 500, 50),
    ("bf16", 100, 784, 64), ("bf16", 130, 1032, 33), ("fp32", 2, 1, 3), ("fp32", 29, 130, 9),
    ("fp32", 128, 131, 16), ("fp32", 129, 784, 64)])
def test_drawn_batch_and_fitness(L, precision, batch, x, z):  # noqa: F811
    pool = _pool(3, 300, x)
    g = _grid(L, 2, 3, 19, pool, precision=precision, batch=batch, z_dim=z, hidden=40, x_dim=x)
    ev = g.eval()
    gx, gz = g.batch()
    lg = g.logits().reshape(6, 5, 6, batch).astype(np.float64)
    arch = O.Arch(z_dim=z, hidden=40, x_dim=x, batch=batch)
    # one rounding of the stored value, and four units in the last place of the fp32 normal
    tol = (2.0 ** -8 if precision == "bf16" else 0.0) + 2.0 ** -20
    for c in range(6):
        ox, oz = O.draw_batch(19, 0, c, pool, arch)
        err = np.abs(gx[c] - ox)
        assert np.all(err <= (2.0 ** -8 if precision == "bf16" else 0.0) * np.abs(ox)), c
        assert np.all(np.abs(gz[c] - oz) <= tol * np.maximum(1.0, np.abs(oz))), c
        sp = np.logaddexp(0.0, lg[c])
        sn = np.logaddexp(0.0, -lg[c])
        fg = sn[:, 1:].mean(2).mean(0)                       # over discriminators and rows
        fd = sn[:, 0].mean(1) + sp[:, 1:].mean(2).mean(1)
        assert np.allclose(ev["fG"][c], fg, rtol=2e-6), c
        assert np.allclose(ev["fD"][c], fd, rtol=2e-6), c
    g.close()
