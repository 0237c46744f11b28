"""The tensor-core backward's tile list: batches at the edges of its 128-row tiles and 64-row K
chunks, output widths that end inside a tile or a 64-column box, grids on both sides of its tile
width rule (64 columns up to three cells, 128 beyond) and one with more cells than SMs; and a first
step on memory that holds NaN."""

import numpy as np
import pytest

from test_gpu_parity import L, _grid, _one_iteration_check, _pool  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,cols,batch,x", [
    (1, 1, 1, 784), (1, 1, 64, 64), (1, 2, 65, 80), (1, 3, 128, 784), (2, 2, 127, 144),
    (1, 4, 129, 208), (2, 2, 192, 192), (1, 5, 256, 784)])
def test_one_iteration_against_the_oracle(L, rows, cols, batch, x):  # noqa: F811
    """Gradients, Adam and weights by the rules of the one-iteration checks (bf16: 2e-2)."""
    pool = _pool(7, 3000, x)
    g = _grid(L, rows, cols, 17, pool, precision="bf16", batch=batch, x_dim=x, keep_grads=1)
    _one_iteration_check(L, g, pool, 2e-2, label="backward tiles %dx%d B=%d x=%d"
                         % (rows, cols, batch, x))


@pytest.mark.parametrize("rows,cols,batch,x", [
    (1, 1, 100, 784), (1, 3, 65, 80), (1, 4, 200, 208), (13, 13, 33, 144)])
def test_fused_adam_equals_stored_gradients_and_repeats(L, rows, cols, batch, x):  # noqa: F811
    """The Adam step in the epilogue equals the stored-gradient path bit for bit, and a second run
    (other CTAs claim other tiles) equals the first."""
    pool = _pool(8, 2000, x)
    kw = dict(precision="bf16", batch=batch, x_dim=x)
    a, b, c = (_grid(L, rows, cols, 5, pool, **kw, **k) for k in ({}, {}, dict(keep_grads=1)))
    for it in range(3):
        for g in (a, b, c):
            g.iterate(1)
        sa = np.frombuffer(a.export_state(), np.uint8)
        assert np.array_equal(sa, np.frombuffer(b.export_state(), np.uint8)), it
        assert np.array_equal(sa, np.frombuffer(c.export_state(), np.uint8)), it


@pytest.mark.parametrize("rows,cols,batch", [(1, 1, 1), (1, 1, 31), (1, 1, 100), (3, 3, 100),
                                             (5, 5, 65), (12, 12, 100)])
def test_first_step_reads_nothing_unwritten(L, rows, cols, batch):  # noqa: F811
    """The first step of a grid whose buffers come from memory full of NaN equals that of a grid on
    memory full of zeros: no tile reads a row that its own dependencies have not written, not even
    against the zeros past a batch that is no multiple of the 64-row K chunk."""
    import torch
    pool = _pool(9, 500, 784)
    states = []
    for byte in (0xFF, 0x00):
        junk = [torch.full((1 << 28,), byte, dtype=torch.uint8, device="cuda") for _ in range(16)]
        torch.cuda.synchronize()
        del junk
        torch.cuda.empty_cache()
        g = _grid(L, rows, cols, 3, pool, precision="bf16", batch=batch)
        g.iterate(1)
        states.append(np.frombuffer(g.export_state(), np.uint8))
        g.close()
    assert np.all(np.isfinite(states[0][64:].view(np.float32)))
    assert np.array_equal(states[0], states[1])
