"""The tensor-core convolutions' tiles: batches whose output pixels end inside a 128-row tile, a
CTA pair or a 256-row tile, one and several cells per launch, and widths with 128- and 256-column
weight tiles. One iteration through the TMA kernels (CTA pairs, 256-row tiles, the shared first
layer) must end in the state of the one-CTA kernels that gather their A rows, and in that of a device
where no pair can be resident and no output map applies, bit for bit, and the evaluation must meet the
oracle. And a grid for whose cells' shared launches the memory is not there."""

import numpy as np
import pytest

from oracle import lipz_oracle as O

from helpers import max_rel
from test_gpu_dcgan import L, _field_pool, _grid, _state  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,cols,batch,ngf,ndf", [
    (1, 1, 1, 64, 64), (1, 2, 3, 64, 64), (1, 1, 7, 64, 64), (2, 2, 20, 64, 64), (1, 2, 35, 64, 64),
    (1, 1, 8, 128, 64)])
def test_tma_pairs_equal_gathered_tiles(L, monkeypatch, rows, cols, batch, ngf, ndf):  # noqa: F811
    pool = _field_pool(6, 64)
    out = []
    for gather, single in (("0", "0"), ("1", "0"), ("0", "1")):
        monkeypatch.setenv("LIPZ_CONV_GATHER", gather)
        monkeypatch.setenv("LIPZ_CONV_SINGLE", single)
        g = _grid(L, rows, cols, 3, pool, precision="bf16", batch=batch, ngf=ngf, ndf=ndf)
        g.iterate(2)
        out.append(np.frombuffer(g.export_state(), np.uint8))
    assert np.array_equal(out[0], out[1])
    assert np.array_equal(out[0], out[2])


@pytest.mark.parametrize("batch", [1, 9])
def test_evaluation_against_the_oracle(L, batch):  # noqa: F811
    pool = _field_pool(5, 30)
    g = _grid(L, 1, 1, 9, pool, precision="bf16", batch=batch, ngf=64, ndf=64)
    s = _state(g)
    ref = O.eval_neighborhoods(s, O.batches(s, pool))
    g.eval()
    assert max_rel(g.logits(), ref["logits"]) < 2e-2


def test_little_memory_means_fewer_cells_per_launch(L):  # noqa: F811
    """Where only one cell's evaluation buffers fit beside what a grid cannot do without, the grid is
    created and computes the same."""
    import torch
    cells, batch = 4, 64
    kw = dict(precision="bf16", batch=batch, ngf=64, ndf=64)
    pool = _field_pool(4, 40)

    def run():
        g = _grid(L, 1, cells, 13, pool, **kw)
        g.iterate(1)
        state = np.frombuffer(g.export_state(), np.uint8)
        g.close()
        return state

    def free():
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        return torch.cuda.mem_get_info()[0]

    run()
    before = free()
    g = _grid(L, 1, cells, 13, pool, **kw)
    used = before - free()
    g.close()
    ref = run()
    cell = 30 * batch * (64 * 32 * 32 + 128 * 16 * 16) * 2
    assert used > cells * cell
    # all but one cell's buffers less than the grid took, and some allocations' rounding more
    room = used - (cells - 1) * cell + (256 << 20)
    hold = torch.empty(free() - room, dtype=torch.uint8, device="cuda")
    try:
        assert np.array_equal(run(), ref)
    finally:
        del hold
        torch.cuda.empty_cache()
