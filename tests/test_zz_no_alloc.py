"""The allocation-free fitness entry point, for callers that cannot call cudaMalloc (a serving
loop whose device memory another allocator has fully reserved, or a latency-critical path that
cannot take the implicit synchronisation of cudaMalloc / cudaFree).

Its output must match the fitness that lipz_eval_neighborhoods returns for the same logits, on calls of
different sizes in a row, on calls that overlap on several streams, and from a captured graph. This
file is collected last.
"""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1811_12843_gb300 import _build
    _build.build()
    import lipz_synth
    import paper_1811_12843_gb300 as L
    return torch, L, lipz_synth


def _reference(L, lipz_synth, rows, cols, precision, batch, seed):
    g = L.Grid(rows, cols, seed=seed, precision=precision, batch=batch)
    g.set_data(lipz_synth.blob_pool(seed, n=1000, dim=784))
    ev = g.eval()
    logits = g.logits()
    g.close()
    return logits, ev["fG"], ev["fD"]


def test_noalloc_fitness_matches_eval_on_two_calls(env):
    torch, L, lipz_synth = env
    cases = [(3, 4, "bf16", 100, 7), (2, 2, "fp32", 37, 8)]
    refs = [_reference(L, lipz_synth, *c) for c in cases]
    stream = torch.cuda.current_stream()
    for (rows, cols, _, batch, _), (logits, fg_ref, fd_ref) in zip(cases, refs):
        cells = rows * cols
        dl = torch.from_numpy(logits).cuda()
        fg = torch.full((cells, 5), float("nan"), device="cuda")
        fd = torch.full((cells, 5), float("nan"), device="cuda")
        L.lipz_fitness_from_logits_noalloc(dl, cells, batch, fg, fd, stream)
        torch.cuda.synchronize()
        for got, ref in ((fg.cpu().numpy(), fg_ref), (fd.cpu().numpy(), fd_ref)):
            assert np.max(np.abs(got - ref)) <= 1e-4 * np.max(np.abs(ref))


def _random_case(torch, L, seed, cells, batch):
    """Logits on the device and the fitnesses that a call alone on the device gives for them."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    logits = torch.randn((cells, 5, 6 * batch), generator=gen, device="cuda")
    out = [torch.full((cells, 5), float("nan"), device="cuda") for _ in range(2)]
    torch.cuda.synchronize()
    L.lipz_fitness_from_logits_noalloc(logits, cells, batch, *out, torch.cuda.current_stream())
    torch.cuda.synchronize()
    return logits, [o.clone() for o in out]


def test_noalloc_calls_overlap_on_streams(env):
    torch, L, _ = env
    shapes = [(4096, 16), (1, 256), (144, 100), (600, 33)]
    cases = [_random_case(torch, L, 40 + i, *s) for i, s in enumerate(shapes)]
    streams = [torch.cuda.Stream() for _ in shapes]
    outs = [[torch.full_like(r, float("nan")) for r in ref] for _, ref in cases]
    torch.cuda.synchronize()
    for _ in range(20):
        for (cells, batch), (logits, _), out, st in zip(shapes, cases, outs, streams):
            L.lipz_fitness_from_logits_noalloc(logits, cells, batch, *out, st)
    torch.cuda.synchronize()
    for (_, ref), out in zip(cases, outs):
        assert all(torch.equal(o, r) for o, r in zip(out, ref))


def test_noalloc_call_in_a_graph(env):
    torch, L, _ = env
    cells, batch = 37, 100
    logits, ref = _random_case(torch, L, 50, cells, batch)
    other, ref2 = _random_case(torch, L, 51, cells, batch)
    out = [torch.full_like(r, float("nan")) for r in ref]
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        L.lipz_fitness_from_logits_noalloc(logits, cells, batch, *out, torch.cuda.current_stream())
    for data, want in ((None, ref), (other, ref2)):
        if data is not None:
            logits.copy_(data)
        graph.replay()
        torch.cuda.synchronize()
        assert all(torch.equal(o, r) for o, r in zip(out, want))


def test_noalloc_rejects_sizes_beyond_the_limit(env):
    torch, L, _ = env
    dl = torch.zeros(30, device="cuda")
    out = torch.zeros(5, device="cuda")
    with pytest.raises(L.LipzError) as e:
        L.lipz_fitness_from_logits_noalloc(dl, 4097, 1, out, out)
    assert e.value.code == L.LIPZ_ERR_INVALID
    with pytest.raises(L.LipzError) as e:
        L.lipz_fitness_from_logits_noalloc(dl, 0, 1, out, out)
    assert e.value.code == L.LIPZ_ERR_INVALID
