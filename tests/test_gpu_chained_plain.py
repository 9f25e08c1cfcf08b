"""Chained step launches against plain ones: the context on the legacy default stream (handle 1)
and the one whose steps go into the caller's own capture launch every step without the
programmatic attribute, the ones on streams of their own with it.  Bit for bit the same
populations and sums after direct launches, captured graphs and calls in between."""
import numpy as np
import pytest

from test_gpu_chained import V, prepared  # noqa: F401  (the fixture and the states of the stream test)

pytestmark = pytest.mark.gpu

CASES = [("ideal", (1, 1)), ("ideal", (64, 64)), ("ideal", (150, 200)), ("ideal", (1, 5, 3)), ("ideal", (40, 41, 39)),
         ("ideal", (64, 128, 128)), ("powell", (12, 20, 33)), ("powell", (64, 128, 128)), ("channel", (8, 32, 32)),
         ("channel", (20, 50, 60)), ("channel", (64, 128, 128))]


@pytest.mark.parametrize("model,shape", CASES)
def test_chained_equals_plain(V, model, shape):  # noqa: F811
    import torch
    side, caller = torch.cuda.Stream(), torch.cuda.Stream()
    plain, captured = prepared(V, model, shape, 1), prepared(V, model, shape, caller.cuda_stream)
    own, given = prepared(V, model, shape, None), prepared(V, model, shape, side.cuda_stream)
    assert V.vlbm_stream(plain.ptr) == 1 and V.vlbm_stream(own.ptr) not in (0, 1, 2)
    out = {c: [] for c in (plain, captured, own, given)}
    for n in (7, 70, 4):
        assert plain.step(n) == V.VLBM_OK
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=caller):
            assert captured.step(n) == V.VLBM_OK
        with torch.cuda.stream(caller):
            graph.replay()
        for c in (own, given):  # together
            assert c.step(n) == V.VLBM_OK
        for c, o in out.items():
            o.append(np.array(c.conservation()))
    cells = np.unique(np.random.default_rng(2).integers(0, int(np.prod(shape)), 200000))
    for c, o in out.items():
        assert c.sync() == V.VLBM_OK
        o.append(c.populations(cells))
    for c in (captured, own, given):
        assert all(np.array_equal(a, b) for a, b in zip(out[plain], out[c]))
    for c in out:
        c.close()
