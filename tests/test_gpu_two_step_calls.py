"""What a step call of large FP32 domains may do besides stepping: the two-step passes'
buffers must not end another stream's capture, block the host or leave an error behind."""
import time

import numpy as np
import pytest

from paper_2606_00641_gb300 import fields

pytestmark = pytest.mark.gpu

SHAPES = [(128, 128, 128), (2048, 2048)]


@pytest.fixture(scope="module")
def V():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2606_00641_gb300 import vlbm
    vlbm.load()
    return vlbm


def context(V, shape, hooks=None, **kw):
    Q = fields.uniform_ideal_state(shape, rho=1.1, u=(0.01, 0.02, 0.0), p=0.02, B=(0.01, 0.0, 0.02), gamma=1.5)
    ctx = V.Context(V.make_params(shape=shape, storage="f32", gamma=1.5, tau=0.6, hooks=hooks, **kw), hooks=hooks)
    assert ctx.init_fields(Q) == V.VLBM_OK
    return ctx


@pytest.mark.parametrize("shape", SHAPES)
def test_first_step_leaves_another_streams_capture_alone(V, shape):
    import torch
    with context(V, shape) as warm:  # kernels loaded before anything is captured
        assert warm.step(4) == V.VLBM_OK and warm.sync() == V.VLBM_OK
    x = torch.zeros(1000, device="cuda")
    with context(V, shape) as ctx:
        before = ctx.launches
        graph, side = torch.cuda.CUDAGraph(), torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.graph(graph, stream=side, capture_error_mode="global"):
            x.add_(1)
            assert ctx.step(4) == V.VLBM_OK
            x.add_(1)
        assert ctx.launches - before == 2  # the passes, with their second buffer
        assert ctx.sync() == V.VLBM_OK
        graph.replay()
        torch.cuda.synchronize()
        assert x.unique().tolist() == [2.0]
