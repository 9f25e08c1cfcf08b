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


@pytest.mark.parametrize("shape", SHAPES)
def test_first_step_does_not_wait_for_the_stream(V, shape):
    import torch
    with context(V, shape) as warm:
        assert warm.step(4) == V.VLBM_OK and warm.sync() == V.VLBM_OK
    side = torch.cuda.Stream()
    with context(V, shape, stream=side.cuda_stream) as ctx:
        done = torch.cuda.Event()
        with torch.cuda.stream(side):
            torch.cuda._sleep(2_000_000_000)  # about a second
        before = ctx.launches
        t = time.perf_counter()
        assert ctx.step(4) == V.VLBM_OK
        took = time.perf_counter() - t
        done.record(side)
        assert not done.query() and took < 0.3
        assert ctx.sync() == V.VLBM_OK and ctx.launches - before == 2


def test_refused_strip_table_takes_single_steps_and_leaves_no_error(V):
    import torch
    shape = (2048, 2048)
    base = V.TorchHooks()
    asked = []

    def alloc(nbytes, stream, user):
        asked.append(nbytes)
        return base.alloc(nbytes, stream, user) if len(asked) != 3 else None  # populations, status block, table

    class Hooks:
        dealloc = base.dealloc

    Hooks.alloc = V.ALLOC_FN(alloc)
    Q = fields.uniform_ideal_state(shape, rho=1.1, u=(0.01, 0.02, 0.0), p=0.02, B=(0.01, 0.0, 0.02), gamma=1.5)
    Qd = torch.as_tensor(Q, device="cuda")
    with V.Context(V.make_params(shape=shape, storage="f32", gamma=1.5, tau=0.6, hooks=Hooks)) as ctx:
        assert V.vlbm_init_fields_device(ctx.ptr, 0, Qd.data_ptr()) == V.VLBM_OK
        before = ctx.launches
        assert ctx.step(8) == V.VLBM_OK and ctx.sync() == V.VLBM_OK
        assert ctx.launches - before == 8 and len(asked) >= 3
        assert V.last_error(ctx.ptr) == ""


@pytest.mark.parametrize("hooked", [False, True])
@pytest.mark.parametrize("shape", SHAPES)
def test_two_step_off_gives_the_memory_back(V, shape, hooked):
    import torch
    cells = np.random.default_rng(1).integers(0, int(np.prod(shape)), 100000)
    f0 = fields.ideal_fields(shape, 23, mach=0.5, beta=1.0, cfl=0.1, device=torch.device("cuda"))
    base, held = V.TorchHooks(), {}

    def alloc(nbytes, stream, user):
        p = base.alloc(nbytes, stream, user)
        held[p] = nbytes
        return p

    def dealloc(ptr, nbytes, stream, user):
        assert held.pop(ptr) == nbytes
        base.dealloc(ptr, nbytes, stream, user)

    class Hooks:
        pass

    Hooks.alloc, Hooks.dealloc = V.ALLOC_FN(alloc), V.FREE_FN(dealloc)
    got = []
    for switched in (False, True):
        p = V.make_params(shape=shape, storage="f32", gamma=f0.gamma, tau=0.6, hooks=Hooks if hooked else None)
        with V.Context(p) as ctx:
            pops = V.vlbm_population_bytes(ctx.ptr)
            assert V.vlbm_init_fields_device(ctx.ptr, 0, f0.Q.data_ptr()) == V.VLBM_OK
            marks = [ctx.launches]
            for n, on in ((40, True), (40, False), (7, False), (8, True)):
                if switched:
                    ctx.set_two_step(on)
                assert ctx.step(n) == V.VLBM_OK and ctx.sync() == V.VLBM_OK
                marks.append(ctx.launches)
                if switched:
                    free = torch.cuda.mem_get_info()[0]
                    ctx.set_two_step(False)
                    if hooked:
                        assert list(held.values()).count(pops) == 1
                    elif on:
                        assert torch.cuda.mem_get_info()[0] - free >= pops
            passes = np.diff(marks).tolist()
            # from step 87 (odd): a single step, a pass of four, three single steps
            assert passes == ([20, 40, 7, 6] if switched else [20, 20, 5, 6])
            got.append(ctx.populations(cells))
    assert np.array_equal(got[0], got[1]) and not held


def test_two_step_off_keeps_what_a_callers_graph_holds(V):
    import torch
    shape = (128, 128, 128)
    cells = np.random.default_rng(1).integers(0, int(np.prod(shape)), 100000)
    f0 = fields.ideal_fields(shape, 23, mach=0.5, beta=1.0, cfl=0.1, device=torch.device("cuda"))
    got = []
    for captured in (False, True):
        side = torch.cuda.Stream()
        p = V.make_params(shape=shape, storage="f32", gamma=f0.gamma, tau=0.6, stream=side.cuda_stream)
        with V.Context(p) as ctx:
            assert V.vlbm_init_fields_device(ctx.ptr, 0, f0.Q.data_ptr()) == V.VLBM_OK
            assert ctx.step(4) == V.VLBM_OK
            if captured:
                graph = torch.cuda.CUDAGraph()
                with torch.cuda.graph(graph, stream=side):
                    assert ctx.step(8) == V.VLBM_OK
                free = torch.cuda.mem_get_info()[0]
                ctx.set_two_step(False)
                assert torch.cuda.mem_get_info()[0] - free < V.vlbm_population_bytes(ctx.ptr)
                other = torch.full((V.vlbm_population_bytes(ctx.ptr),), 7, dtype=torch.uint8, device="cuda")
                with torch.cuda.stream(side):
                    graph.replay()
                torch.cuda.synchronize()
                assert bool((other == 7).all())
            else:
                assert ctx.step(8) == V.VLBM_OK
            assert ctx.sync() == V.VLBM_OK and ctx.step_count == 12
            got.append(ctx.populations(cells))
    assert np.array_equal(got[0], got[1])


def test_two_step_off_is_refused_under_capture(V):
    import torch
    side = torch.cuda.Stream()
    with context(V, (128, 128, 128), stream=side.cuda_stream) as ctx:
        assert ctx.step(4) == V.VLBM_OK and ctx.sync() == V.VLBM_OK
        graph = torch.cuda.CUDAGraph()
        x = torch.zeros(10, device="cuda")
        with torch.cuda.graph(graph, stream=side):
            x.add_(1)
            with pytest.raises(V.VlbmError):
                ctx.set_two_step(False)
        before = ctx.launches
        assert ctx.step(4) == V.VLBM_OK and ctx.sync() == V.VLBM_OK and ctx.launches - before == 2
