"""The two-step pass of large plain 3-D FP32 boxes: bit for bit the single steps.

A run advanced in one call (pairs of steps in one pass) equals the same run advanced
one step per call (a launch per step) in every population, at even and odd step
counts, from an odd step count, with sources, on boxes whose sides divide neither the
pass's columns (30 x 6) nor its height (16), and through captured graphs; and the
oracle's result on light-cone boxes at the repository's FP32 tolerance."""
import numpy as np
import pytest

from paper_2606_00641_gb300 import fields

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def V():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2606_00641_gb300 import vlbm
    vlbm.load()
    return vlbm


def populations(V, ctx, shape, seed):
    n = int(np.prod(shape))
    cells = np.unique(np.concatenate([np.random.default_rng(seed).integers(0, n, 200000), np.arange(3000),
                                      np.arange(n - 3000, n)]))
    return ctx.populations(cells)


@pytest.mark.parametrize("shape,calls", [((128, 128, 128), (4,)), ((128, 128, 128), (1, 7, 8, 6)),
                                         ((161, 127, 178), (9, 6)), ((200, 149, 149), (40, 3)),
                                         ((111, 203, 239), (70,))])
def test_equals_single_steps(V, shape, calls):
    import torch
    f0 = fields.ideal_fields(shape, 21, mach=0.5, beta=1.0, cfl=0.2, device=torch.device("cuda"))
    tau = np.array([0.51, 0.6, 0.55, 0.7, 0.52, 0.8, 0.65, 0.9])
    src = np.array([1e-7, -2e-7, 3e-7, 0.0, 1e-8, 2e-8, -1e-8, 0.0])
    p = V.make_params(shape=shape, storage="f32", gamma=f0.gamma, tau=tau, source=src)
    got = []
    for one in (False, True):
        with V.Context(p) as ctx:
            assert V.vlbm_init_fields_device(ctx.ptr, 0, f0.Q.data_ptr()) == V.VLBM_OK
            before = ctx.launches
            for n in calls:
                for _ in range(n if one else 1):
                    assert ctx.step(1 if one else n) == V.VLBM_OK
            assert ctx.step_count == sum(calls)
            passes = ctx.launches - before
            assert ctx.sync() == V.VLBM_OK
            got.append(populations(V, ctx, shape, 22))
            # a launch per step, or two per four steps after a single one from an odd step count
            want, at = 0, 0
            for n in calls:
                want += at % 2 + (n - at % 2) // 4 * 2 + (n - at % 2) % 4
                at += n
            assert passes == (sum(calls) if one else want)
    assert np.array_equal(got[0], got[1])


@pytest.mark.parametrize("shape,calls", [((90, 130, 150), (40, 5)), ((121, 141, 178), (6, 8))])
def test_powell_equals_single_steps(V, shape, calls):
    import torch
    f0 = fields.ideal_fields(shape, 28, mach=0.5, beta=1.0, cfl=0.2, device=torch.device("cuda"))
    Q = torch.cat([f0.Q, 1e-3 * (f0.Q[:1] - 1.0)])
    p = V.make_params(model=V.VLBM_IDEAL_POWELL, shape=shape, storage="f32", gamma=f0.gamma, tau=0.55, tau_d=0.6,
                      tau_m=1.5)
    got, passes = [], []
    for one in (False, True):
        with V.Context(p) as ctx:
            assert V.vlbm_init_fields_device(ctx.ptr, 0, Q.data_ptr()) == V.VLBM_OK
            before = ctx.launches
            for n in calls:
                for _ in range(n if one else 1):
                    assert ctx.step(1 if one else n) == V.VLBM_OK
            passes.append(ctx.launches - before)
            assert ctx.sync() == V.VLBM_OK
            got.append(populations(V, ctx, shape, 29))
    assert np.array_equal(got[0], got[1])
    assert passes[0] < passes[1] == sum(calls)


@pytest.mark.parametrize("shape,calls", [((2048, 2048), (4, 10)), ((1999, 2311), (41, 8)), ((4099, 1030), (6,))])
def test_2d_equals_single_steps(V, shape, calls):
    import torch
    f0 = fields.ideal_fields(shape, 25, mach=0.5, beta=1.0, cfl=0.1, device=torch.device("cuda"))
    tau = np.array([0.51, 0.6, 0.55, 0.7, 0.52, 0.8, 0.65, 0.9])
    src = np.array([1e-7, -2e-7, 3e-7, 0.0, 1e-8, 2e-8, -1e-8, 0.0])
    p = V.make_params(shape=shape, storage="f32", gamma=f0.gamma, tau=tau, source=src)
    got, passes = [], []
    for one in (False, True):
        with V.Context(p) as ctx:
            assert V.vlbm_init_fields_device(ctx.ptr, 0, f0.Q.data_ptr()) == V.VLBM_OK
            before = ctx.launches
            for n in calls:
                for _ in range(n if one else 1):
                    assert ctx.step(1 if one else n) == V.VLBM_OK
            passes.append(ctx.launches - before)
            assert ctx.sync() == V.VLBM_OK
            got.append(populations(V, ctx, shape, 26))
    assert np.array_equal(got[0], got[1])
    assert passes[0] < passes[1] == sum(calls)


def test_batch_equals_single_steps(V):
    import torch
    sides = [(1024, 1024), (64, 64), (31, 33), (512, 700), (128, 130), (1, 90), (90, 1), (800, 1000)]
    params, Q = [], []
    for i, shape in enumerate(sides):
        f0 = fields.ideal_fields(shape, 30 + i, gamma=1.4 + 0.03 * i, mach=0.2, cfl=0.1, k_rho=1, k_u=1, k_b=1,
                                 device=torch.device("cuda")) if min(shape) > 2 else None
        if f0 is None:
            u = fields.uniform_ideal_state(shape, rho=1.1, u=(0.01, 0.02, 0.0), p=0.02, B=(0.01, 0.0, 0.02), gamma=1.5)
            Q.append(torch.as_tensor(u, device="cuda"))
        else:
            Q.append(f0.Q)
        params.append(V.make_params(shape=shape, storage="f32", gamma=1.4 + 0.03 * i, tau=0.55 + 0.01 * i))
    got, passes = [], []
    for one in (False, True):
        with V.Context(params, batch=True) as ctx:
            for d, q in enumerate(Q):
                assert V.vlbm_init_fields_device(ctx.ptr, d, q.data_ptr()) == V.VLBM_OK
            before = ctx.launches
            for n in (4, 36, 7):
                for _ in range(n if one else 1):
                    assert ctx.step(1 if one else n) == V.VLBM_OK
            passes.append(ctx.launches - before)
            assert ctx.sync() == V.VLBM_OK
            got.append([ctx.populations(np.arange(int(np.prod(s))), d) for d, s in enumerate(sides)])
    for a, b in zip(*got):
        assert np.array_equal(a, b)
    assert passes[0] < passes[1] == 47


def test_refused_second_buffer_takes_single_steps(V):
    """An allocator that has no second buffer to give: every step its own launch, same state."""
    import torch
    shape = (128, 128, 128)
    f0 = fields.ideal_fields(shape, 23, mach=0.5, beta=1.0, cfl=0.2, device=torch.device("cuda"))
    base = V.TorchHooks()
    big = 56 * int(np.prod(shape)) * 4
    seen = []

    def once(nbytes, stream, user):
        if nbytes >= big:
            seen.append(nbytes)
            if len(seen) > 1:
                return None
        return base.alloc(nbytes, stream, user)

    base_alloc = V.ALLOC_FN(once)

    class Hooks:
        alloc, dealloc = base_alloc, base.dealloc

    out = []
    for hooks in (Hooks, None):
        with V.Context(V.make_params(shape=shape, storage="f32", gamma=f0.gamma, tau=0.6, hooks=hooks)) as ctx:
            V.vlbm_init_fields_device(ctx.ptr, 0, f0.Q.data_ptr())
            n0 = ctx.launches
            assert ctx.step(8) == V.VLBM_OK and ctx.sync() == V.VLBM_OK
            out.append((ctx.launches - n0, populations(V, ctx, shape, 24)))
    assert len(seen) == 2 and out[0][0] == 8 and out[1][0] == 4
    assert np.array_equal(out[0][1], out[1][1])
