"""Steps chained on a stream of the caller (a launch is set up while the one before it
ends) against plain launches on the default stream: bit for bit the same populations and
sums, from one cell to several CTAs per SM, through direct launches and captured graphs,
with sums between the calls and a second state stepping on another stream."""
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


def prepared(V, model, shape, stream):
    if model == "channel":
        h = fields.hartmann_setup(shape, 5)
        Q = h.Q
        kw = dict(model=V.VLBM_RESISTIVE, tau=[h.tau_f] + [h.tau_m] * 3, force=h.force, b_wall=h.b_wall, walls_y=True)
    elif min(shape) < 4:
        Q = fields.uniform_ideal_state(shape, rho=1.1, u=(0.01, 0.02, 0.0), p=0.02, B=(0.01, 0.0, 0.02), gamma=1.5)
        kw = dict(gamma=1.5, tau=0.6)
    else:
        f0 = fields.ideal_fields(shape, 5, mach=0.3, cfl=0.1, k_rho=1, k_u=1, k_b=1)
        Q, kw = f0.Q, dict(gamma=f0.gamma, tau=0.6)
        if model == "powell":
            Q = np.concatenate([Q, 1e-3 * (Q[:1] - 1.0)])
            kw.update(model=V.VLBM_IDEAL_POWELL, tau_d=0.6, tau_m=1.5)
    ctx = V.Context(V.make_params(shape=shape, storage="f32", stream=stream, **kw))
    ctx.init_fields(np.ascontiguousarray(Q))
    return ctx


@pytest.mark.parametrize("model,shape", [("ideal", (1, 1)), ("ideal", (64, 64)), ("ideal", (150, 200)),
                                         ("ideal", (1, 5, 3)), ("ideal", (40, 41, 39)), ("ideal", (64, 128, 128)),
                                         ("powell", (12, 20, 33)), ("channel", (8, 32, 32)),
                                         ("channel", (20, 50, 60))])
def test_equals_plain_launches(V, model, shape):
    import torch
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    ctxs = [prepared(V, model, shape, s) for s in (None, streams[0].cuda_stream, streams[1].cuda_stream)]
    out = [[] for _ in ctxs]
    for n in (7, 70, 4):
        for ctx in ctxs:
            assert ctx.step(n) == V.VLBM_OK
        for ctx, o in zip(ctxs, out):
            o.append(np.array(ctx.conservation()))
    cells = np.arange(int(np.prod(shape)))
    for ctx, o in zip(ctxs, out):
        assert ctx.sync() == V.VLBM_OK
        o.append(ctx.populations(cells))
        ctx.close()
    for o in out[1:]:
        assert all(np.array_equal(a, b) for a, b in zip(out[0], o))
