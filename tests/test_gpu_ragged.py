"""Steps on rows that no CTA width divides, where a CTA takes consecutive cells of a
plane across rows: row lengths around the CTA's 128 threads and its warps, planes of
one cell to several CTAs, against the oracle with the repository's tolerances
(relative L-infinity 1e-12 in FP64, 1e-5 in FP32)."""
import numpy as np
import pytest

import oracle
from paper_2606_00641_gb300 import fields

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def V():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2606_00641_gb300 import vlbm
    vlbm.load()
    oracle.build()
    return vlbm


def rel(got, ref):
    n = ref.shape[0]
    scale = np.abs(ref).reshape(n, -1).max(1)
    scale[1:4] = max(scale[1:4].max(), 1e-3)
    scale[5:8] = max(scale[5:8].max(), 1e-3)
    return (np.abs(got - ref).reshape(n, -1).max(1) / scale).max()


@pytest.mark.parametrize("steps", [2, 3])
@pytest.mark.parametrize("storage,tol", [("f64", 1e-12), ("f32", 1e-5)])
@pytest.mark.parametrize("shape", [(9, 3), (5, 31), (7, 33), (3, 64), (3, 127), (2, 129), (3, 130), (2, 255), (1, 257),
                                   (4, 5, 3), (3, 4, 43), (2, 3, 64), (3, 2, 129), (2, 1, 300)])
def test_ideal_rows_of_any_length(V, shape, storage, tol, steps):
    f0 = fields.ideal_fields(shape, 11, mach=0.3, cfl=0.1, k_rho=1, k_u=1, k_b=1)
    p = V.make_params(shape=shape, storage=storage, gamma=f0.gamma, tau=0.6)
    with V.Context(p) as ctx:
        ctx.init_fields(f0.Q)
        assert ctx.step(steps) == V.VLBM_OK
        got = ctx.moments()
    assert rel(got, oracle.ideal_run(f0.Q, f0.gamma, 0.6, steps)) < tol


def test_division_by_any_row_length(V):
    """Cell numbers of large planes: a step of a uniform state shifted by one marked cell ends in its neighbours."""
    for nx, ny in ((1000, 997), (65537, 3), (3, 65535)):
        Q = fields.uniform_ideal_state((ny, nx), rho=1.0, u=(0.0, 0.0, 0.0), p=0.02, B=(0.0, 0.0, 0.0))
        y, x = ny - 2, nx - 2
        Q[0, y, x] += 0.01
        p = V.make_params(shape=(ny, nx), storage="f64", tau=1.0)
        with V.Context(p) as ctx:
            ctx.init_fields(Q)
            ctx.step(1)
            d = ctx.moments()[0] - 1.0
        where = {(int(a), int(b)) for a, b in zip(*np.nonzero(np.abs(d) > 1e-9))}
        assert where == {(y, x), (y, x - 1), (y, x + 1), (y - 1, x), (y + 1, x)}
