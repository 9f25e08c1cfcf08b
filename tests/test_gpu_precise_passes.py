"""The channel's initial populations and moments, carried in split FP32, and the
domain sums, at the sizes and states where they could go wrong.

Initial populations are FP64 expressions rounded to FP32 once: the split form
keeps about 46 bits, so a population is the correctly rounded value or, next to
a rounding boundary, its neighbour (tolerance: half an ulp plus 2^-40 of the
largest term).  Moments are sums of 40 FP32 populations: exact up to a few
units of 2^-52 of the sum of magnitudes, FP64's own bound for adding them.
Domain sums of N cells: each CTA adds at most a few thousand values in FP64, so
N 2^-52 of the sum of magnitudes is far beyond what any order gives.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

C19 = np.array([(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0),
                (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1),
                (0, 1, -1), (0, -1, 1)], dtype=float)
W19 = np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12)


@pytest.fixture(scope="module")
def V():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2606_00641_gb300 import vlbm
    vlbm.load()
    return vlbm


def state(shape, seed, scale):
    rng = np.random.default_rng(seed)
    Q = rng.uniform(-1, 1, size=(7,) + shape) * scale
    Q[0] = rng.uniform(0.5, 2.0, size=shape)
    return Q


def equilibrium(Q, F):
    """[cells, 40] FP64 populations and the largest term of each."""
    q = Q.reshape(7, -1)
    rho, m, B = q[0], q[1:4], q[4:7]
    j = m - 0.5 * np.array(F)[:, None]
    u, v = m / rho, j / rho
    B2, v2 = (B * B).sum(0), (v * v).sum(0)
    out, big = [], []
    for c, w in zip(C19, W19):
        cv, cj, cB, c2 = c @ v, c @ j, c @ B, c @ c
        second = rho * (cv * cv - v2 / 3) + 0.5 * B2 * (c2 - 1) - (cB * cB - B2 / 3)
        out.append(w * (rho + 3 * cj + 4.5 * second))
        big.append(w * (rho + 3 * np.abs(j).sum(0) + 4.5 * (rho * v2 + 2 * B2)))
    for b in range(3):
        for i in range(7):
            a, s = (i - 1) // 2, 1.0 if i % 2 else -1.0
            phi = 0.0 if i == 0 or a == b else s * (u[a] * B[b] - B[a] * u[b])
            out.append((0.25 if i == 0 else 0.125) * (B[b] + 4 * phi))
            big.append(np.abs(B[b]) + np.abs(u).sum(0) * np.abs(B).sum(0))
    return np.array(out).T, np.array(big).T


@pytest.mark.parametrize("scale", [1e-8, 0.05, 0.5, 3e6])  # the last beyond the split form's range
@pytest.mark.parametrize("shape", [(1, 1, 1), (3, 5, 43), (2, 4, 128)])
def test_channel_init_is_fp64_rounded_once(V, shape, scale):
    F = (1e-5, -2e-6, 3e-7)
    Q = state(shape, 3, scale)
    p = V.make_params(model=V.VLBM_RESISTIVE, shape=shape, storage="f32", tau=[0.6, 0.7, 0.7, 0.7], force=F)
    with V.Context(p) as ctx:
        ctx.init_fields(Q)
        got = ctx.populations(np.arange(int(np.prod(shape))))
    ref, big = equilibrium(Q, F)
    tol = 0.5 * np.spacing(np.abs(ref).astype(np.float32)).astype(float) + 2.0 ** -40 * big
    assert (np.abs(got - ref) <= tol).all()


@pytest.mark.parametrize("steps", [0, 1, 2])
@pytest.mark.parametrize("walls", [False, True])
@pytest.mark.parametrize("shape", [(1, 3, 1), (3, 6, 43), (2, 4, 128)])
def test_channel_moments_are_fp64_sums(V, shape, walls, steps):
    F = (1e-5, -2e-6, 3e-7)
    Q = state(shape, 4, 0.03)
    bw = (0.01, 0.02, -0.03)
    p = V.make_params(model=V.VLBM_RESISTIVE, shape=shape, storage="f32", tau=[0.6, 0.7, 0.7, 0.7], force=F,
                      b_wall=bw, walls_y=walls)
    n = int(np.prod(shape))
    with V.Context(p) as ctx:
        ctx.init_fields(Q)
        ctx.step(steps)
        f = ctx.populations(np.arange(n))
        got = ctx.moments().reshape(7, n)
        sums = ctx.conservation()
    ref = np.empty((7, n))
    mag = np.empty((7, n))
    ref[0], mag[0] = f[:, :19].sum(1), np.abs(f[:, :19]).sum(1)
    for a in range(3):
        ref[1 + a] = f[:, :19] @ C19[:, a] + 0.5 * F[a]
        ref[4 + a] = f[:, 19 + 7 * a:26 + 7 * a].sum(1)
        mag[1 + a] = mag[0]
        mag[4 + a] = np.abs(f[:, 19 + 7 * a:26 + 7 * a]).sum(1)
    if walls:
        y = (np.arange(n) // shape[2]) % shape[1]
        on = (y == 0) | (y == shape[1] - 1)
        ref[:, on] = np.array([1.0, 0, 0, 0] + list(bw))[:, None]
    assert (np.abs(got - ref) <= 2.0 ** -47 * mag + 1e-300).all()
    assert (np.abs(sums - got.sum(1)) <= n * 2.0 ** -52 * mag.sum(1) + 1e-300).all()


def test_channel_moments_keep_what_is_not_finite(V):
    """A NaN or an infinity in one cell stays in that cell's moments and leaves the others as they were."""
    shape = (2, 3, 40)
    Q = state(shape, 5, 0.03)
    Q[0, 1, 1, 7] = np.inf
    Q[5, 0, 2, 3] = np.nan
    p = V.make_params(model=V.VLBM_RESISTIVE, shape=shape, storage="f32", tau=0.7)
    with V.Context(p) as ctx:
        ctx.init_fields(Q)
        got = ctx.moments()
    assert not np.isfinite(got[0, 1, 1, 7]) and np.isnan(got[5, 0, 2, 3])
    ok = np.ones(shape, bool)
    ok[1, 1, 7] = ok[0, 2, 3] = False
    assert np.abs(got - Q)[:, ok].max() < 1e-6


@pytest.mark.parametrize("storage", ["f64", "f32", "f16dev"])
@pytest.mark.parametrize("shape", [(1, 1), (1, 255), (16, 16), (1, 257), (7, 300), (640, 511)])
def test_domain_sums_over_block_edges(V, shape, storage):
    from paper_2606_00641_gb300 import fields
    Q = fields.uniform_ideal_state(shape, rho=1.2, u=(0.03, -0.02, 0.01), p=0.02, B=(0.05, 0.04, -0.03))
    Q[0] += 0.01 * np.random.default_rng(6).uniform(-1, 1, size=shape)
    ref = np.array([1.2, 0.04, -0.02, 0.01, 0.03, 0.05, 0.04, -0.03])
    p = V.make_params(shape=shape, storage=storage, tau=0.7, q_ref=ref, q_scale=0.01 + np.abs(ref))
    with V.Context(p) as ctx:
        ctx.init_fields(Q)
        for _ in range(2):
            got, m = ctx.conservation(), ctx.moments().reshape(8, -1)
            n = m.shape[1]
            assert (np.abs(got - m.sum(1)) <= (n + 8) * 2.0 ** -52 * np.abs(m).sum(1)).all()
            ctx.step(1)
