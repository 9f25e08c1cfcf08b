"""The channel's initial populations are the FP64 expressions' values rounded to FP32 once, also
next to a rounding boundary.

The FP64 expressions add fewer than eight rounded terms, each at most the largest one, so they
are within 2^-50 of it: a population is asserted to be the correctly rounded value wherever that
does not change over +-2^-50 of the largest term.  The reference is formed in extended precision.
States: densities whose populations lie 2^-50 to 2^-42 from the middle of two floats along each
class of directions, and random ones with large velocities and fields."""
import numpy as np
import pytest

from test_gpu_precise_passes import C19, V, W19  # noqa: F401

pytestmark = pytest.mark.gpu

F = (1e-5, -2e-6, 3e-7)


def near_ties(n, w, seed):
    rng = np.random.default_rng(seed)
    t = rng.uniform(0.5, 2.0, n).astype(np.float32) * np.float32(w)
    mid = (t.astype(float) + np.nextafter(t, np.float32(9)).astype(float)) / 2
    delta = 2.0 ** rng.uniform(-50, -42, n) * rng.choice([-1.0, 1.0], n)
    Q = np.zeros((7, n))
    Q[0] = mid * (1.0 + delta) / w
    Q[1:4] = 0.5 * np.array(F)[:, None]
    return Q


def random_states(n, scale, seed):
    rng = np.random.default_rng(seed)
    Q = rng.uniform(-1, 1, size=(7, n)) * scale
    Q[0] = rng.uniform(0.5, 2.0, n)
    Q[1:, rng.random(n) < 0.2] = 0.0
    # tiny components among ordinary ones, and cells of tiny components only
    Q[1 + rng.integers(0, 6, n), np.arange(n)] *= 10.0 ** rng.uniform(-32, -10, n)
    Q[1:, ::50] *= 10.0 ** rng.uniform(-24, -8, (n + 49) // 50)
    return Q


def reference(Q):
    L = np.longdouble
    q, one = Q.astype(L), L(1)
    rho, m, B = q[0], q[1:4], q[4:7]
    j = m - (0.5 * np.array(F)).astype(L)[:, None]
    u, v = m / rho, j / rho
    B2, v2 = (B * B).sum(0), (v * v).sum(0)
    out, big = [], []
    for i in range(19):
        c = C19[i].astype(L)
        w = one / (3 if i == 0 else 18 if i <= 6 else 36)
        cv, cj, cB = c @ v, c @ j, c @ B
        out.append(w * (rho + 3 * cj + L(4.5) * (rho * (cv * cv - v2 / 3) + B2 * (c @ c - 1) / 2 - (cB * cB - B2 / 3))))
        big.append(w * (rho + 3 * np.abs(j).sum(0) + L(4.5) * (rho * v2 + 2 * B2)))
    for b in range(3):
        for i in range(7):
            a, s = (i - 1) // 2, 1 if i % 2 else -1
            x, y = (0 * rho, 0 * rho) if i == 0 or a == b else (u[a] * B[b], B[a] * u[b])
            w = one / (4 if i == 0 else 8)
            out.append(w * (B[b] + 4 * s * (x - y)))
            big.append(w * (np.abs(B[b]) + 4 * (np.abs(x) + np.abs(y))))
    return np.array(out), np.array(big)


@pytest.mark.parametrize("what", ["1/3", "1/18", "1/36", "random 0.1", "random 1.5"])
def test_channel_init_is_correctly_rounded(V, what):  # noqa: F811
    nx, ny, nz = 128, 16, 16
    n = nx * ny * nz
    kind, _, arg = what.partition(" ")
    Q = random_states(n, float(arg), 8) if arg else near_ties(n, 1.0 / float(kind.split("/")[1]), 7)
    p = V.make_params(model=V.VLBM_RESISTIVE, shape=(nz, ny, nx), storage="f32", tau=[0.6, 0.7, 0.7, 0.7], force=F)
    with V.Context(p) as ctx:
        ctx.init_fields(Q.reshape(7, nz, ny, nx))
        got = ctx.populations(np.arange(n)).T.astype(np.float32)
    ref, big = reference(Q)
    slack = big * np.longdouble(2.0) ** -50
    lo, hi = (ref - slack).astype(np.float32), (ref + slack).astype(np.float32)
    sure = lo == hi
    assert sure.mean() > 0.9
    bad = sure & (got != lo)
    assert not bad.any(), (int(bad.sum()), np.unique(np.nonzero(bad)[0]))
