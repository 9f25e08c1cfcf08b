"""The closure's network in whole numbers, over grids where a CTA of the tcgen05
convolution marches far enough to take every accumulator block and every entry of
the plane ring again (more than 16, and more than 32, slices a CTA, so that each
barrier flips its parity twice, and the blocks wrap).

Features, weights and output gradients are small integers and hidden
pre-activations multiples of 32, so that tanh gives -1, 0 or 1 and every sum of
products is a whole number below 2^24: exact in FP32 in any order, and equal to
the sums formed in FP64.  Hidden-layer gradients are kept in BF16, one rounding of
a whole number.  Everything is therefore compared for equality; an update lost or
doubled between two planes of the march would show as an integer."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

TAPS = [(dx, dy, dz) for dz in (-1, 0, 1) for dy in (-1, 0, 1) for dx in (-1, 0, 1)]


@pytest.fixture(scope="module")
def V():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2606_00641_gb300 import vlbm
    vlbm.load()
    return vlbm


def shifted(x, e, sign):
    import torch
    dx, dy, dz = e
    return torch.roll(x, (-sign * dz, -sign * dy, -sign * dx), (-3, -2, -1)).reshape(x.shape[0], -1)


def conv(x, W, sign=1):
    """sum_{c, t} W[o, c, t] x[c, p + sign e_t] in FP64."""
    y = sum(W[:, :, t] @ shifted(x, e, sign) for t, e in enumerate(TAPS))
    return y.reshape((W.shape[0],) + x.shape[1:])


def weight_grad(g, x):
    import torch
    flat = g.reshape(g.shape[0], -1)
    return torch.stack([flat @ shifted(x, e, 1).T for e in TAPS], dim=2)


def slices_per_cta(shape):
    import torch
    nz, ny, nx = shape
    slices = nx // 8 * (ny // 16) * nz
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    return slices / min(slices, sms, max(64, slices // 4))


@pytest.mark.parametrize("shape,march", [((128, 64, 48), 17), ((128, 64, 80), 33)])
def test_long_march_is_exact(V, shape, march):
    import torch
    assert slices_per_cta(shape) > march
    rng = np.random.default_rng(41)
    ints = lambda *size: rng.integers(-1, 2, size=size).astype(float)
    n = int(np.prod(shape))
    Q = ints(8, *shape)
    w = {"W1": 32 * ints(32, 8, 27), "b1": 32 * ints(32), "W2": 32 * ints(32, 32, 27), "b2": 32 * ints(32),
         "W3": ints(24, 32, 27), "b3": ints(24)}
    gy = ints(24, *shape) * (rng.random((24,) + shape) < 0.04)
    D = {k: torch.as_tensor(v, device="cuda") for k, v in w.items()}
    x, g = torch.as_tensor(Q, device="cuda"), torch.as_tensor(gy, device="cuda")

    def act(z, b):
        return torch.tanh(z + b[:, None, None, None]).bfloat16().double()

    def keep(z, a):
        return (z * (1.0 - a * a)).bfloat16().double()

    a1 = act(conv(x, D["W1"]), D["b1"])
    a2 = act(conv(a1, D["W2"]), D["b2"])
    assert set(torch.unique(torch.cat([a1, a2])).tolist()) == {-1.0, 0.0, 1.0}
    y = conv(a2, D["W3"]) + D["b3"][:, None, None, None]
    gz2 = keep(conv(g, D["W3"].transpose(0, 1).contiguous(), -1), a2)
    gz1 = keep(conv(gz2, D["W2"].transpose(0, 1).contiguous(), -1), a1)
    want = [weight_grad(gz1, x), gz1.sum((1, 2, 3)), weight_grad(gz2, a1), gz2.sum((1, 2, 3)),
            weight_grad(g, a2), g.sum((1, 2, 3))]
    # every partial sum of the gradients is a whole number below 2^24 (the other factor is -1, 0 or 1)
    assert all(t.abs().sum((1, 2, 3)).max() < 2 ** 24 for t in (gz1, gz2, g))
    assert gz2.count_nonzero() > 1000 and gz1.count_nonzero() > 1000

    cl = V.Closure(shape, 5 / 3, 0.6, np.zeros(8), np.ones(8), np.ones(8))
    cl.set_weights(np.concatenate([w[k].ravel() for k in ("W1", "b1", "W2", "b2", "W3", "b3")]).astype(np.float32))
    gyd = torch.as_tensor(np.ascontiguousarray(gy.reshape(24, n).T), dtype=torch.float32, device="cuda")
    flat = np.concatenate([t.cpu().numpy().ravel() for t in want])
    for _ in range(3):
        out = torch.full((n, 24), -1.0, dtype=torch.float32, device="cuda")
        cl.forward(x.data_ptr(), out.data_ptr())
        assert torch.equal(out.double(), y.reshape(24, n).T)
        assert np.array_equal(np.asarray(cl.backward(x.data_ptr(), gyd.data_ptr()), dtype=float), flat)
    cl.close()
