"""The tcgen05 convolution's march along z: grids with fewer slices than CTAs, several
runs per CTA, columns of one tile's width, depths around the sixteen accumulator
blocks (where a plane's three blocks wrap), every column on the boundary.  Network
output and gradients against the FP64 reference under the kernels' BF16 storage, with
the repository's tolerance for that contract (1e-2 of the largest magnitude)."""
import numpy as np
import pytest

from oracle import closure_ref as ref

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def V():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2606_00641_gb300 import vlbm
    vlbm.load()
    return vlbm


def bf16(a):
    import torch
    return torch.as_tensor(np.asarray(a, dtype=np.float32)).bfloat16().double().numpy()


@pytest.mark.parametrize("shape", [(4, 16, 16), (8, 16, 16), (12, 32, 16), (16, 16, 32), (20, 16, 16), (36, 16, 16),
                                   (4, 64, 48), (160, 16, 16)])
def test_march_against_reference(V, shape):
    import torch
    rng = np.random.default_rng(9)
    Q = rng.uniform(-1, 1, size=(8,) + shape)
    mu, sigma, scale = np.zeros(8), np.ones(8), np.linspace(0.5, 2.0, 8)
    cl = V.Closure(shape, 5 / 3, 0.6, mu, sigma, scale)
    w = ref.init_params(rng, last_scale=1.0)
    for k in ("b1", "b2", "b3"):
        w[k] = rng.uniform(-0.2, 0.2, size=w[k].shape)
    flat = np.concatenate([w[k].ravel() for k in ("W1", "b1", "W2", "b2", "W3", "b3")]).astype(np.float32)
    cl.set_weights(flat)
    wb = {k: (bf16(v) if k[0] == "W" else v) for k, v in w.items()}
    Qd = torch.as_tensor(Q).cuda()
    n = int(np.prod(shape))
    out = torch.empty((n, 24), dtype=torch.float32, device="cuda")
    cl.forward(Qd.data_ptr(), out.data_ptr())
    y, cache = ref.net_forward(wb, bf16(ref.features(Q, mu, sigma)), store=bf16)
    want = ref.dphi_from_output(y, scale).reshape(24, n).T
    assert np.abs(out.cpu().numpy() - want).max() < 1e-2 * np.abs(want).max()
    gy = rng.uniform(-1, 1, size=(24,) + shape)
    gyd = torch.as_tensor(np.ascontiguousarray(gy.reshape(24, n).T), dtype=torch.float32).cuda()
    got = cl.backward(Qd.data_ptr(), gyd.data_ptr())
    g = ref.net_backward(wb, cache, bf16(gy), store=bf16)
    at = 0
    for k in ("W1", "b1", "W2", "b2", "W3", "b3"):
        part = got[at:at + g[k].size].reshape(g[k].shape)
        assert np.abs(part - g[k]).max() < 1e-2 * np.abs(g[k]).max(), k
        at += g[k].size
    cl.close()
