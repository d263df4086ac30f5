"""The training loop (one launch, a grid barrier per minibatch) against the same
minibatches taken one by one through the gradient and Adam calls, and the
gradient's sums at sizes around the kernels' tiles (16 samples a warp, 128 a
block, 152 blocks).

A step's update is lr m / (sqrt(v) + eps).  The two paths sum a gradient in
different orders (relative 1e-6), and a weight that rounds to the other BF16
neighbour (relative 2^-8) changes a gradient by under 1 %, so a step's update by
under 1 % of lr; over the at most 24 steps here the parameters stay within
24 * 1 % * lr."""
import numpy as np
import pytest

from paper_2206_11998_gb300 import lp

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from tests.gpu_util import ensure_built
    ensure_built()


def _data(n, offset=0):
    g = torch.Generator(device="cuda").manual_seed(n)
    X = torch.randn(n * 8 + offset, generator=g, device="cuda")[offset:].view(n, 8)     # offset: a base off 16 bytes
    return X, (torch.rand(n, generator=g, device="cuda") < 0.3).float()


def _ctx():
    ctx = lp.Context(lp.make_config(3, 16, radius_mode=lp.RADIUS_FIXED, radius=0.1, k_max=8))
    ctx.mlp_set_params(lp.mlp_init_params(3))
    return ctx


@pytest.mark.parametrize("n,batch,epochs,offset", [(1, 1, 2, 0), (15, 16, 2, 0), (33, 16, 3, 1), (129, 128, 2, 0),
                                                   (4000, 1000, 2, 3), (30000, 8192, 3, 0), (50000, 1 << 20, 4, 0),
                                                   (2459, 103, 1, 0)])
def test_training_equals_single_steps(n, batch, epochs, offset):
    X, y = _data(n, offset)
    a, b = _ctx(), _ctx()
    losses = a.mlp_train(X, y, epochs, batch, 1e-2, 2.0)
    want = []
    for _ in range(epochs):
        total = 0.0
        for k in range(0, n, batch):
            g, loss = b.mlp_grad(X[k:k + batch], y[k:k + batch], 2.0)
            b.mlp_adam_step(g, 1e-2)
            total += float(loss.cpu()[0])
        want.append(total / -(-n // batch))
    assert np.allclose(losses, want, rtol=1e-2)
    pa, pb = a.mlp_get_params(), b.mlp_get_params()
    assert np.abs(pa[0] - pb[0]).max() < 24 * 1e-2 * 1e-2
    assert np.abs(pa[1] - pa[0]).max() <= np.abs(pa[0]).max() * 2.0 ** -8
    # a further call goes on from this one's moments and step count
    a.mlp_train(X, y, 1, batch, 1e-2, 2.0)
    assert np.isfinite(a.mlp_get_params()[0]).all()
    a.close()
    b.close()


@pytest.mark.parametrize("n", [1, 15, 16, 17, 127, 128, 129, 19455, 19456, 19457, 200001])
def test_gradient_matches_float64(n):
    X, y = _data(n)
    ctx = _ctx()
    w = torch.as_tensor(ctx.mlp_get_params()[1], device="cuda", dtype=torch.float64)
    g, loss = ctx.mlp_grad(X, y, 2.0)
    Xd, yd = X.double(), y.double()
    a = Xd @ w[:256].view(32, 8).T + w[256:288]
    h = a.clamp_min(0)
    z = h @ w[288:320] + w[320]
    cw = torch.where(yd > 0.5, 2.0, 1.0) / n
    dz = cw * (torch.sigmoid(z) - yd)
    dh = dz[:, None] * w[288:320] * (a > 0)
    ref = torch.cat([(dh.T @ Xd).reshape(-1), dh.sum(0), h.T @ dz, dz.sum()[None]])
    L = (cw * torch.nn.functional.softplus(torch.where(yd > 0.5, -z, z))).sum()
    # FP32 sums of n terms of size 1/n, some 10 flops each: a few 1e-6 of the terms' sum of magnitudes
    scale = torch.cat([(dh.abs().T @ Xd.abs()).reshape(-1), dh.abs().sum(0), h.T @ dz.abs(), dz.abs().sum()[None]])
    assert ((g.double() - ref).abs() <= 1e-5 * scale + 1e-12).all()
    assert abs(float(loss[0]) - float(L)) <= 1e-5 * float(L)
    ctx.close()
