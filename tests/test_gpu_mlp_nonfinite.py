"""Training samples that are not finite: a NaN activation is not positive, so a
sample with a NaN feature gives no gradient to W1, b1 and w2, and an infinite
feature none to the units it switches off (a particle without neighbours has such
features)."""
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


def _ctx(off_feature=None):
    ctx = lp.Context(lp.make_config(3, 16, radius_mode=lp.RADIUS_FIXED, radius=0.1, k_max=8))
    p = lp.mlp_init_params(3)
    if off_feature is not None:                       # every unit off where that feature is large
        p[:256].reshape(32, 8)[:, off_feature] = -1.0
    ctx.mlp_set_params(p)
    return ctx


def _data(n):
    g = torch.Generator(device="cuda").manual_seed(n)
    return torch.randn(n, 8, generator=g, device="cuda"), (torch.rand(n, generator=g, device="cuda") < 0.3).float()


@pytest.mark.parametrize("value,feature", [(float("nan"), 2), (float("nan"), 7), (float("inf"), 5)])
@pytest.mark.parametrize("n", [1, 16, 300, 20001])
def test_gradient(n, value, feature):
    X, y = _data(n)
    bad = torch.arange(0, n, 7)
    X[bad, feature] = value
    ctx = _ctx(None if np.isnan(value) else feature)
    w = torch.as_tensor(ctx.mlp_get_params()[1], device="cuda", dtype=torch.float64)
    g, loss = ctx.mlp_grad(X, y, 2.0)
    ctx.close()
    Xd, yd = X.double(), y.double()
    Xd[bad] = 0.0                                     # off: nothing of such a sample is used
    a = Xd @ w[:256].view(32, 8).T + w[256:288]
    a[bad] = -1.0
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


@pytest.mark.parametrize("n,batch", [(5000, 512), (20000, 20000)])
def test_training_stays_finite(n, batch):
    X, y = _data(n)
    X[::11, 3] = float("nan")
    ctx = _ctx()
    losses = ctx.mlp_train(X, y, 3, batch, 1e-2, 2.0)
    assert np.isfinite(losses).all() and np.isfinite(ctx.mlp_get_params()[0]).all()
    ctx.close()
