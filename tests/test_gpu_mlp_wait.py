"""The training launch's wait for its blocks: where it runs out the call fails,
whatever the host does with denormal floats, the weights, moments and step count
stay together, and later training goes on as if the call had not been.
Minibatches of up to 128 samples run in one block, whose sums have one order, so
these results are compared bit for bit."""
import ctypes

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


def _data(n):
    g = torch.Generator(device="cuda").manual_seed(n)
    return torch.randn(n, 8, generator=g, device="cuda"), (torch.rand(n, generator=g, device="cuda") < 0.3).float()


def _ctx():
    ctx = lp.Context(lp.make_config(3, 16, radius_mode=lp.RADIUS_FIXED, radius=0.1, k_max=8))
    ctx.mlp_set_params(lp.mlp_init_params(3))
    return ctx


DEFAULT = 1 << 22


@pytest.mark.parametrize("flush", [False, True])
@pytest.mark.parametrize("n,batch", [(1000, 128), (20000, 20000)])
def test_a_wait_that_runs_out(n, batch, flush):
    X, y = _data(n)
    a, b = _ctx(), _ctx()
    for c in (a, b):
        c.mlp_train(X[:500], y[:500], 2, 100, 1e-2, 2.0)
    before = a.mlp_get_params()
    a.mlp_wait_limit(0)
    torch.set_flush_denormal(flush)
    try:
        with pytest.raises(lp.LPError) as e:
            a.mlp_train(X, y, 3, batch, 1e-2, 2.0)
    finally:
        torch.set_flush_denormal(False)
    assert e.value.code == lp.ERR_TIMEOUT and a.stats()["status"] & (1 << lp.ERR_TIMEOUT)
    # without the losses nothing waits for the launch: the status word tells, and
    # the launches after the first (of 1024 epochs) are left out
    rc = lp.lib().lp_mlp_train(a.h, ctypes.c_void_p(X.data_ptr()), ctypes.c_void_p(y.data_ptr()), n, 2100, batch, 1e-2,
                               2.0, None, ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert rc == lp.OK
    for p, q in zip(before, a.mlp_get_params()):
        assert np.array_equal(p, q)
    a.mlp_wait_limit(DEFAULT)
    la, lb = (c.mlp_train(X[:500], y[:500], 3, 100, 1e-2, 2.0) for c in (a, b))
    assert np.array_equal(la, lb)
    for p, q in zip(a.mlp_get_params(), b.mlp_get_params()):
        assert np.array_equal(p, q)
    a.close()
    b.close()


def test_more_epochs_than_a_launch_takes():
    X, y = _data(100)
    a, b = _ctx(), _ctx()
    la = a.mlp_train(X, y, 2100, 40, 1e-3, 2.0)
    lb = np.concatenate([b.mlp_train(X, y, k, 40, 1e-3, 2.0) for k in (1000, 24, 1, 1075)])
    assert np.array_equal(la, lb)
    for p, q in zip(a.mlp_get_params(), b.mlp_get_params()):
        assert np.array_equal(p, q)
    a.close()
    b.close()


def test_training_and_single_steps_share_the_step_count():
    X, y = _data(128)
    a, b = _ctx(), _ctx()
    a.mlp_train(X, y, 2, 128, 1e-2, 2.0)
    for _ in range(2):
        b.mlp_adam_step(b.mlp_grad(X, y, 2.0)[0], 1e-2)
    for c in (a, b):
        g, _ = c.mlp_grad(X, y, 2.0)
        c.mlp_adam_step(g, 1e-2)
        c.mlp_train(X, y, 1, 128, 1e-2, 2.0)
    # (the two kernels may contract an update's operations differently: a few
    # roundings of values below 1)
    assert np.abs(a.mlp_get_params()[0] - b.mlp_get_params()[0]).max() < 1e-5
    a.close()
    b.close()
