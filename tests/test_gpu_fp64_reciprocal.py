"""The reciprocals of the FP64 rotations are correctly rounded.  With one
neighbour a side in 1D a one-sided derivative is a single rotation: of offset d
and difference b it is ((d * (1 / (d d))) * b), every operation rounded once (the
scale of the stencil is a power of two).  Offsets of every size and mantissa,
bit for bit."""
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


@pytest.mark.parametrize("lo,hi", [(0, 0), (-40, 40), (-300, 300)])
def test_onesided_derivative_of_one_neighbour(lo, hi):
    n = 20000
    r = np.random.Generator(np.random.PCG64(hi))
    if hi == 0:
        x = np.cumsum(1.0 + r.uniform(0, 1, n))                  # mantissas over [1, 2)
    else:
        x = np.sort(np.concatenate([-np.exp2(r.uniform(lo, hi, n // 2)), np.exp2(r.uniform(lo, hi, n - n // 2))]))
    f = r.normal(size=n)
    st = {"x": [x], "V": np.ones(n), "u": [np.zeros(n)], "P": np.ones(n), "m": np.ones(n),
          "id": np.arange(n, dtype=np.uint32), "n_fluid": n}
    ctx = lp.Context(lp.make_config(1, n, precision=lp.PREC_FP64, radius_mode=lp.RADIUS_KSIDE, k_per_side=1, k_max=2))
    ps = lp.ParticleSet.from_state(st)
    ctx.build_neighbors(ps)
    got = ctx.onesided_derivs(ps, [torch.as_tensor(f, device="cuda")]).cpu().numpy()[:, 0, :, 0]
    ctx.close()
    i = np.arange(1, n - 1)
    for s, j in ((0, i - 1), (1, i + 1)):
        d, b = x[j] - x[i], f[j] - f[i]
        want = (d * (1.0 / (d * d))) * b
        assert np.array_equal(got[i, s], want), int((got[i, s] != want).sum())
