"""The one-block front of a build (extent, cube, keys, sort; up to 8192 particles)
and the general one above it: the order of the particles against numpy's stable
sort of the same keys, at sizes around the block's rounds, the rule's limit and
the general sort's (up to 96 tiles of 2048 without a scan kernel),
with shuffled, ordered, reversed and equal positions; builds of changing size on
one context (the table entries of the build before are cleared); and a captured
step replayed against eager ones."""
import numpy as np
import pytest

from paper_2206_11998_gb300 import inputs, lp

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from tests.gpu_util import ensure_built
    ensure_built()


SIZES = [1, 2, 33, 1023, 1024, 1025, 2049, 8191, 8192, 8193, 20000, 131071, 96 * 2048, 96 * 2048 + 1]


def _points(kind, d, n):
    x = np.random.Generator(np.random.PCG64(n + d)).uniform(-3.0, 5.0, (d, n))
    if kind == "ordered":
        x.sort(axis=1)
    elif kind == "reversed":
        x = -np.sort(x, axis=1)
    elif kind == "coarse":                     # many equal cells and, in 1D, equal keys
        x = np.round(x)
    elif kind == "point":
        x[:] = 0.25
    return x


def _keys(x):
    d, n = x.shape
    if d == 1:
        b = np.where(x[0] == 0.0, 0.0, x[0]).view(np.uint64)
        return np.where(b >> np.uint64(63), ~b, b | np.uint64(1 << 63)), 0
    lo = x.min(1)
    L = (x.max(1) - lo).max()
    L = L if L > 0 else 1.0
    q = np.clip(np.floor((x - lo[:, None]) * (2.0 ** 21 / L)), 0, 2 ** 21 - 1).astype(np.uint64)
    key = np.zeros(n, np.uint64)
    for b in range(21):
        for k in range(d):
            key |= ((q[k] >> np.uint64(b)) & np.uint64(1)) << np.uint64(d * b + k)
    return key, d * 21 - 27                    # ordered by the first 27 bits


@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("d", [1, 2, 3])
@pytest.mark.parametrize("kind", ["shuffled", "ordered", "reversed", "coarse", "point"])
def test_order_is_the_stable_sort_of_the_keys(kind, d, n):
    x = _points(kind, d, n)
    key, low = _keys(x)
    want = np.argsort(key >> np.uint64(low), kind="stable")
    xs = [torch.as_tensor(a, device="cuda") for a in x]
    ko = torch.empty(n, dtype=torch.int64, device="cuda")
    po = torch.empty(n, dtype=torch.int32, device="cuda")
    lp.sort_keys_noalloc(xs, ko, po)
    assert np.array_equal(po.cpu().numpy(), want)
    assert np.array_equal(ko.cpu().numpy().view(np.uint64), key[want])
    if d == 1 or kind == "point":
        return
    ctx = lp.Context(lp.make_config(d, n, radius_mode=lp.RADIUS_FIXED, radius=1e-3, k_max=4))
    st = {"x": list(x), "V": np.ones(n), "u": [np.zeros(n)] * d, "P": np.ones(n), "m": np.ones(n),
          "id": np.arange(n, dtype=np.uint32)}
    ps = lp.ParticleSet.from_state(st)
    ctx.build_neighbors(ps)
    assert np.array_equal(ps.id.cpu().numpy(), want)
    assert np.array_equal(ctx.export_neighbors(n)[4].cpu().numpy().view(np.uint64), key[want])
    ctx.close()


def test_builds_of_changing_size_on_one_context():
    cap = 12000
    one = lp.Context(lp.make_config(3, cap, kappa=2.2, k_max=64))
    for n in (9000, 500, 8192, 8193, 37, 12000, 4000):
        st = inputs.gas_cloud_3d(n, seed=n)
        lists = []
        for ctx in (one, lp.Context(lp.make_config(3, cap, kappa=2.2, k_max=64))):
            ps = lp.ParticleSet.from_state(st)
            ctx.build_neighbors(ps)
            cnt, tot, idx, d2, keys = ctx.export_neighbors(n)
            idx.masked_fill_(torch.arange(64, device="cuda") >= cnt[:, None], -1)
            lists.append([a.cpu().numpy() for a in (cnt, tot, idx, d2, keys, ps.id)])
        for a, b in zip(*lists):
            assert np.array_equal(a, b)


@pytest.mark.parametrize("n", [3000, 9000])
def test_replayed_steps_equal_eager_ones(n):
    st = inputs.gas_cloud_3d(n, seed=2)
    out = []
    for graph in (False, True):
        ctx = lp.Context(lp.make_config(3, n, kappa=2.2, k_max=64, gamma=5.0 / 3.0, s_ref=inputs.field_scales(st)))
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            ps = lp.ParticleSet.from_state(st)
            t = torch.zeros(1, dtype=torch.float64, device="cuda")
            ctx.step(ps, dt=0.0, cfl=0.3, t=t, stream=s)
            if graph:
                ctx.graph_capture(ps, dt=0.0, cfl=0.3, t=t, stream=s)
            for _ in range(5):
                ctx.graph_launch(stream=s) if graph else ctx.step(ps, dt=0.0, cfl=0.3, t=t, stream=s)
            s.synchronize()
        out.append([a.cpu().numpy() for a in (*ps.x, ps.V, *ps.u, ps.P, ps.id, t)])
        ctx.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)
