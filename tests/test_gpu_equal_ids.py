"""Particles that share ids: at equal distances and ids a list keeps its
neighbours in key order, so every path gives one list, the same on every run."""
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


def _want(x, ids, radius, k_max, octant):
    """Lists by (d2, id, place) of lattice particles x [n][d] (int, key order): idx [n][k_max] or -1, totals."""
    n, d = x.shape
    m = x.max() + 1
    at = np.full((m,) * d, -1, np.int64)
    at[tuple(x.T)] = np.arange(n)
    w = int(radius)
    o = np.stack(np.meshgrid(*[np.arange(-w, w + 1)] * d, indexing="ij")).reshape(d, -1).T
    d2 = (o * o).sum(1)
    o, d2 = o[(d2 > 0) & (d2 <= radius * radius)], d2[(d2 > 0) & (d2 <= radius * radius)]
    y = x[:, None, :] + o[None]
    ok = ((y >= 0) & (y < m)).all(2)
    j = np.where(ok, at[tuple(np.clip(y, 0, m - 1).transpose(2, 0, 1))], -1)
    big = 1 << 62
    key = np.where(j >= 0, (d2[None] * (int(ids.max()) + 1) + ids[j]) * n + j, big)
    s = np.argsort(key, axis=1, kind="stable")
    j, key = np.take_along_axis(j, s, 1), np.take_along_axis(key, s, 1)
    total = (key < big).sum(1)
    if octant:
        oc = ((o >= 0).astype(int) << np.arange(d)).sum(1)[s]
        rank = np.zeros(j.shape, np.int64)
        for q in range(1 << d):
            hit = (oc == q) & (key < big)
            rank = np.where(hit, np.cumsum(hit, 1) - 1, rank)
        pos = np.arange(j.shape[1])
        pick = np.where(key < big, rank * 4096 + pos, big)
        nth = np.sort(pick, 1)[:, min(k_max, pick.shape[1]) - 1]
        j = np.where((pick <= nth[:, None]) | (total[:, None] <= k_max), j, -1)
        s = np.argsort(j < 0, axis=1, kind="stable")
        j = np.take_along_axis(j, s, 1)
    j = np.pad(j, ((0, 0), (0, max(0, k_max - j.shape[1]))), constant_values=-1)[:, :k_max]
    return np.where(np.arange(k_max)[None] < np.minimum(total, k_max)[:, None], j, -1), total


@pytest.mark.parametrize("octant", [False, True])
@pytest.mark.parametrize("share", [1 << 30, 7, 1])            # all ids equal; runs of seven; no two equal
@pytest.mark.parametrize("d,m,radius,k_max", [(3, 16, 2.3, 64), (3, 16, 3.3, 20), (3, 16, 3.3, 80), (3, 16, 4.2, 50),
                                              (3, 47, 3.3, 40), (2, 60, 3.7, 16), (2, 60, 4.1, 64)])
def test_order_at_equal_distances_and_ids(d, m, radius, k_max, share, octant):
    g = np.stack(np.meshgrid(*[np.arange(m)] * d, indexing="ij")).reshape(d, -1)
    n = g.shape[1]
    st = {"x": list(g.astype(float)), "V": np.ones(n), "u": [np.zeros(n)] * d, "P": np.ones(n), "m": np.ones(n),
          "id": (np.arange(n) // share).astype(np.uint32), "n_fluid": n}
    want = None
    for sched in (0, lp.SCHED_QUEUE_QUERY, lp.SCHED_QUERY_WARP):
        ctx = lp.Context(lp.make_config(d, n, radius_mode=lp.RADIUS_FIXED, radius=radius, k_max=k_max,
                                        select=lp.SELECT_OCTANT if octant else lp.SELECT_NEAREST))
        ctx.set_schedule(sched)
        ps = lp.ParticleSet.from_state(st)
        ctx.build_neighbors(ps)
        cnt, tot, idx, _, _ = (a.cpu().numpy() for a in ctx.export_neighbors(n))
        if want is None:
            want = _want(np.stack([a.cpu().numpy() for a in ps.x], 1).astype(np.int64),
                         ps.id.cpu().numpy().astype(np.int64), radius, k_max, octant)
        ctx.close()
        idx = np.where(np.arange(k_max)[None] < cnt[:, None], idx, -1)
        assert np.array_equal(np.minimum(want[1], 4 * k_max), tot), sched
        bad = (idx != want[0]).any(1)
        assert not bad.any(), (sched, int(bad.sum()))
