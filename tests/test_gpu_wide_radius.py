"""Neighbour lists in periodic boxes whose particles reach over more than 3/8 of
the box (up to the half that the minimum image allows): there the cells within
reach of a particle outnumber those of an axis, so a cell can be within reach at
two of its images.  Every path of the query against brute force in FP64, on sets
that the tiles finish alone and on sets left to the per-particle kernels."""
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


def _brute(x, V, k_max, octant):
    """Per particle: ids kept in (d2, id) order, number inside."""
    d, n = x.shape
    dx = x[:, None, :] - x[:, :, None]                    # [k][i][j] = x_j - x_i
    dx = np.where(dx > 0.5, dx - 1.0, np.where(dx < -0.5, dx + 1.0, dx))
    d2 = dx[0] * dx[0]
    for k in range(1, d):
        d2 = d2 + dx[k] * dx[k]
    w = V[:, None]                                        # m = kappa = 1
    inside = (d2 * d2) * d2 <= w * w if d == 3 else d2 * d2 <= w * w
    np.fill_diagonal(inside, False)
    oct_ = sum((dx[k] >= 0).astype(int) << k for k in range(d))
    out = []
    for i in range(n):
        j = np.flatnonzero(inside[i])
        j = j[np.lexsort((j, d2[i, j]))]
        total = len(j)
        if octant and total > k_max:
            o = oct_[i, j]
            rank = np.zeros(total, int)
            for q in range(1 << d):
                rank[o == q] = np.arange((o == q).sum())
            keep = np.sort(np.argsort(rank, kind="stable")[:k_max])
            j = j[keep]
        out.append((j[:k_max], total))
    return out


@pytest.mark.parametrize("octant", [False, True])
@pytest.mark.parametrize("mixed", [False, True])          # radii of every size: finer cells, cells split
@pytest.mark.parametrize("rad", [0.4, 0.45, 0.49])
@pytest.mark.parametrize("d,n", [(2, 20), (2, 60), (2, 300), (2, 2500), (3, 25), (3, 60), (3, 400), (3, 2500)])
def test_lists_match_brute_force(d, n, rad, mixed, octant):
    r = np.random.Generator(np.random.PCG64(n))
    x = r.uniform(0, 1, (d, n))
    if mixed:
        x[:, : n // 3] = 0.97 + 0.05 * x[:, : n // 3]     # a dense corner across the period
        x %= 1.0
    R = np.where(np.arange(n) % 4 == 0, 0.02, rad) if mixed else np.full(n, rad)
    V, k_max = R ** d, 64
    want = _brute(x, V, k_max, octant)
    st = {"x": list(x), "V": V, "u": [np.zeros(n)] * d, "P": np.ones(n), "m": np.ones(n),
          "id": np.arange(n, dtype=np.uint32), "n_fluid": n}
    for sched in (0, lp.SCHED_QUEUE_QUERY, lp.SCHED_QUERY_WARP):
        ctx = lp.Context(lp.make_config(d, n, kappa=1.0, k_max=k_max, periodic=(1,) * d + (0,) * (3 - d),
                                        box_hi=(1, 1, 1), select=lp.SELECT_OCTANT if octant else lp.SELECT_NEAREST))
        ctx.set_schedule(sched)
        ps = lp.ParticleSet.from_state(st)
        ctx.build_neighbors(ps)
        cnt, tot, idx, _, _ = (a.cpu().numpy() for a in ctx.export_neighbors(n))
        ids = ps.id.cpu().numpy()
        assert ctx.stats()["status"] & (1 << lp.ERR_ARG) == 0
        ctx.close()
        for q in range(n):
            j, total = want[ids[q]]
            assert tot[q] == min(total, 4 * k_max), (sched, q)
            assert np.array_equal(ids[idx[q, :cnt[q]]], j), (sched, q)
