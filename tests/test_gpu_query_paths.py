"""The neighbour query's paths against one another: tiles (with the parts of
too-large groups and the left-over particles) and the tiles of the work queue
give the lists of the warp-per-particle query, bit for bit, on particle sets
that reach each of them: scattered and dense regions, lists of more than 64,
128 and 1024 in-radius particles, equal distances past the buffer, equal ids,
periodic boxes small against the radius, and the smallest sets."""
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


def _points(pts, radius=None, ids=None):
    """Particles at pts; radius: per-particle radii through the volume rule with kappa = 1 and m = 1."""
    pts = np.atleast_2d(np.asarray(pts, float))
    d, n = pts.shape
    V = np.ones(n) if radius is None else np.broadcast_to(radius, (n,)).astype(float) ** d
    st = {"x": [a.copy() for a in pts], "V": V, "u": [np.zeros(n) for _ in range(d)], "P": np.ones(n), "m": np.ones(n),
          "id": np.arange(n, dtype=np.uint32) if ids is None else ids.astype(np.uint32), "n_fluid": n}
    return st


def _rng(k):
    return np.random.Generator(np.random.PCG64(k))


def _cases():
    r = _rng(1)
    yield "cloud-20k", inputs.gas_cloud_3d(20037, seed=3), dict(dim=3, kappa=2.2, k_max=64)
    yield "cloud-tail", inputs.gas_cloud_3d(30011, seed=4, r_max_sigma=0), dict(dim=3, kappa=2.6, k_max=80)
    yield "few-kept", inputs.gas_cloud_3d(5000, seed=5), dict(dim=3, kappa=4.0, k_max=7)
    yield "jet", inputs.jet_snapshot_3d(40000, seed=6), dict(dim=3, kappa=2.2, k_max=80)
    yield "jet-octant", inputs.jet_snapshot_3d(40000, seed=6), dict(dim=3, kappa=2.2, k_max=80, select=lp.SELECT_OCTANT)
    # a dense ball inside a sparse box: counts from a few to thousands, radii of every size
    p = np.concatenate([r.normal(0, 0.02, (3, 6000)), r.uniform(-1, 1, (3, 3000))], 1)
    yield "dense-core", _points(p, r.uniform(0.01, 0.5, 9000)), dict(dim=3, kappa=1.0, k_max=64)
    # an exact lattice: shells of equal distances, cut inside a shell and past the 128-entry buffer
    g = np.stack(np.meshgrid(*[np.arange(16.0)] * 3, indexing="ij")).reshape(3, -1)
    for rad, km in ((2.3, 64), (3.3, 20), (3.3, 80), (4.2, 50), (7.1, 64)):
        yield "lattice-%g-%d" % (rad, km), _points(g), dict(dim=3, radius_mode=lp.RADIUS_FIXED, radius=rad, k_max=km)
    # every particle at the same distance of the middle one: a run of ties longer than the buffer
    q = r.normal(size=(3, 400))
    q = np.concatenate([np.round(q / np.abs(q).max(0)), np.zeros((3, 1))], 1)
    yield "shell", _points(q), dict(dim=3, radius_mode=lp.RADIUS_FIXED, radius=1.8, k_max=30)
    yield "equal-ids", dict(inputs.gas_cloud_3d(3000, seed=8), id=np.zeros(3000, np.uint32)), dict(dim=3, kappa=5.0, k_max=64)
    for n in (1, 2, 31, 32, 33, 127, 129):
        yield "n%d" % n, _points(r.uniform(0, 1, (3, n)), 0.8), dict(dim=3, kappa=1.0, k_max=64)
    # periodic boxes: regions far below, near and above half a period
    for rad in (0.02, 0.1, 0.2, 0.24, 0.3, 0.49):
        n = 4000 if rad < 0.15 else 600
        yield "periodic-%g" % rad, _points(r.uniform(0, 1, (2, n)), rad), dict(dim=2, kappa=1.0, k_max=40,
                                                                               periodic=(1, 1, 0), box_hi=(1, 1, 1))
    yield "periodic-3d", _points(r.uniform(0, 1, (3, 4000)), r.uniform(0.05, 0.3, 4000)), dict(
        dim=3, kappa=1.0, k_max=64, periodic=(1, 1, 1), box_hi=(1, 1, 1))
    yield "kh", inputs.kh_2d(30000, 0.03, seed=9), dict(dim=2, kappa=2.2, k_max=40, periodic=(1, 1, 0), box_hi=(1, 1, 1))
    # more particles at one point than the left-over particles' buffers hold: all in one bin
    p = np.concatenate([np.full((3, 1500), 0.5), r.uniform(0, 1, (3, 1500))], 1)
    yield "clump", _points(p, 0.2), dict(dim=3, kappa=1.0, k_max=40)
    # as above past the size where the left-over particles change to the smaller blocks
    p = np.concatenate([r.normal(0, 0.02, (3, 12000)), r.uniform(-1, 1, (3, 89000))], 1)
    yield "dense-core-many", _points(p, r.uniform(0.01, 0.2, 101000)), dict(dim=3, kappa=1.0, k_max=64)
    g = np.stack(np.meshgrid(*[np.arange(47.0)] * 3, indexing="ij")).reshape(3, -1)
    for rad, km in ((3.3, 80), (4.2, 50), (5.1, 20)):
        yield "lattice-many-%g" % rad, _points(g), dict(dim=3, radius_mode=lp.RADIUS_FIXED, radius=rad, k_max=km)
    yield "few-kept-2d-many", _points(r.uniform(0, 1, (2, 100000)), 0.03), dict(dim=2, kappa=1.0, k_max=9)
    yield "scattered-2d", _points(r.normal(size=(2, 3000)) ** 5, r.uniform(0.01, 3.0, 3000)), dict(dim=2, kappa=1.0, k_max=33)


OCTANT = ("cloud-20k", "few-kept", "dense-core", "clump", "lattice-2.3-64", "lattice-3.3-20", "lattice-3.3-80", "lattice-4.2-50",
          "lattice-7.1-64", "shell", "n1", "n33", "n129", "periodic-0.2", "periodic-0.49", "periodic-3d", "kh", "scattered-2d")

ALL = list(_cases())
ALL += [(name + "-octant", st, dict(cfg, select=lp.SELECT_OCTANT)) for name, st, cfg in ALL if name in OCTANT]


@pytest.mark.parametrize("name,st,cfg", ALL, ids=[c[0] for c in ALL])
def test_query_paths_agree(name, st, cfg):
    out = []
    for sched in (lp.SCHED_QUERY_WARP, 0, lp.SCHED_QUEUE_QUERY):
        ctx = lp.Context(lp.make_config(capacity=st["V"].shape[0], **cfg))
        ctx.set_schedule(sched)
        ps = lp.ParticleSet.from_state(st)
        ctx.build_neighbors(ps)
        cnt, tot, idx, d2, keys = ctx.export_neighbors(ps.n)
        idx.masked_fill_(torch.arange(cfg["k_max"], device="cuda") >= cnt[:, None], -1)
        out.append([a.cpu().numpy() for a in (cnt, tot, idx, d2, keys, ps.id)])
        ctx.close()
    if name == "equal-ids":            # equal distances are then in no order: compare the sets
        out = [[o[0], o[1], np.sort(o[2], 1), o[3]] for o in out]
    for o in out[1:]:
        for a, b, what in zip(out[0], o, ("count", "total", "idx", "d2min", "keys", "id")):
            assert np.array_equal(a, b), (what, int((a != b).sum()))
