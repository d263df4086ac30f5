"""Calls that take another kernel by the size of the set: the same particles alone
(below the rule's line) and beside others far away (above it) have the same
neighbours, so their results are the same bit for bit.  And neighbour lists of
many particles that the blocks put off for their warps, against the
warp-per-particle query."""
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


def _state(x):
    n = x.shape[1]
    return {"x": list(x), "V": np.ones(n), "u": [np.zeros(n)] * x.shape[0], "P": np.ones(n), "m": np.ones(n),
            "id": np.arange(n, dtype=np.uint32), "n_fluid": n}


def _set(d, n, extra, seed):
    """n random particles in a box with about 20 (2D) or 40 (3D) per unit ball, and extra ones on a far, wide lattice."""
    r = np.random.Generator(np.random.PCG64(seed))
    box = (n * {1: 1.0, 2: np.pi / 20, 3: 4 * np.pi / 3 / 40}[d]) ** (1 / d)
    x = np.sort(r.uniform(0, box, (1, n))) if d == 1 else r.uniform(0, box, (d, n))
    if extra:
        m = int(np.ceil(extra ** (1 / d)))
        g = np.stack(np.meshgrid(*[1.1 * np.arange(m)] * d, indexing="ij")).reshape(d, -1)[:, :extra]
        x = np.concatenate([x, g + 2 * box + 100], 1)
    return x


def _run(d, x, n, fields, call, **cfg):
    """Results of the first n particles by id, and whether their lists were whole."""
    ctx = lp.Context(lp.make_config(d, x.shape[1], radius_mode=lp.RADIUS_FIXED, radius=1.0, k_max=64, **cfg))
    ps = lp.ParticleSet.from_state(_state(x))
    ctx.build_neighbors(ps)
    f = [torch.cos((1 + 0.3 * q) * ps.x[0]) + ps.x[-1] ** 2 * 1e-3 for q in range(fields)]
    out = call(ctx, ps, f)
    ids = ps.id.long()
    out = out if isinstance(out, tuple) else (out,)
    res = []
    for o in out:
        ax = 1 if o.dim() == 3 else 0                # derivs [field][particle][u]; others by particle first
        back = torch.empty_like(o)
        back.index_copy_(ax, ids, o)
        res.append(back.narrow(ax, 0, n).cpu().numpy())
    ctx.close()
    return res


def _derivs(ctx, ps, f):
    status = torch.zeros(ps.n, dtype=torch.int32, device="cuda")
    return ctx.gfd_derivs(ps, f, status=status), status


@pytest.mark.parametrize("refine", [lp.REFINE_AUTO, lp.REFINE_ALWAYS, lp.REFINE_NEVER])
@pytest.mark.parametrize("d,fields,n,total", [(3, 1, 30000, 400000), (3, 5, 30000, 400000), (3, 7, 30000, 400001),
                                              (2, 3, 30000, 1500000)])
def test_derivs(d, fields, n, total, refine):
    a = _run(d, _set(d, n, 0, n), n, fields, _derivs, refine=refine)
    b = _run(d, _set(d, n, total - n, n), n, fields, _derivs, refine=refine)
    for p, q in zip(a, b):
        assert np.array_equal(p, q)


@pytest.mark.parametrize("d,fields,n,total", [(3, 5, 30000, 65536), (3, 2, 1000, 65537), (2, 5, 30000, 131072),
                                              (2, 1, 131071, 140001)])
def test_onesided(d, fields, n, total):
    call = lambda ctx, ps, f: ctx.onesided_derivs(ps, f)
    a = _run(d, _set(d, n, 0, n), n, fields, call)
    b = _run(d, _set(d, n, total - n, n), n, fields, call)
    assert np.array_equal(a[0], b[0])


@pytest.mark.parametrize("d,clumps,size", [(3, 18, 2500), (2, 18, 2500), (3, 41, 2500)])
def test_lists_that_blocks_put_off(d, clumps, size):
    # (a clump's particles fill one bin of distances past a block's buffer)
    r = np.random.Generator(np.random.PCG64(size))
    x = np.repeat(3.0 * np.arange(clumps)[None] + np.arange(d)[:, None], size, 1)
    x = np.concatenate([x, r.uniform(0, 3 * clumps, (d, 1000))], 1)
    out = []
    for sched in (lp.SCHED_QUERY_WARP, 0):
        ctx = lp.Context(lp.make_config(d, x.shape[1], radius_mode=lp.RADIUS_FIXED, radius=1.0, k_max=24))
        ctx.set_schedule(sched)
        ps = lp.ParticleSet.from_state(_state(x))
        ctx.build_neighbors(ps)
        cnt, tot, idx, d2, _ = ctx.export_neighbors(ps.n)
        idx.masked_fill_(torch.arange(24, device="cuda") >= cnt[:, None], -1)
        out.append([a.cpu().numpy() for a in (cnt, tot, idx, d2, ps.id)])
        ctx.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)
