"""Device words that a call leaves for the next one (counts of finished blocks,
extents, smallest time steps) are not trusted: overlapping calls, which corrupt
each other's results, may leave anything in them, and the calls after those must
be right again.  The words are found through captured kernels' parameters and
overwritten with values that no call leaves behind."""
import struct

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


def _find(kernels, name):
    return next(p for k, p in kernels if name in k)


@pytest.mark.parametrize("d", [1, 2, 3])
def test_sort_keys_noalloc(d):
    from tests.graph_util import captured_kernels, pointer_param, poke
    from tests.test_gpu_small_front import _keys
    n = 20000                                            # above the one-block front
    x = np.random.Generator(np.random.PCG64(d)).uniform(0, 1, (d, n))
    keys = torch.empty(n, dtype=torch.int64, device="cuda")
    perm = torch.empty(n, dtype=torch.int32, device="cuda")

    pts = {c: [torch.as_tensor(c * a, device="cuda") for a in x] for c in (1.0, 0.375)}

    def sort(scale, stream=None):
        lp.sort_keys_noalloc(pts[scale], keys, perm, stream=stream)
    sort(1.0)
    kernels, graph = captured_kernels(lambda s: sort(1.0, s))
    ext = pointer_param(_find(kernels, "k_init_extent"), 0)
    poke(ext + 64, struct.pack("<I", 1000000))           # the block count, behind the eight extent words
    sort(0.375)                                          # another cube than the last call's
    got = keys.cpu().numpy().view(np.uint64)
    key, lo_bit = _keys(0.375 * x)
    order = np.argsort(key >> np.uint64(lo_bit), kind="stable")
    assert np.array_equal(got, key[order])


def _state(d, n):
    x = np.random.Generator(np.random.PCG64(n)).uniform(0, 1, (d, n))
    return {"x": list(x), "V": np.full(n, 1.0 / n), "u": list(0.0 * x), "P": np.ones(n), "m": np.ones(n),
            "id": np.arange(n, dtype=np.uint32), "n_fluid": n}


@pytest.mark.parametrize("nsim", [1, 3])
def test_context(nsim):
    from tests.graph_util import captured_kernels, pointer_param, poke
    d, n = 2, 30000
    off = torch.tensor([n * k // nsim for k in range(nsim + 1)], dtype=torch.int64, device="cuda")
    results = []
    for spoil in (False, True):
        ctx = lp.Context(lp.make_config(d, n, kappa=1.6, max_sims=nsim))
        ps = lp.ParticleSet.from_state(_state(d, n))
        t = torch.zeros(nsim, dtype=torch.float64, device="cuda")
        step = lambda stream=None: ctx.step_batched(ps, off, nsim, cfl=1e-3, t=t, stream=stream)
        step()
        kernels, graph = captured_kernels(step)
        begin, cfl = _find(kernels, "k_begin"), _find(kernels, "k_cfl")
        ext, tickets, dt_min = pointer_param(begin, 5), pointer_param(begin, 9), pointer_param(cfl, 8)
        assert pointer_param(cfl, 15) == tickets + 4
        if spoil:
            poke(tickets, struct.pack("<II", 1000000, 1000000))
            poke(dt_min, struct.pack("<d", 1e-12) * nsim)
            # extents [-2, 3] in order keys: larger than the particles'
            key = lambda v: (lambda b: b ^ (1 << 63 if b >> 63 == 0 else (1 << 64) - 1))(
                struct.unpack("<Q", struct.pack("<d", v))[0])
            for s in range(nsim):
                poke(ext + 64 * s, struct.pack("<6Q", *([key(-2.0)] * 3 + [key(3.0)] * 3)))
        step()                                           # may still be wrong ...
        ps = lp.ParticleSet.from_state({**_state(d, n), "x": [0.4 * a for a in _state(d, n)["x"]]})
        step()                                           # ... the next one is right
        results.append((ctx.grid_info(), ctx.stats()["dt"], [a.cpu().numpy() for a in ps.x + [ps.V, ps.P]],
                        ps.id.cpu().numpy()))
        ctx.close()
    (g0, dt0, a0, i0), (g1, dt1, a1, i1) = results
    assert g0[:4] == g1[:4] and dt0 == dt1
    assert np.array_equal(i0, i1) and all(np.array_equal(p, q) for p, q in zip(a0, a1))
