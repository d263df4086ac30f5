"""kernel_launches and the phases' launch counts are the kernels that a call
enqueues, as a stream capture of the call shows them: FP64 passes order their
particles by cost only in 2D and 3D and from 2,048 particles on."""
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


@pytest.mark.parametrize("precision", [lp.PREC_FP64, lp.PREC_FP32])
@pytest.mark.parametrize("d,n", [(1, 1000), (1, 3000), (2, 2047), (2, 2048), (3, 2047), (3, 2048), (3, 9000)])
def test_counts_are_the_enqueued_kernels(d, n, precision):
    from tests.graph_util import captured_kernels
    r = np.random.Generator(np.random.PCG64(n))
    x = r.uniform(0, 1, (d, n))
    st = {"x": list(x), "V": np.full(n, 1.0 / n), "u": list(0.01 * x), "P": 1.0 + 0.1 * x[0], "m": np.ones(n),
          "id": np.arange(n, dtype=np.uint32), "n_fluid": n}
    cfg = dict(radius_mode=lp.RADIUS_KSIDE, k_per_side=4) if d == 1 else dict(kappa=1.6)
    ctx = lp.Context(lp.make_config(d, n, precision=precision, **cfg))
    ps = lp.ParticleSet.from_state(st)
    fields = [1.0 + ps.x[0] * q for q in range(7)]
    calls = {"build": lambda s: ctx.build_neighbors(ps, stream=s),
             "derivs": lambda s: ctx.gfd_derivs(ps, fields[:1], stream=s),
             "derivs-7": lambda s: ctx.gfd_derivs(ps, fields, stream=s),
             "onesided": lambda s: ctx.onesided_derivs(ps, fields[:3], stream=s),
             "step": lambda s: ctx.step(ps, cfl=0.1, stream=s)}
    for sched in (lp.SCHED_FUSED, lp.SCHED_SPLIT):
        ctx.set_schedule(sched)
        ctx.build_neighbors(ps)
        for what, call in calls.items():
            ctx.phase_times()                                  # clears the counts
            before = ctx.stats()["kernel_launches"]
            kernels, _ = captured_kernels(call)
            assert ctx.stats()["kernel_launches"] - before == len(kernels), (what, [k[0] for k in kernels])
            assert sum(v[1] for v in ctx.phase_times().values()) == len(kernels), what
            ctx.build_neighbors(ps)                            # what was captured did not run
    ctx.close()
