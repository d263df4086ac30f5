"""The FP64 redo of listed stencils: a block per particle for short lists, a
thread per particle for long ones.  With tau32 above 1 every FP32 fit is listed,
so an FP32 context has to give the FP64 context's results bit for bit: steps
(plain and learned estimator), central and one-sided derivatives, in 1D, 2D and
3D, with deficient stencils, on both sides of the rule's list length (4096)."""
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


def _planar(n):
    """Particles on a plane (no second-order and no 3D first-order fit), and a line of them."""
    rng = np.random.Generator(np.random.PCG64(3))
    x = [rng.uniform(0, 1, n), rng.uniform(0, 1, n), np.zeros(n)]
    x[1][: n // 4] = 0.5
    one = np.ones(n)
    st = {"x": x, "V": one + 0.1 * x[0], "u": [0.1 * x[1], 0.2 * x[0], 0.0 * one], "P": one + 0.2 * x[1], "m": one / n,
          "id": np.arange(n, dtype=np.uint32), "n_fluid": n}
    return st


CASES = {
    "cloud": lambda n: (inputs.gas_cloud_3d(n, seed=5), dict(dim=3, kappa=2.2, k_max=64, gamma=5.0 / 3.0)),
    "cloud-80": lambda n: (inputs.gas_cloud_3d(n, seed=6, r_max_sigma=0), dict(dim=3, kappa=2.8, k_max=80, k_side=16,
                                                                               gamma=5.0 / 3.0)),
    "planar": lambda n: (_planar(n), dict(dim=3, radius_mode=lp.RADIUS_FIXED, radius=0.06, k_max=40)),
    "kh": lambda n: (inputs.kh_2d(n, 0.03, seed=9), dict(dim=2, kappa=2.0, k_max=40, gamma=1.4, periodic=(1, 1, 0),
                                                         box_hi=(1, 1, 1))),
    "line": lambda n: (inputs.sod_1d(n * 8 // 9, n // 9), dict(dim=1, kappa=4.5, k_max=16, k_side=2)),
}
SIZES = [37, 1500, 4096, 4500]


def _both(name, n, **kw):
    st, cfg = CASES[name](n)
    total = st["V"].shape[0]
    cfg = dict(cfg, n_fluid=st["n_fluid"], s_ref=inputs.field_scales(st), **kw)
    return st, [lp.Context(lp.make_config(capacity=total, **cfg, precision=p, tau32=t))
                for p, t in ((lp.PREC_FP64, 1e-3), (lp.PREC_FP32, 8.0))]


def _equal(a, b, what):
    a, b = a.cpu().numpy(), b.cpu().numpy()
    same = (a == b) | (np.isnan(a) & np.isnan(b)) if a.dtype.kind == "f" else a == b
    assert same.all(), "%s: %d of %d differ" % (what, (~same).sum(), same.size)


@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("name", list(CASES))
@pytest.mark.parametrize("learned", [False, True])
def test_redone_step_equals_the_fp64_step(name, n, learned):
    kw = dict(estimator=lp.EST_MLP, mlp_tau_lo=0.5, mlp_audit=n % 2) if learned else dict(limiter=lp.LIM_PAPER)
    st, ctxs = _both(name, n, **kw)
    res = []
    for ctx in ctxs:
        if learned:
            ctx.mlp_set_params(lp.mlp_init_params(2))
        ps = lp.ParticleSet.from_state(st)
        nf = ps.dim + 2
        d = {"flag": torch.zeros(ps.n, dtype=torch.uint8, device="cuda"),
             "phi": torch.zeros((ps.n, nf), device="cuda"), "r": torch.zeros((ps.n, nf), device="cuda")}
        if learned:
            d.update(features=torch.zeros((ps.n, 8), device="cuda"), gate_p=torch.zeros(ps.n, device="cuda"))
        ctx.step(ps, dt=0.0, cfl=0.2, **d)
        d.update({"x%d" % k: a for k, a in enumerate(ps.x)}, **{"u%d" % k: a for k, a in enumerate(ps.u)}, V=ps.V,
                 P=ps.P, m=ps.m, id=ps.id)
        res.append((d, ctx.stats()))
        ctx.close()
    (d0, s0), (d1, s1) = res
    assert s1["n_fp64_redo"] == min(st["n_fluid"], st["V"].shape[0])
    for k in d0:
        _equal(d0[k], d1[k], k)
    for k in ("n_flagged", "n_linear", "n_nofit", "n_nonfinite", "n_mlp_skip", "n_mlp_miss", "n_mlp_uncertain", "dt"):
        assert s0[k] == s1[k], k


@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("name", list(CASES))
@pytest.mark.parametrize("nf", [1, 3, 5])
def test_redone_derivatives_equal_the_fp64_ones(name, n, nf):
    st, ctxs = _both(name, n, refine=lp.REFINE_AUTO if nf != 3 else lp.REFINE_NEVER)
    out = []
    for ctx in ctxs:
        ps = lp.ParticleSet.from_state(st)
        ctx.build_neighbors(ps)
        fields = ([ps.P, ps.V] + ps.u + [ps.x[0]] * 5)[:nf]
        status = torch.zeros(ps.n, dtype=torch.int32, device="cuda")
        out.append((ctx.gfd_derivs(ps, fields, lp.OUT_F64, status=status), ctx.onesided_derivs(ps, fields), status & 7))
        ctx.close()
    for a, b, what in zip(*out, ("central", "one-sided", "status")):
        _equal(a, b, what)
