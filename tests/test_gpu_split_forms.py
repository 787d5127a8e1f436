"""The split-axis passes where one launch is not like the next: last segments of several recomputed levels, several
instances on sides with partial tiles and 8-byte rows, and more CTAs than the shared-memory slots place.
"""
import numpy as np
import pytest

import pat_synth as ps
from tests._problems import grid_params, gpu_plan

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float32, device="cuda")


def _problem(ng, K, nt, M=17):
    n = ng - 40
    rng = ps.rng_for(ng)
    c = ps.ellipse_phantom(n, 3, rng)
    p0 = np.stack([ps.blob_p0(n, 5, rng, sigma_cells=(2.0, 8.0)) for _ in range(K)])
    xy = ps.rng_for(ng + 2).uniform(0.2 * n, 0.8 * n, size=(M, 2)) * 1e-4
    return grid_params(n, nt, pml=20), c, p0, xy


@pytest.mark.parametrize("ng,s,nt", [(80, 4, 20), (108, 5, 23), (90, 6, 28), (250, 4, 19), (96, 8, 9), (100, 30, 30)])
def test_recomputed_levels_repeat_the_sweep(ng, s, nt):
    """The second vjp recomputes the last segment, of which the first has the sweep's own history: levels that are a
    re-entry (or the initial condition) and levels stepped from it (one case of a single level)."""
    gp, c, p0, xy = _problem(ng, 2, nt)
    plan = gpu_plan(gp, xy, 2, ckpt_every=s)
    assert plan.ng == ng
    yb = _dev(ps.rng_for(3).standard_normal((2, nt, xy.shape[0])))
    cd, pd = _dev(c), _dev(p0)
    plan.forward(cd, pd, keep_checkpoints=True)
    g1 = plan.vjp(cd, pd, yb)
    g2 = plan.vjp(cd, pd, yb)
    assert torch.equal(g1[0], g2[0]) and torch.equal(g1[1], g2[1])
    assert bool(torch.isfinite(g1[1]).all()) and float(g1[1].abs().max()) > 0


@pytest.mark.parametrize("ng,Ks", [(90, [1, 3, 2]), (150, [2, 1]), (250, [1, 2]), (96, [8, 1, 16, 7, 8])])
def test_instances_equal_single_plans(ng, Ks):
    """The last case has 960 CTAs per pair pass, beyond five per SM."""
    nt = 17
    gp, c, p0, xy = _problem(ng, sum(Ks), nt)
    n = gp["n"]
    cs = np.stack([np.where(c > 1500.0, c + 20.0 * i, c) for i in range(len(Ks))])
    plan = gpu_plan(gp, xy, Ks, ckpt_every=5)
    assert plan.ng == ng
    K = sum(Ks)
    ym = _dev(0.05 * ps.rng_for(9).standard_normal((K, nt, xy.shape[0])))
    w = _dev(np.linspace(0.5, 1.5, K))
    J, gp0, gc = plan.adjoint_grad(_dev(cs), _dev(p0), ym, w)
    y = plan.forward(_dev(cs), _dev(p0))
    o = 0
    for i, k in enumerate(Ks):
        one = gpu_plan(gp, xy, k, ckpt_every=5)
        sl = slice(o, o + k)
        o += k
        ci, pi = _dev(cs[i]), _dev(p0[sl])
        assert torch.equal(one.forward(ci, pi), y[sl])
        J1, a, b = one.adjoint_grad(ci, pi, ym[sl].contiguous(), w[sl].contiguous())
        assert torch.equal(a, gp0[sl]) and torch.equal(b, gc[i])
        assert J1.item() == J[i].item()
    assert n == plan.n
