"""The split-axis passes (three launches per time step) against the oracle at every compiled grid side.

Each side has its own factorisation, tile remainders (the pairs of rows and columns and the lines of
a launch are rarely multiples of a tile) and copy width (16 bytes where a row is a multiple of 16 bytes).
Tolerances are those of the other parity tests: traces 1e-4, gradients 1e-3 relative L2.
"""
import ctypes

import numpy as np
import pytest

import pat_synth as ps
from tests._problems import grid_params, gpu_plan, oracle_grid, rel_l2

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SIDES = (72, 80, 90, 96, 100, 108, 120, 128, 144, 150, 160, 180, 192, 200, 216, 240, 250, 256, 270, 288, 300, 320,
         324, 360, 384, 400)


def _dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float32, device="cuda")


def _case(ng, K, nt, M=24):
    n, P = ng - 2 * 20, 20
    rng = ps.rng_for(ng)
    c = ps.ellipse_phantom(n, 3, rng)
    # smooth random fields over the whole domain: every sensor has signal from the first sample on
    yy, xx = np.meshgrid(np.arange(n), np.arange(n), indexing="ij")
    p0 = np.stack([sum(rng.uniform(0.2, 1.0) * np.sin(rng.uniform(0.1, 0.6) * xx + rng.uniform(0.1, 0.6) * yy +
                                                      rng.uniform(0, 6.28)) for _ in range(6)) for _ in range(K)])
    xy = ps.rng_for(ng + 1).uniform(0.2 * n, 0.8 * n, size=(M, 2)) * 1e-4
    return grid_params(n, nt, pml=P), c, p0, xy


@pytest.mark.parametrize("ng", SIDES)
def test_forward_and_gradient_match_oracle(ng):
    from oracle.adjoint import adjoint_grad
    from oracle.forward import forward
    from oracle.sensors import sensor_matrix
    K, nt = (3, 26) if ng <= 200 else (1, 15)
    gp, c, p0, xy = _case(ng, K, nt)
    g = oracle_grid(gp)
    S = sensor_matrix(g, xy)
    ref = forward(g, c, p0, S)
    plan = gpu_plan(gp, xy, K, ckpt_every=6)      # ragged segments, re-entered from checkpoints
    assert plan.ng == ng
    assert rel_l2(plan.forward(_dev(c), _dev(p0)).cpu().numpy(), ref) <= 1e-4
    ym = 1.01 * ref + 0.01 * np.abs(ref).max()
    wt = np.linspace(1.0, 2.0, K)
    c0 = np.full_like(c, 1520.0)
    J, gp0, gc = adjoint_grad(g, c0, 0.5 * p0, S, ym, wt)
    Jg, a, b = plan.adjoint_grad(_dev(c0), _dev(0.5 * p0), _dev(ym), _dev(wt))
    assert abs(Jg.item() - J) <= 1e-4 * J
    assert rel_l2(a.cpu().numpy(), gp0) <= 1e-3
    assert rel_l2(b.cpu().numpy(), gc) <= 1e-3


@pytest.mark.parametrize("ng,s", [(80, 1), (108, 5), (250, 4)])
def test_recompute_repeats_the_sweep(ng, s):
    """A last segment recomputed from its checkpoint gives the adjoint of the sweep's own history."""
    gp, c, p0, xy = _case(ng, 2, 4 * s + 1)
    plan = gpu_plan(gp, xy, 2, ckpt_every=s)
    ybar = _dev(ps.rng_for(3).standard_normal((2, gp["nt"], xy.shape[0])))
    cd, pd = _dev(c), _dev(p0)
    plan.forward(cd, pd, keep_checkpoints=True)
    g1 = [t.clone() for t in plan.vjp(cd, pd, ybar)]
    g2 = plan.vjp(cd, pd, ybar)
    assert torch.equal(g1[0], g2[0]) and torch.equal(g1[1], g2[1])


def test_checkpoints_are_shared_with_the_other_forms():
    """Checkpoints are real fields in every form: kept by one form, used by another."""
    gp, c, p0, xy = _case(108, 2, 40)
    plan = gpu_plan(gp, xy, 2, ckpt_every=8)
    ybar = _dev(ps.rng_for(4).standard_normal((2, 40, xy.shape[0])))
    cd, pd = _dev(c), _dev(p0)
    plan.variant = 1
    plan.forward(cd, pd, keep_checkpoints=True)
    ref = [t.cpu().numpy() for t in plan.vjp(cd, pd, ybar)]
    for keep, use in ((0, 0), (0, 1), (1, 0), (-1, 0)):
        plan.variant = keep
        plan.forward(cd, pd, keep_checkpoints=True)
        plan.variant = use
        for a, b in zip(plan.vjp(cd, pd, ybar), ref):
            assert rel_l2(a.cpu().numpy(), b) <= 1e-4, (keep, use)


def test_allocation_free_form_of_a_plan_whose_lines_do_not_fit():
    """The static scratch holds the four-pass step of this plan but not the split-axis lines."""
    from paper_2505_08482_gb300 import _binding as B
    K = 46
    gp, c, p0, xy = _case(108, 1, 12, M=8)
    plan = gpu_plan(gp, xy, K)
    assert plan.workspace_bytes(B.PAT_WS_FORWARD) > B.PAT_NOALLOC_SCRATCH_BYTES
    cd, pd = _dev(c), _dev(np.repeat(p0, K, axis=0) * np.linspace(0.5, 1.5, K)[:, None, None])
    ref = plan.forward(cd, pd)
    y = torch.empty_like(ref)
    stream = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    assert B.lib().pat_forward_noalloc(plan._h, cd.data_ptr(), pd.data_ptr(), y.data_ptr(), stream) == B.PAT_OK
    assert rel_l2(y.cpu().numpy(), ref.cpu().numpy()) <= 1e-5
