"""The generic Stockham passes stay selectable on the sides whose default is the split-axis step."""
import ctypes

import numpy as np
import pytest

import pat_synth as ps
from tests._problems import grid_params, gpu_plan, oracle_grid, rel_l2

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float32, device="cuda")


def _launches():
    from paper_2505_08482_gb300 import _binding as B
    return int(B.lib().pat_kernel_launches())


def _problem(ng, K, nt, M=10):
    n = ng - 40
    rng = ps.rng_for(ng)
    c = ps.ellipse_phantom(n, 2, rng)
    p0 = np.stack([ps.blob_p0(n, 4, rng, sigma_cells=(1.5, 4.0)) for _ in range(K)])
    xy = ps.rng_for(ng + 3).uniform(0.15 * n, 0.85 * n, size=(M, 2)) * 1e-4
    return grid_params(n, nt, pml=20), c, p0, xy


@pytest.mark.parametrize("ng", [72, 90, 100, 250])
def test_generic_passes_of_a_split_side_match_oracle(ng):
    from oracle.adjoint import adjoint_grad
    from oracle.forward import forward
    from oracle.sensors import sensor_matrix
    from paper_2505_08482_gb300 import _binding as B
    K, nt = 2, 25
    gp, c, p0, xy = _problem(ng, K, nt)
    g = oracle_grid(gp)
    S = sensor_matrix(g, xy)
    ref = forward(g, c, p0, S)
    plan = gpu_plan(gp, xy, K, ckpt_every=7)
    assert plan.ng == ng and plan.variants == 0 and plan.variant == -1
    l0 = _launches()
    split = plan.forward(_dev(c), _dev(p0))
    l1 = _launches()
    plan.variant = B.PAT_VARIANT_GENERIC
    assert plan.variant == B.PAT_VARIANT_GENERIC
    y = plan.forward(_dev(c), _dev(p0))
    l2 = _launches()
    # four launches per step instead of three
    assert (l2 - l1) - (l1 - l0) >= nt - 4
    assert rel_l2(y.cpu().numpy(), ref) <= 1e-4
    ym = 1.01 * ref + 0.01 * np.abs(ref).max()
    wt = np.linspace(1.0, 2.0, K)
    J, gp0, gc = adjoint_grad(g, c, 0.5 * p0, S, ym, wt)
    Jg, a, b = plan.adjoint_grad(_dev(c), _dev(0.5 * p0), _dev(ym), _dev(wt))
    assert abs(Jg.item() - J) <= 1e-4 * J
    assert rel_l2(a.cpu().numpy(), gp0) <= 1e-3 and rel_l2(b.cpu().numpy(), gc) <= 1e-3
    plan.variant = -1
    assert plan.variant == -1 and torch.equal(plan.forward(_dev(c), _dev(p0)), split)


@pytest.mark.parametrize("ng", [108, 60])
def test_generic_constant_where_minus_one_is_generic(ng):
    """Sides with variants, and sides without the split-axis step: the same passes under both names."""
    from paper_2505_08482_gb300 import _binding as B
    gp, c, p0, xy = _problem(ng, 1, 12)
    plan = gpu_plan(gp, xy, 1)
    plan.variant = -1
    y = plan.forward(_dev(c), _dev(p0))
    plan.variant = B.PAT_VARIANT_GENERIC
    assert plan.variant == -1 and torch.equal(plan.forward(_dev(c), _dev(p0)), y)


def test_allocation_free_form_falls_back_to_the_generic_passes():
    """A side without variants whose lines do not fit the static scratch, while its four-pass state does."""
    from paper_2505_08482_gb300 import _binding as B
    ng, K = 100, 54
    gp, c, p0, xy = _problem(ng, 1, 12)
    plan = gpu_plan(gp, xy, K)
    assert plan.workspace_bytes(B.PAT_WS_FORWARD) > B.PAT_NOALLOC_SCRATCH_BYTES
    cd, pd = _dev(c), _dev(np.repeat(p0, K, axis=0) * np.linspace(0.5, 1.5, K)[:, None, None])
    ref = plan.forward(cd, pd)
    y = torch.full_like(ref, float("nan"))
    stream = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    assert B.lib().pat_forward_noalloc(plan._h, cd.data_ptr(), pd.data_ptr(), y.data_ptr(), stream) == B.PAT_OK
    assert rel_l2(y.cpu().numpy(), ref.cpu().numpy()) <= 1e-5
