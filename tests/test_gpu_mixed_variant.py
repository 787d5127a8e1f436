"""The four-pass form with mixed factorisations and four rows per CTA is a variant of its own, the last one, on the sides
whose variant 0 is the split-axis step.  Its traces and gradients are compared with the oracle's and the other variants' by
the tests that go through all variants of a side; here, that it is that form: four launches per step.
"""
import numpy as np
import pytest

import pat_synth as ps
from tests._problems import grid_params, gpu_plan

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


@pytest.mark.parametrize("ng,count", [(108, 9), (144, 9), (180, 9), (200, 9), (240, 9), (300, 12)])
def test_the_mixed_four_pass_form_is_the_last_variant(ng, count):
    gp, c, p0, xy = _problem(ng, 1, 14)
    plan = gpu_plan(gp, xy, 1, ckpt_every=5)
    assert plan.variants == count and plan.variant == 0
    l0 = _launches()
    plan.forward(_dev(c), _dev(p0))
    l1 = _launches()
    plan.variant = count - 1
    assert plan.variant == count - 1
    plan.forward(_dev(c), _dev(p0))
    assert (_launches() - l1) - (l1 - l0) >= 14 - 4
