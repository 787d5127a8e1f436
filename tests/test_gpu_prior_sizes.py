"""Priors of different sizes in one process: the shared-memory limit of the transforms belongs to the kernels, so creating a
smaller prior must leave a larger one able to launch.
"""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,nf", [(240, 9), (136, 3), (400, 2)])
def test_a_smaller_prior_leaves_a_larger_one_usable(n, nf):
    from paper_2505_08482_gb300.solver import Prior
    gen = torch.Generator(device="cuda").manual_seed(n)
    v = torch.randn((nf, n, n), device="cuda", generator=gen)
    large = Prior(n, 1e-4, 4e-4, nf)
    ref = large.xi(v).clone()
    small = Prior(32, 1e-4, 4e-4, 1)
    assert torch.equal(large.xi(v), ref)
    small.xi(torch.ones((1, 32, 32), device="cuda"))
    assert torch.equal(large.xi(v), ref)
