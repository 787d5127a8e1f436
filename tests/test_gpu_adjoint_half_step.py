"""The adjoint of the initial half step is its transpose, isolated from FP32 rounding by a projection over many cells.

The factors of the four-pass step carry the inverse of the transforms' mean gain (a float transform pair is not
exactly unitary, up to 7e-8): a half step without it makes the gradient's adjoint not the transpose of the forward step.
The rounding of the factors themselves (up to 6e-8 for one time step size) averages out over several of them.
"""
import numpy as np
import pytest

from tests._problems import oracle_grid

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DX, C = 1e-4, 1500.0


def _dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float32, device="cuda")


def _plan(n, pml, nt, dt, xy, K):
    from paper_2505_08482_gb300.solver import GridSpec, Plan
    gp = dict(n=n, pml=pml, dx=DX, dt=dt, nt=nt, c_ref=C, rho0=1000.0, pml_alpha=0.0 if pml == 0 else 2.0, c_bg=C)
    return Plan(GridSpec(**gp), xy, K, ckpt_every=nt), gp


@pytest.mark.parametrize("variant", [1, 5])
def test_adjoint_initial_half_step(variant):
    """The transpose of the initial half step carries the same factor as the step.  Two time samples, c uniform, source
    at the second one: away from the PML the adjoint of the step is pb, that of the half step t = -pb / 2, and the gradient
    S^T r + pb / 2.  The part of the error along t is the half step's relative error (minus twice the step's, which is
    corrected).

    Tolerance 6e-8: half of what a half step without the correction has at Ng 200 (gain 6.1e-8 per pair, two pairs).
    """
    from oracle.adjoint import adjoint_linear
    from oracle.sensors import sensor_matrix
    n, P, K, m = 160, 20, 6, 64
    rng = np.random.default_rng(11)
    lo = (n - m) // 2
    iy, ix = np.meshgrid(np.arange(lo, lo + m), np.arange(lo, lo + m), indexing="ij")
    xy = np.stack([(ix.ravel() + 0.5) * DX, (iy.ravel() + 0.5) * DX], -1)
    f = np.fft.fftfreq(m)
    smooth = np.exp(-0.5 * (2 * np.pi * 1.5) ** 2 * (f[:, None] ** 2 + f[None, :] ** 2))
    r = np.fft.ifft2(np.fft.fft2(rng.standard_normal((K, m, m))) * smooth).real
    yb = np.zeros((K, 2, m * m))
    yb[:, 1] = (r / np.abs(r).max()).reshape(K, -1).astype(np.float32)
    alphas = []
    for cfl in (0.91, 0.93, 0.95, 0.96, 0.97, 0.98, 0.99, 1.0):
        plan, gp = _plan(n, P, 2, cfl * DX / C, xy, K)
        assert plan.ng == 200
        plan.variant = variant
        c = np.full((n, n), C)
        got, _ = plan.vjp(_dev(c), _dev(np.zeros((K, n, n))), _dev(yb))
        g = oracle_grid(gp)
        S = sensor_matrix(g, xy)
        ref = adjoint_linear(g, c, S, yb)
        src = np.stack([g.crop((S.T @ yb[k, 1]).reshape(1, g.ng, g.ng))[0] for k in range(K)])
        t = -(ref - src)
        err = got.cpu().numpy().astype(np.float64) - ref
        cut = (slice(None), slice(lo + 8, lo + m - 8), slice(lo + 8, lo + m - 8))
        alphas.append(np.sum(err[cut] * t[cut]) / np.sum(t[cut] ** 2))
    mean = float(np.mean(alphas))
    print("mean relative error along the half step", variant, mean, np.std(alphas))
    assert abs(mean) <= 6e-8
