"""The generic passes carry the gain of their own transforms, isolated from FP32 rounding by a projection over many modes
and time steps.

The factors of the step carry the inverse of the transforms' mean gain (a float transform pair is not exactly unitary,
up to 7e-8), so the gain of another transform is a systematic error of 1e-8 and more: a wrong speed of sound.
The rounding of the factors themselves (up to 6e-8 for one time step size) averages out over several of them.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DX, C = 1e-4, 1500.0


def _dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float32, device="cuda")


def _plan(n, pml, nt, dt, xy, K):
    from paper_2505_08482_gb300.solver import GridSpec, Plan
    gp = dict(n=n, pml=pml, dx=DX, dt=dt, nt=nt, c_ref=C, rho0=1000.0, pml_alpha=0.0 if pml == 0 else 2.0, c_bg=C)
    return Plan(GridSpec(**gp), xy, K, ckpt_every=nt)


def _rounding(v):
    return float(np.float32(v)) / v - 1.0


@pytest.mark.parametrize("ng,variant", [(180, -1), (300, -1), (160, -3), (320, -3)])
def test_frequency_of_plane_waves(ng, variant):
    """Without a PML and with c = c_ref the scheme propagates a plane wave as cos(c k t) exactly.  The mean relative error
    of the measured frequencies, with the known FP32 rounding of the tables taken out, is that of the factors.

    Tolerance 2.7e-8: half of what the gain of another transform (12 x 15 instead of 4 5 3 3, side 180: -0.7e-8 instead of
    2.0e-8 per pair) does to the frequency, which meets two pairs: 2 (2.0 + 0.7) 1e-8.  What is left of the right
    gain's mean over the modes (single modes +-4e-8, 24 modes) and of the factors' rounding (6 step sizes) is 1e-8 each.
    """
    rng = np.random.default_rng(ng)
    K, M, nt = 24, 400, 400
    cells = rng.integers(0, ng - 1, size=(M, 2))
    xy = (cells + 0.5) * DX
    kk = rng.integers(1, ng // 8 + 1, size=(K, 2))
    phase = rng.uniform(0, 2 * np.pi, size=K)
    ax = np.arange(ng)
    arg = 2 * np.pi / ng * (kk[:, 0, None, None] * ax[None, None, :] + kk[:, 1, None, None] * ax[None, :, None]) + \
        phase[:, None, None]
    p0 = np.cos(arg).astype(np.float32)
    at = np.cos(2 * np.pi / ng * (kk[:, 0, None] * cells[None, :, 0] + kk[:, 1, None] * cells[None, :, 1]) +
                phase[:, None])                                          # [K][M]
    kx, ky = 2 * np.pi / (ng * DX) * kk[:, 0], 2 * np.pi / (ng * DX) * kk[:, 1]
    kabs = np.sqrt(kx ** 2 + ky ** 2)
    errs = []
    for cfl in (0.27, 0.283, 0.297, 0.306, 0.311, 0.322):
        dt = cfl * DX / C
        plan = _plan(ng, 0, nt, dt, xy, K)
        assert plan.ng == ng
        plan.variant = variant
        y = plan.forward(_dev(np.full((ng, ng), C)), _dev(p0)).cpu().numpy().astype(np.float64)
        t = np.arange(nt) * dt
        w = C * kabs
        for k in range(K):
            # y = at cos(w (1 + d) t): d by least squares over the second half
            s = slice(nt // 2, None)
            ref = np.cos(w[k] * t[s])[:, None] * at[k][None, :]
            dir_ = (-w[k] * t[s] * np.sin(w[k] * t[s]))[:, None] * at[k][None, :]
            d = np.sum((y[k, s] - ref) * dir_) / np.sum(dir_ * dir_)
            a = 0.5 * C * kabs[k] * dt
            f = [q * np.array([-np.sin(0.5 * q * DX), np.cos(0.5 * q * DX)]) for q in (kx[k], ky[k])]
            ef = [np.dot(v.astype(np.float32).astype(np.float64), v) / np.dot(v, v) - 1.0 for v in f]
            table = _rounding(np.sin(a) / a) + (kx[k] ** 2 * ef[0] + ky[k] ** 2 * ef[1]) / kabs[k] ** 2
            errs.append(d - table)
    mean = float(np.mean(errs))
    print("mean relative frequency error", ng, variant, mean)
    assert abs(mean) <= 2.7e-8
