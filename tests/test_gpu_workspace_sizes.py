"""Workspaces of the four-pass step's size.

The split-axis step asks for a larger state than the four-pass step (pat_workspace_bytes), but a workspace that holds
the four-pass step is accepted on every side: the calls then run that step.  Checkpoints and the pressure
history lie at the same place in a workspace of either size, so calls of different sizes share them.  The traces and
gradients of the two steps agree to the parity tolerances between forms (1e-4).
"""
import ctypes

import numpy as np
import pytest

import pat_synth as ps
from tests._problems import grid_params, gpu_plan, rel_l2

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float32, device="cuda")


def _al(b):
    return (b + 255) // 256 * 256


def _four_pass_bytes(ng, n, K, ninst, nt, m, s):
    """Bytes of the four-pass step: state, spectra, medium, sums; gradient: checkpoints, history, adjoint, traces."""
    field, hc = 4 * K * ng * ng, ng // 2 + 1
    spec = 8 * K * ng * ((hc + 3) // 4 * 4)
    s = min(s, nt)
    nseg = (nt + s - 1) // s
    fwd = _al(4 * field) + _al(4 * ninst * ng * ng) + 2 * _al(spec) + _al(8 * ninst) + _al(8 * K * 32) + _al(16) + \
        _al(4 * (K + 2))
    grad = fwd + _al((nseg - 1) * 4 * field) + _al((2 if nseg > 1 else 1) * s * field) + _al(4 * field) + 2 * _al(spec) + \
        _al(4 * K * n * n) + 2 * _al(4 * K * nt * m)
    return fwd, grad


class _Calls:
    """The C entry points with a workspace of a given size; the bytes behind it stay as they are."""

    def __init__(self, plan, most):
        from paper_2505_08482_gb300 import _binding as B
        self.B, self.L, self.plan = B, B.lib(), plan
        self.buf = torch.full((most + 65536,), 0xA5, dtype=torch.uint8, device="cuda")

    def _stream(self):
        return ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)

    def forward(self, c, p0, nbytes):
        y = torch.full((self.plan.K, self.plan.nt, self.plan.m), float("nan"), device="cuda")
        rc = self.L.pat_forward(self.plan._h, c.data_ptr(), p0.data_ptr(), y.data_ptr(), self.buf.data_ptr(), nbytes,
                                self._stream())
        return rc, y

    def vjp(self, c, p0, yb, nbytes):
        gp, gc = torch.full_like(p0, float("nan")), torch.full_like(c, float("nan"))
        rc = self.L.pat_vjp(self.plan._h, c.data_ptr(), p0.data_ptr(), yb.data_ptr(), gp.data_ptr(), gc.data_ptr(),
                            self.buf.data_ptr(), nbytes, self._stream())
        return rc, gp, gc

    def grad(self, c, p0, ym, w, nbytes):
        gp, gc = torch.full_like(p0, float("nan")), torch.full_like(c, float("nan"))
        J = torch.zeros((), dtype=torch.float64, device="cuda")
        rc = self.L.pat_adjoint_grad(self.plan._h, c.data_ptr(), p0.data_ptr(), ym.data_ptr(), w.data_ptr(), gp.data_ptr(),
                                     gc.data_ptr(), J.data_ptr(), None, self.buf.data_ptr(), nbytes, self._stream())
        return rc, J, gp, gc

    def untouched_from(self, nbytes):
        return bool((self.buf[nbytes:] == 0xA5).all())


def _close(a, b):
    return rel_l2(a.cpu().numpy(), b.cpu().numpy()) <= 1e-4


@pytest.mark.parametrize("ng,s", [(108, 7), (80, 7), (100, 40), (90, 1)])
def test_four_pass_sizes_are_accepted(ng, s):
    from paper_2505_08482_gb300 import _binding as B
    n, K, nt, M = ng - 40, 3, 23, 12
    rng = ps.rng_for(ng)
    c = _dev(ps.ellipse_phantom(n, 3, rng))
    p0 = _dev(np.stack([ps.blob_p0(n, 4, rng, sigma_cells=(2.0, 6.0)) for _ in range(K)]))
    xy = ps.rng_for(ng + 1).uniform(0.2 * n, 0.8 * n, size=(M, 2)) * 1e-4
    plan = gpu_plan(grid_params(n, nt, pml=20), xy, K, ckpt_every=s)
    assert plan.ng == ng
    fwd, grad = _four_pass_bytes(ng, n, K, 1, nt, M, s)
    full_f, full_g = plan.workspace_bytes(B.PAT_WS_FORWARD), plan.workspace_bytes(B.PAT_WS_GRADIENT)
    assert fwd < full_f and grad < full_g
    ref = plan.forward(c, p0)
    yb = torch.randn(ref.shape, device="cuda", generator=torch.Generator(device="cuda").manual_seed(1))
    w, ym = torch.ones(K, device="cuda"), 0.5 * ref
    plan.forward(c, p0, keep_checkpoints=True)
    rv = plan.vjp(c, p0, yb)
    rg = plan.adjoint_grad(c, p0, ym, w)
    k = _Calls(plan, full_g)
    # forward and gradients in a workspace of exactly the four-pass size
    rc, y = k.forward(c, p0, fwd)
    assert rc == B.PAT_OK and _close(y, ref) and k.untouched_from(fwd)
    rc, J, gp, gc = k.grad(c, p0, ym, w, grad)
    assert rc == B.PAT_OK and _close(gp, rg[1]) and _close(gc, rg[2]) and k.untouched_from(grad)
    assert abs(J.item() - rg[0].item()) <= 1e-4 * rg[0].item()
    # kept checkpoints, the two calls with either size
    for kept, used in ((grad, grad), (grad, full_g), (full_g, grad)):
        rc, y = k.forward(c, p0, kept)
        assert rc == B.PAT_OK and _close(y, ref)
        for _ in range(2):   # with the sweep's own last segment, then recomputed
            rc, gp, gc = k.vjp(c, p0, yb, used)
            assert rc == B.PAT_OK and _close(gp, rv[0]) and _close(gc, rv[1]), (kept, used)
    # less than that is refused, a forward workspace is no gradient workspace
    assert k.forward(c, p0, fwd - 1)[0] == B.PAT_ENOMEM
    assert k.grad(c, p0, ym, w, grad - 1)[0] == B.PAT_ENOMEM
    assert k.vjp(c, p0, yb, full_f)[0] == B.PAT_ENOMEM


@pytest.mark.parametrize("ng", [108, 80])
def test_autotune_in_a_four_pass_workspace(ng):
    """The form that does not fit is left out (reported as infinite), the choice is one that fits."""
    from paper_2505_08482_gb300 import _binding as B
    n, K, nt = ng - 40, 2, 40
    xy = ps.circle_sensors(n, 9, 1e-4)
    plan = gpu_plan(grid_params(n, nt, pml=20), xy, K, ckpt_every=8)
    for nbytes in _four_pass_bytes(ng, n, K, 1, nt, 9, 8):
        buf = torch.full((nbytes + 65536,), 0xA5, dtype=torch.uint8, device="cuda")
        ms = (ctypes.c_double * (plan.variants + 1))()
        B.check(B.lib().pat_plan_autotune(plan._h, buf.data_ptr(), nbytes, ms, None), "pat_plan_autotune")
        torch.cuda.synchronize()
        assert bool((buf[nbytes:] == 0xA5).all())
        if plan.variants:
            assert np.isinf(ms[1]) and plan.variant != 0 and ms[plan.variant + 1] == min(ms)
        else:
            assert plan.variant == -1


@pytest.mark.parametrize("ng,s", [(108, 7), (80, 6), (150, 5), (60, 7)])
def test_forward_calls_leave_the_checkpoints_alone(ng, s):
    """A forward-size call in a gradient workspace (either size) between the kept forward pass and vjp."""
    from paper_2505_08482_gb300 import _binding as B
    n, K, nt, M = ng - 40, 2, 24, 9
    rng = ps.rng_for(ng)
    c = _dev(ps.ellipse_phantom(n, 3, rng))
    p0 = _dev(np.stack([ps.blob_p0(n, 4, rng, sigma_cells=(2.0, 5.0)) for _ in range(K)]))
    xy = ps.rng_for(ng + 1).uniform(0.2 * n, 0.8 * n, size=(M, 2)) * 1e-4
    plan = gpu_plan(grid_params(n, nt, pml=20), xy, K, ckpt_every=s)
    assert plan.ng == ng
    fwd, grad = _four_pass_bytes(ng, n, K, 1, nt, M, s)
    full_f, full_g = plan.workspace_bytes(B.PAT_WS_FORWARD), plan.workspace_bytes(B.PAT_WS_GRADIENT)
    yb = torch.randn((K, nt, M), device="cuda", generator=torch.Generator(device="cuda").manual_seed(2))
    k = _Calls(plan, full_g)
    for size in (full_g, grad):
        assert k.forward(c, p0, size)[0] == B.PAT_OK
        assert k.vjp(c, p0, yb, size)[0] == B.PAT_OK
        rc, gp, gc = k.vjp(c, p0, yb, size)          # every segment recomputed
        assert rc == B.PAT_OK and float(gc.abs().max()) > 0
        for between in (fwd, full_f):
            assert k.forward(c, p0, size)[0] == B.PAT_OK
            assert k.forward(c, 2.0 * p0, between)[0] == B.PAT_OK
            rc, a, b = k.vjp(c, p0, yb, size)
            assert rc == B.PAT_OK and torch.equal(a, gp) and torch.equal(b, gc), (size, between)
