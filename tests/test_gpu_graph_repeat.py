"""Graph replays of a gradient repeat it bit for bit.

The reverse sweep overlaps the segment recompute (which writes the pressure history) with the adjoint of the next
segment on another stream.  The first adjoint pass of a segment reads that history, so it must not start before the
recompute has finished: with the programmatic launch attribute a captured graph made the edge from the recompute a
programmatic one as well, and dJ/dc of some replays was built from the previous contents of the buffer.
"""
import numpy as np
import pytest

import pat_synth as ps
from tests._problems import grid_params, gpu_plan

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float32, device="cuda")


@pytest.mark.parametrize("variant", [0, 1, 5])
def test_replayed_gradients_are_bit_identical(variant):
    n, K, nt = 96, 7, 400
    rng = ps.rng_for(50)
    xy = ps.circle_sensors(n, 61, 1e-4)
    plan = gpu_plan(grid_params(n, nt), xy, K, ckpt_every=50)
    plan.variant = variant
    c = _dev(ps.ellipse_phantom(n, 4, rng))
    p0 = _dev(np.stack([ps.vessel_p0(n, rng) for _ in range(K)]))
    ym, w = torch.zeros((K, nt, 61), device="cuda"), torch.ones(K, device="cuda")
    ref = [t.clone() for t in plan.adjoint_grad(c, p0, ym, w)]          # eager: ordered by the event itself
    gp, gc = torch.empty_like(ref[1]), torch.empty_like(ref[2])
    J = torch.empty_like(ref[0])
    stream = torch.cuda.Stream()
    plan.set_graphs(True)
    torch.cuda.synchronize()
    for _ in range(8):
        plan.adjoint_grad(c, p0, ym, w, grad_p0=gp, grad_c=gc, J=J, stream=stream)
        stream.synchronize()
        for a, b in zip((J, gp, gc), ref):
            assert torch.equal(a, b)
