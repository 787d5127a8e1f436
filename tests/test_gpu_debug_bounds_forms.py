"""The bounds-checked library on the forms that its other test does not reach: the generic Stockham passes (a side
without any compiled transform, and variant -1 of one with variants), and the split-axis step with several
instances on a side with 8-byte rows.  No check may fail, and the results are those of the release library.
"""
import os
import subprocess
import sys

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def run_forms():
    import pat_synth as ps
    from tests._problems import grid_params, gpu_plan
    f32 = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float32, device="cuda")
    out = {}
    for name, ng, Ks, variant in (("stockham60", 60, [3], None), ("stockham108", 108, [2], -1), ("split90", 90, [1, 2], None)):
        n, K = ng - 40, sum(Ks)
        rng = ps.rng_for(ng)
        xy = rng.uniform(0.15 * n, 0.85 * n, size=(11, 2)) * 1e-4
        c = np.stack([ps.ellipse_phantom(n, 2, rng) for _ in Ks])
        p0 = np.stack([ps.blob_p0(n, 3, rng, sigma_cells=(1.5, 3.0)) for _ in range(K)])
        plan = gpu_plan(grid_params(n, 50, pml=20), xy, Ks, ckpt_every=16)
        if variant is not None:
            plan.variant = variant
        y = plan.forward(f32(c), f32(p0))
        s0 = plan.status(0)
        J, gp, gc = plan.adjoint_grad(f32(c), f32(0.5 * p0), (0.9 * y + 0.01).contiguous(), f32(np.ones(K)))
        out.update({f"{name}_y": y.cpu().numpy(), f"{name}_J": J.cpu().numpy(), f"{name}_gp": gp.cpu().numpy(),
                    f"{name}_gc": gc.cpu().numpy(), f"{name}_status": np.array([s0, plan.status(1)])})
    return out


def test_forms_pass_the_bounds_checks(tmp_path):
    from paper_2505_08482_gb300 import _binding as B
    rel = run_forms()
    out = str(tmp_path / "debug.npz")
    code = ("import sys; sys.path.insert(0, %r); import numpy as np; import paper_2505_08482_gb300 as pkg; "
            "pkg.build(debug=True); from paper_2505_08482_gb300 import _binding as B; assert B.lib().pat_debug_bounds() == 1; "
            "from tests.test_gpu_debug_bounds_forms import run_forms; np.savez(%r, **run_forms())" % (ROOT, out))
    r = subprocess.run([sys.executable, "-c", code], env=dict(os.environ, PAT_DEBUG_BOUNDS="1"), capture_output=True,
                       text=True, timeout=900, cwd=ROOT)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-4000:]
    dbg = dict(np.load(out))
    for key, v in rel.items():
        if key.endswith("_status"):
            assert (dbg[key] & B.PAT_STATUS_BOUNDS).sum() == 0 and (v & B.PAT_STATUS_BOUNDS).sum() == 0, key
        else:   # the checks may change where the compiler fuses a product and a sum
            err = np.linalg.norm(dbg[key].astype(np.float64) - v) / np.linalg.norm(v.astype(np.float64))
            assert np.isfinite(dbg[key]).all() and err <= 1e-6, (key, err)
