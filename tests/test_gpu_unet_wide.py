"""The final convolution of the U-Net beyond 2048 channels.

A block of its backward pass covers 256 groups of eight channels: 2048 channels fill one block, 2056 and 2064 leave
one and two groups to a second one (2056 takes the im2col form of the convolutions, 2064 the implicit one).
Reference and tolerances as in the network's other parity tests (BF16 against FP64).  The final convolution's own
gradients are compared by themselves: a part that is missing there is small beside the other weights.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _rel(a, b):
    a, b = np.asarray(a, dtype=np.float64), np.asarray(b, dtype=np.float64)
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.mark.parametrize("base", [2048, 2056, 2064])
def test_wide_final_convolution(base):
    from oracle import unet as U
    from paper_2505_08482_gb300.warmstart import UNet
    rng = np.random.default_rng(base)
    p = U.init_params(1, base, 1, rng)
    x = rng.standard_normal((1, 1, 8, 8)).astype(np.float32)
    t = rng.standard_normal((1, 8, 8)).astype(np.float32)
    net = UNet(1, base, 1, 8, 8, max_batch=1)
    net.set_params(p)
    loss, g = net.grads(torch.as_tensor(x, device="cuda"), torch.as_tensor(t, device="cuda"))
    pb = torch.as_tensor(p, dtype=torch.float32).to(torch.bfloat16).double().numpy()
    xb = torch.as_tensor(x).to(torch.bfloat16).double().numpy()
    lref, gref = U.loss_and_grad(pb, xb, t, 1, base, 1, dtype=torch.float64)
    g = g.cpu().numpy()
    assert net.status() == 0
    assert abs(loss - lref) <= 3e-2 * lref
    assert _rel(g, gref) <= 6e-2
    head = slice(-base - 1, None)   # weights and bias of the last convolution
    assert _rel(g[head], gref[head]) <= 6e-2
