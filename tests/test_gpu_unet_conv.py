"""The implicit-GEMM convolutions of the U-Net (no im2col) at ragged sizes: image sides that are not multiples of
the 16 x 8 and 16 x 4 pixel tiles, channel counts of every box width (16, 32, 48, 64, 96 channels) and first
layers of one and two channel groups, against the plain-PyTorch reference (the tolerances of the existing parity
test: BF16 against FP32) and against the im2col GEMMs of the warp-level path, from which only the order of the
FP32 sums differs (rare one-step changes of a BF16 value: an order of magnitude below the former).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _rel(a, b):
    a, b = np.asarray(a, dtype=np.float64), np.asarray(b, dtype=np.float64)
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.mark.parametrize("levels,base,in_ch,H,W,B", [
    (3, 16, 3, 20, 36, 8), (4, 16, 9, 40, 104, 8), (2, 48, 16, 18, 26, 8), (1, 32, 1, 8, 8, 1), (3, 64, 4, 52, 28, 8)])
def test_ragged_sizes(levels, base, in_ch, H, W, B):
    from oracle import unet as U
    from paper_2505_08482_gb300.warmstart import UNet
    rng = np.random.default_rng(base + H)
    p = U.init_params(levels, base, in_ch, rng)
    x = torch.as_tensor(rng.standard_normal((B, in_ch, H, W)), dtype=torch.float32, device="cuda")
    t = torch.as_tensor(rng.standard_normal((B, H, W)), dtype=torch.float32, device="cuda")
    net = UNet(levels, base, in_ch, H, W, max_batch=B + 1)
    net.set_params(p)
    out = net.forward(x).cpu().numpy()
    loss, g = net.grads(x, t)
    g = g.cpu().numpy()
    assert net.status() == 0
    net.gemm_path = 0
    out0 = net.forward(x).cpu().numpy()
    loss0, g0 = net.grads(x, t)
    assert _rel(out, out0) <= 3e-3 and abs(loss - loss0) <= 3e-3 * loss0
    assert _rel(g, g0.cpu().numpy()) <= 6e-3
    pb = torch.as_tensor(p, dtype=torch.float32).to(torch.bfloat16).double().numpy()
    xb = x.cpu().to(torch.bfloat16).double().numpy()
    ref = U.forward(pb, xb, levels, base, in_ch, dtype=torch.float64).detach().numpy()
    assert _rel(out, ref) <= 3e-2
    lref, gref = U.loss_and_grad(pb, xb, t.cpu().numpy(), levels, base, in_ch, dtype=torch.float64)
    assert abs(loss - lref) <= 3e-2 * lref
    assert _rel(g, gref) <= 6e-2


def test_gradients_refuse_a_pixel_count_that_is_no_multiple_of_8():
    """As ever on both paths: the im2col GEMMs need it, and a network's answer does not depend on the path."""
    from paper_2505_08482_gb300 import _binding as Bd
    from paper_2505_08482_gb300.warmstart import UNet, init_params
    net = UNet(3, 16, 3, 20, 36, max_batch=3)
    net.set_params(init_params(3, 16, 3))
    x = torch.zeros((3, 3, 20, 36), device="cuda")
    assert net.forward(x).shape == (3, 20, 36)
    for path in (1, 0):
        net.gemm_path = path
        with pytest.raises(Bd.PatError):
            net.grads(x, torch.zeros((3, 20, 36), device="cuda"))


def test_overlapped_launches_repeat():
    """Forward passes and gradients repeat while their launches overlap, eagerly and from a captured graph: the outputs,
    the loss and the bias gradients bit for bit, the weight gradients up to the order of their FP32 sums (1e-5: the
    rounding of sums of a few thousand terms)."""
    from paper_2505_08482_gb300.warmstart import UNet, init_params
    B, in_ch, H, W = 8, 4, 64, 32
    net = UNet(3, 32, in_ch, H, W, max_batch=B)
    net.set_params(init_params(3, 32, in_ch))
    gen = torch.Generator(device="cuda").manual_seed(5)
    x = torch.randn((B, in_ch, H, W), device="cuda", generator=gen)
    t = torch.randn((B, H, W), device="cuda", generator=gen)
    ref = net.forward(x).clone()
    loss, g = net.grads(x, t)
    g = g.clone()
    head = g[-1].item()   # the last convolution's bias
    for _ in range(10):
        assert torch.equal(net.forward(x), ref)
        l1, g1 = net.grads(x, t)
        assert l1 == loss and g1[-1].item() == head and _rel(g1.cpu(), g.cpu()) <= 1e-5
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        out = net.forward(x)
    for _ in range(10):
        out.zero_()
        graph.replay()
        assert torch.equal(out, ref)
    assert net.status() == 0
