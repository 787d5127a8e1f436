"""Gradients of the U-Net repeat, eagerly and replayed from a captured graph: the loss and the bias gradients of every
convolution bit for bit (fixed order of their sums), the weight gradients up to the order of their FP32 sums.

The bias sum of a convolution has a last block that adds the parts up and resets a counter, and the weight gradient
runs beside it, reading its inputs before it waits: in a graph their edge is a programmatic one.
"""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("levels,base,B,H,W", [(3, 32, 8, 64, 32), (2, 16, 4, 24, 40), (1, 8, 1, 8, 8)])
def test_captured_gradients_repeat(levels, base, B, H, W):
    from paper_2505_08482_gb300 import _binding as Bd
    from paper_2505_08482_gb300.warmstart import UNet, init_params
    in_ch = 4
    net = UNet(levels, base, in_ch, H, W, max_batch=B)
    net.set_params(init_params(levels, base, in_ch))
    gen = torch.Generator(device="cuda").manual_seed(6)
    x = torch.randn((B, in_ch, H, W), device="cuda", generator=gen)
    t = torch.randn((B, H, W), device="cuda", generator=gen)
    nconv = ctypes.c_int(0)
    L = Bd.lib()
    Bd.check(L.pat_unet_param_layout(net._h, ctypes.byref(nconv), None), "pat_unet_param_layout")
    desc = (ctypes.c_int * (6 * nconv.value))()
    Bd.check(L.pat_unet_param_layout(net._h, ctypes.byref(nconv), desc), "pat_unet_param_layout")
    d = np.array(desc).reshape(-1, 6)                         # cin, cout, k, weight offset, bias offset, H
    biases = [slice(r[4], r[4] + r[1]) for r in d]
    weights = [slice(r[3], r[3] + r[0] * r[1] * r[2] ** 2) for r in d]
    loss, ref = net.grads(x, t)
    assert all(float(ref[b].abs().max()) > 0 for b in biases)

    def same(g, l):
        assert l == loss
        for b in biases:
            assert torch.equal(g[b], ref[b])
        for q in weights:   # sums of up to 1e5 products, reordered: 1e-5 as a norm
            a, r = g[q].double(), ref[q].double()
            assert float((a - r).norm()) <= 1e-5 * float(r.norm())

    for _ in range(10):
        l1, g1 = net.grads(x, t)
        same(g1, l1)
    g = torch.empty_like(ref)
    lo = torch.zeros((), dtype=torch.float64, device="cuda")
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        Bd.check(L.pat_unet_grads(net._h, x.data_ptr(), t.data_ptr(), B, g.data_ptr(), lo.data_ptr(),
                                  ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)), "pat_unet_grads")
    for _ in range(20):
        g.fill_(float("nan"))
        lo.fill_(float("nan"))
        graph.replay()
        torch.cuda.synchronize()
        same(g, lo.item())
    assert net.status() == 0
