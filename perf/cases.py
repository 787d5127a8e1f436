"""Performance cases of the photoacoustic solver: what a user of this package has it compute.

The listed cases are single operators on the sizes of this repository's configurations (the
64, 128 and 256 workloads, the levels and the data grid of the simple-phantom study, the batched
sweep's sides, the warm start's network) plus one small whole reconstruction.  ``draw`` spreads
the same operators over the ranges between and around those sizes.

The inputs come from the seed alone: speed-of-sound maps with elliptic inclusions, vessel-like
initial pressures, sensors on a circle, and (for gradients) noisy traces simulated here with a
plain torch version of the scheme, which in 64 bits is also what ``exact`` returns.
"""
import math

import numpy as np
import torch

from paper_2505_08482_gb300.solver import GridSpec, Plan, Prior, ReconConfig, pml_auto, reconstruct
from paper_2505_08482_gb300.warmstart import UNet, init_params

DX = 1e-4          # cell size of the workloads (m)
C_HI = 1750.0      # upper bound of the speed of sound: c_ref of every plan
C_BG = 1500.0
RHO0 = 1000.0
PML_ALPHA = 2.0
CFL = 0.3


def listed():
    return [
        # traces of one data set on the smallest workload: what a single simulation costs, all latency
        {"name": "forward_64", "kind": "forward", "n": 64, "Ks": "1", "M": 64, "nt": 400, "ckpt": 32, "graphs": False},
        # one objective-and-gradient evaluation of the same problem: the inner step of a small reconstruction
        {"name": "gradient_64", "kind": "gradient", "n": 64, "Ks": "1", "M": 64, "nt": 400, "ckpt": 32, "graphs": False},
        # a coarse multigrid level of the simple-phantom study (58 pixels, 236 sensors, four illuminations)
        {"name": "gradient_58_level", "kind": "gradient", "n": 58, "Ks": "4", "M": 236, "nt": 347, "ckpt": 32,
         "graphs": False},
        # the 128 workload
        {"name": "gradient_128", "kind": "gradient", "n": 128, "Ks": "4", "M": 256, "nt": 900, "ckpt": 32,
         "graphs": False},
        # the headline workload, replayed from a CUDA graph as in an optimiser's loop on its own stream
        {"name": "gradient_256", "kind": "gradient", "n": 256, "Ks": "8", "M": 512, "nt": 1800, "ckpt": 32,
         "graphs": True},
        # several reconstructions of one grid side solved as a batch (serving)
        {"name": "gradient_96_batch", "kind": "gradient", "n": 96, "Ks": "1,2,4,8", "M": 192, "nt": 672, "ckpt": 32,
         "graphs": False},
        # data generated on a finer grid than any reconstruction level (334 pixels, no inverse crime)
        {"name": "forward_334_data", "kind": "forward", "n": 334, "Ks": "4", "M": 236, "nt": 1991, "ckpt": 32,
         "graphs": False},
        # back-projections of a batch of samples at a constant speed of sound (training pairs of the
        # warm start): many data sets, whole pressure history kept
        {"name": "backproject_128", "kind": "backproject", "n": 128, "Ks": "4," * 15 + "4", "M": 256, "nt": 600,
         "ckpt": 600, "graphs": False},
        # the warm start's network: the prediction for a few samples, and a training step's gradients
        {"name": "unet_forward_128", "kind": "unet_forward", "n": 128, "levels": 4, "base": 32, "in_ch": 4, "batch": 8},
        {"name": "unet_grads_128", "kind": "unet_grads", "n": 128, "levels": 4, "base": 32, "in_ch": 4, "batch": 32},
        # the Ornstein-Uhlenbeck prior's value and gradient on the finest simple-phantom level (four p0 and c)
        {"name": "prior_136", "kind": "prior", "n": 136, "nf": 5},
        # a whole reconstruction of the smallest workload, two levels, a few iterations
        {"name": "reconstruct_64", "kind": "reconstruct", "n": 64, "Ks": "1", "M": 64, "nt": 400, "iters": 4},
    ]


# the most cell-steps a drawn sweep may have (the headline workload's)
_MOST = 8 * 300 * 300 * 1800


def draw(rng):
    kind = rng.choice(["forward", "forward", "gradient", "gradient", "gradient", "backproject", "unet_forward",
                       "unet_grads", "prior", "reconstruct"])
    if kind in ("unet_forward", "unet_grads"):
        n = 8 * rng.randint(6, 16)
        return {"kind": kind, "n": n, "levels": rng.choice([3, 4]), "base": rng.choice([16, 32]),
                "in_ch": rng.randint(1, 8), "batch": max(1, round(2 ** rng.uniform(0, 5)))}
    if kind == "prior":
        return {"kind": kind, "n": rng.randint(32, 136), "nf": rng.randint(2, 9)}
    if kind == "reconstruct":
        n = 2 * rng.randint(24, 40)
        return {"kind": kind, "n": n, "Ks": str(rng.randint(1, 3)), "M": rng.randint(32, 128),
                "nt": round(n * rng.uniform(4.0, 7.0)), "iters": rng.randint(3, 5)}
    n = 2 * round(2 ** rng.uniform(4, math.log2(168 if kind == "forward" else 128)))
    nt = round(n * rng.uniform(3.0, 7.5))
    side = n + 50
    top = max(1, min(64 if kind == "backproject" else 24, int(_MOST / (side * side * nt))))
    total = max(1, round(2 ** rng.uniform(0, math.log2(top)))) if top > 1 else 1
    if rng.random() < 0.5 or total == 1:
        Ks = [total]
    else:
        Ks, left = [], total
        while left > 0:
            k = min(left, rng.randint(1, 8))
            Ks.append(k)
            left -= k
    ckpt = nt if kind == "backproject" else rng.choice([16, 32, 32, 50, nt])
    return {"kind": kind, "n": n, "Ks": ",".join(str(k) for k in Ks), "M": rng.randint(48, 2 * n), "nt": nt,
            "ckpt": ckpt, "graphs": kind == "gradient" and rng.random() < 0.3}


# ---- inputs ---------------------------------------------------------------

def _gen(seed):
    return np.random.Generator(np.random.PCG64(int(seed)))


def _dev(a):
    return torch.as_tensor(np.ascontiguousarray(a, dtype=np.float32), device="cuda")


def _sound(n, rng, count=5):
    """Speed of sound: elliptic inclusions of 1400-1650 m/s in water."""
    yy, xx = np.meshgrid(np.arange(n) + 0.5, np.arange(n) + 0.5, indexing="ij")
    c = np.full((n, n), C_BG)
    for _ in range(count):
        cx, cy = rng.uniform(0.25 * n, 0.75 * n, size=2)
        a, b = rng.uniform(0.05 * n, 0.15 * n, size=2)
        t = rng.uniform(0, np.pi)
        u = (xx - cx) * np.cos(t) + (yy - cy) * np.sin(t)
        v = -(xx - cx) * np.sin(t) + (yy - cy) * np.cos(t)
        c[(u / a) ** 2 + (v / b) ** 2 <= 1.0] = rng.uniform(1400.0, 1650.0)
    return _dev(c)


def _pressures(n, K, rng):
    """K initial pressures of a few vessel-like segments each, in [0, 1]; finer grids resolve them better."""
    ax = torch.arange(n, device="cuda", dtype=torch.float32) + 0.5
    out = torch.zeros((K, n, n), device="cuda")
    for k in range(K):
        for _ in range(4):
            cx, cy = rng.uniform(0.3 * n, 0.7 * n, size=2)
            t, length, s = rng.uniform(0, np.pi), rng.uniform(0.1, 0.4) * n, rng.uniform(2.0, 4.0) * max(1.0, n / 128)
            dx, dy = ax[None, :] - cx, ax[:, None] - cy
            along = (dx * math.cos(t) + dy * math.sin(t)).abs() - 0.5 * length
            across = -dx * math.sin(t) + dy * math.cos(t)
            d2 = along.clamp_min(0.0) ** 2 + across ** 2
            out[k] += rng.uniform(0.4, 1.0) * torch.exp(-0.5 * d2 / s ** 2)
    return out.clamp_(0.0, 1.0).contiguous()


def _sensors(n, M, rng):
    t = 2.0 * np.pi * (np.arange(M) + rng.uniform()) / M
    r = 0.4375 * n * DX
    return np.stack([0.5 * n * DX + r * np.cos(t), 0.5 * n * DX + r * np.sin(t)], axis=1)


def _ks(case):
    return [int(k) for k in case["Ks"].split(",")]


def _grid(case):
    n = case["n"]
    return GridSpec(n=n, pml=pml_auto(n), dx=DX, dt=CFL * DX / C_HI, nt=case["nt"], c_ref=C_HI, rho0=RHO0,
                    pml_alpha=PML_ALPHA, c_bg=C_BG)


class _Scheme:
    """The scheme in plain torch: k-space staggered leapfrog with a split-field PML, its discrete
    adjoint, and bilinear point sensors; K data sets, each with its own c."""

    def __init__(self, n, P, nt, xy, dtype):
        N = n + 2 * P
        f64 = dict(dtype=torch.float64, device="cuda")
        self.n, self.P, self.N, self.nt, self.dtype = n, P, N, nt, dtype
        dt = CFL * DX / C_HI
        q = torch.fft.fftfreq(N, 1.0 / N, **f64)
        k = 2.0 * math.pi * q / (N * DX)
        kx, ky = k[:N // 2 + 1], k
        kx = torch.where(torch.arange(N // 2 + 1, device="cuda") == N // 2, -kx.abs(), kx)
        kk = torch.sqrt(kx[None, :] ** 2 + ky[:, None] ** 2)
        kap = torch.sinc(0.5 * C_HI * kk * dt / math.pi)

        def gfac(v):   # i k exp(i k dx/2), real at the Nyquist wavenumber
            im = v * torch.cos(0.5 * v * DX)
            im = torch.where((v.abs() * DX - math.pi).abs() < 1e-9, torch.zeros_like(im), im)
            return torch.complex(-v * torch.sin(0.5 * v * DX), im)

        cdt = torch.complex128 if dtype == torch.float64 else torch.complex64
        self.Gx = (kap * gfac(kx)[None, :]).to(cdt)
        self.Gy = (kap * gfac(ky)[:, None]).to(cdt)
        self.Dx, self.Dy = -self.Gx.conj().resolve_conj(), -self.Gy.conj().resolve_conj()

        def pml(shift):
            s = torch.arange(N, **f64) + shift
            depth = torch.clamp(torch.maximum(P - s, s - (P + n - 1)), min=0.0)
            return torch.exp(-0.5 * dt * PML_ALPHA * (C_HI / DX) * (depth / max(P, 1)) ** 4).to(dtype)

        a, b = pml(0.0), pml(0.5)
        self.ax, self.ay, self.bx, self.by = a[None, :], a[:, None], b[None, :], b[:, None]
        self.sg, self.sd = dt / RHO0, dt * RHO0
        g = xy / DX - 0.5 + P
        i0 = np.floor(g).astype(np.int64)
        f = g - i0
        idx, wts = [], []
        for oy in (0, 1):
            for ox in (0, 1):
                idx.append((i0[:, 1] + oy) * N + i0[:, 0] + ox)
                wts.append((f[:, 1] if oy else 1 - f[:, 1]) * (f[:, 0] if ox else 1 - f[:, 0]))
        self.idx = torch.as_tensor(np.stack(idx), device="cuda")
        self.wts = torch.as_tensor(np.stack(wts), device="cuda").to(dtype)

    def pad(self, v, fill):
        P, n = self.P, self.n
        out = torch.full(v.shape[:-2] + (self.N, self.N), fill, dtype=self.dtype, device="cuda")
        out[..., P:P + n, P:P + n] = v.to(self.dtype)
        return out

    def crop(self, v):
        P, n = self.P, self.n
        return v[..., P:P + n, P:P + n]

    def gather(self, p):
        v = p.flatten(1)[:, self.idx.flatten()].view(p.shape[0], 4, -1)
        return (v * self.wts).sum(1)

    def scatter(self, p, r):
        p.flatten(1).index_add_(1, self.idx.flatten(), (r[:, None, :] * self.wts).flatten(1))

    def inv(self, S):
        return torch.fft.irfft2(S, s=(self.N, self.N))

    def forward(self, c, p0, keep=False):
        """c [K][n][n], p0 [K][n][n] -> traces [K][nt][m] (and the pressures of every step)."""
        c2 = self.pad(c, C_BG) ** 2
        p = self.pad(p0, 0.0)
        K = p.shape[0]
        y = torch.empty((K, self.nt, self.wts.shape[1]), dtype=self.dtype, device="cuda")
        hist = torch.empty((self.nt,) + p.shape, dtype=self.dtype, device="cuda") if keep else None
        rx = ry = p / (2 * c2)
        ux = uy = None
        for t in range(self.nt):
            if t > 0:
                S = torch.fft.rfft2(p)
                gx, gy = self.sg * self.inv(self.Gx * S), self.sg * self.inv(self.Gy * S)
                if ux is None:
                    ux, uy = 0.5 * gx, 0.5 * gy
                ux, uy = self.bx * (self.bx * ux - gx), self.by * (self.by * uy - gy)
                rx = self.ax * (self.ax * rx - self.sd * self.inv(self.Dx * torch.fft.rfft2(ux)))
                ry = self.ay * (self.ay * ry - self.sd * self.inv(self.Dy * torch.fft.rfft2(uy)))
                p = c2 * (rx + ry)
            y[:, t] = self.gather(p)
            if keep:
                hist[t] = p
        return (y, hist) if keep else y

    def adjoint(self, c, p0, hist, r):
        """(dJ/dp0 [K][n][n], dJ/dc [K][n][n]) for the adjoint source r [K][nt][m]."""
        cg = self.pad(c, C_BG)
        c2 = cg ** 2
        zero = torch.zeros_like(cg)
        ubx, uby, rbx, rby, q, cbar = zero, zero, zero, zero, zero, zero.clone()
        for t in range(self.nt - 1, 0, -1):
            pb = q.clone()
            self.scatter(pb, r[:, t])
            cbar += 2 * hist[t] * pb / cg
            tx, ty = self.ax * (rbx + c2 * pb), self.ay * (rby + c2 * pb)
            rbx, rby = self.ax * tx, self.ay * ty
            tx = self.bx * (ubx + self.sd * self.inv(self.Gx * torch.fft.rfft2(tx)))
            ty = self.by * (uby + self.sd * self.inv(self.Gy * torch.fft.rfft2(ty)))
            ubx, uby = self.bx * tx, self.by * ty
            q = self.sg * self.inv(self.Dx * torch.fft.rfft2(tx) + self.Dy * torch.fft.rfft2(ty))
        pb = q.clone()
        self.scatter(pb, r[:, 0])
        if self.nt > 1:
            pb = pb - 0.5 * self.sg * self.inv(self.Dx * torch.fft.rfft2(ubx) + self.Dy * torch.fft.rfft2(uby))
        rs = rbx + rby
        gp = self.crop(pb + rs / (2 * c2))
        return gp, self.crop(cbar) - self.crop(rs / (c2 * cg)) * p0.to(self.dtype)


def _by_set(v, Ks):
    return torch.repeat_interleave(v, torch.as_tensor(Ks, device=v.device), dim=0)


def _sweep_inputs(case, seed):
    """c [ninst][n][n], p0 [K][n][n] and the sensors of a sweep; for gradients also the current
    point, the noisy data and their weights; for back-projections the noisy data."""
    rng = _gen(seed)
    n, Ks = case["n"], _ks(case)
    K = sum(Ks)
    c = torch.stack([_sound(n, rng) for _ in Ks])
    p0 = _pressures(n, K, rng)
    xy = _sensors(n, case["M"], rng)
    d = {"c": c, "p0": p0, "xy": xy, "Ks": Ks, "K": K}
    if case["kind"] in ("gradient", "reconstruct"):
        y = _Scheme(n, pml_auto(n), case["nt"], xy, torch.float32).forward(_by_set(c, Ks), p0)
        gen = torch.Generator(device="cuda")
        gen.manual_seed(int(seed))
        span = y.amax(dim=(1, 2)) - y.amin(dim=(1, 2))
        noise = torch.randn(y.shape, generator=gen, device="cuda")
        d["y"] = (y + 0.01 * span[:, None, None] * noise).contiguous()
        d["w"] = (1.0 / (0.01 * span) ** 2).contiguous()
        d["c"] = (C_BG + 0.5 * (c - C_BG)).contiguous()
        d["p0"] = (0.2 * p0).contiguous()   # an early iterate
    if case["kind"] == "backproject":
        gen = torch.Generator(device="cuda")
        gen.manual_seed(int(seed))
        # traces are smooth in time: noise smoothed over a few samples
        z = torch.randn((K, case["nt"] + 8, case["M"]), generator=gen, device="cuda")
        d["y"] = z.unfold(1, 9, 1).mean(-1).contiguous()
        d["c"] = torch.full_like(c, C_BG)
        d["p0"] = torch.zeros_like(p0)
    return d


def _net_inputs(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    n, B = case["n"], case["batch"]
    x = torch.randn((B, case["in_ch"], n, n), generator=gen, device="cuda")
    x = torch.nn.functional.avg_pool2d(x, 5, 1, 2, count_include_pad=True)   # images, not white noise
    x = (x / x.abs().amax(dim=(1, 2, 3), keepdim=True)).contiguous()
    t = torch.randn((B, 1, n, n), generator=gen, device="cuda")
    t = torch.nn.functional.avg_pool2d(t, 9, 1, 4)[:, 0].contiguous() * 9.0
    return x, t, init_params(case["levels"], case["base"], case["in_ch"], seed)


def _prior_inputs(case, seed):
    rng = _gen(seed)
    n, nf = case["n"], case["nf"]
    x = torch.cat([_pressures(n, nf - 1, rng), _sound(n, rng)[None]]).contiguous()
    eta = [0.5] * (nf - 1) + [C_BG]
    sigma = [0.25] * (nf - 1) + [50.0]
    return x, eta, sigma


PRIOR_TAU = 1.5e-3


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("unet_forward", "unet_grads"):
        x, t, p = _net_inputs(case, seed)
        net = UNet(case["levels"], case["base"], case["in_ch"], case["n"], case["n"], max_batch=case["batch"])
        net.set_params(p)
        return {"kind": kind, "net": net, "x": x, "t": t}
    if kind == "prior":
        x, eta, sigma = _prior_inputs(case, seed)
        return {"kind": kind, "prior": Prior(case["n"], DX, PRIOR_TAU, case["nf"]), "x": x, "eta": eta, "sigma": sigma}
    d = _sweep_inputs(case, seed)
    if kind == "reconstruct":
        n = case["n"]
        cfg = ReconConfig(levels=(n // 2 + (n // 2) % 2, n), L=n * DX, dt_data=CFL * DX / C_HI, nt_data=case["nt"],
                          sensors_xy=d["xy"], K=d["K"], c_hi=C_HI, iters=case["iters"])
        return {"kind": kind, "cfg": cfg, "y": d["y"], "w": d["w"],
                "c": torch.full((n, n), C_BG, dtype=torch.float32, device="cuda")}
    n, Ks, K = case["n"], d["Ks"], d["K"]
    plan = Plan(_grid(case), d["xy"], Ks, ckpt_every=case["ckpt"])
    s = {"kind": kind, "plan": plan, "c": d["c"], "p0": d["p0"], "stream": None}
    if kind == "forward":
        s["out"] = torch.empty((K, case["nt"], case["M"]), device="cuda")
        plan.workspace(0)
    else:
        s["y"] = d["y"]
        plan.workspace(1)
    if kind == "gradient":
        s["w"] = d["w"]
        s["gp"], s["gc"] = torch.empty((K, n, n), device="cuda"), torch.empty((len(Ks), n, n), device="cuda")
        s["J"] = torch.empty(len(Ks), dtype=torch.float64, device="cuda")
        if case["graphs"]:
            s["stream"] = torch.cuda.Stream()
            plan.set_graphs(True)
    return s


def run(s):
    kind = s["kind"]
    if kind == "forward":
        return s["plan"].forward(s["c"], s["p0"], y=s["out"])
    if kind == "gradient":
        if s["stream"] is None:
            J, gp, gc = s["plan"].adjoint_grad(s["c"], s["p0"], s["y"], s["w"], grad_p0=s["gp"], grad_c=s["gc"],
                                               J=s["J"])
            return {"J": J.float(), "grad_p0": gp, "grad_c": gc}   # J is a sum over single-precision traces
        with torch.cuda.stream(s["stream"]):
            J, gp, gc = s["plan"].adjoint_grad(s["c"], s["p0"], s["y"], s["w"], grad_p0=s["gp"], grad_c=s["gc"],
                                               J=s["J"], stream=s["stream"])
            return {"J": J.float(), "grad_p0": gp, "grad_c": gc}
    if kind == "backproject":
        s["plan"].forward(s["c"], s["p0"], keep_checkpoints=True)
        gp, gc = s["plan"].vjp(s["c"], s["p0"], s["y"])
        return {"images": gp}
    if kind == "unet_forward":
        return s["net"].forward(s["x"])
    if kind == "unet_grads":
        loss, g = s["net"].grads(s["x"], s["t"])
        return {"loss": loss, "grads": g}
    if kind == "prior":
        value, grad, z, iterations = s["prior"].eval(s["x"], s["eta"], s["sigma"])
        return {"value": value, "grad": grad, "z": z, "iterations": iterations}
    c, p0, rows, status, ms = reconstruct(s["cfg"], s["y"], s["w"], s["c"])
    return {"c": c, "p0": p0, "status": status}


# ---- what a pass cannot do without ----------------------------------------

def _conv_specs(levels, base, in_ch, n):
    """(cin, cout, k, side) of every convolution of the network, in order."""
    specs, prev = [], in_ch
    for l in range(levels):
        specs += [(prev, base << l, 3, n >> l), (base << l, base << l, 3, n >> l)]
        prev = base << l
    for l in range(levels - 2, -1, -1):
        specs += [(prev + (base << l), base << l, 3, n >> l), (base << l, base << l, 3, n >> l)]
        prev = base << l
    return specs + [(prev, 1, 1, n)]


def work(case):
    kind, n = case["kind"], case["n"]
    if kind in ("unet_forward", "unet_grads"):
        specs = _conv_specs(case["levels"], case["base"], case["in_ch"], n)
        B = case["batch"]
        flops = sum(2.0 * B * h * h * k * k * ci * co for ci, co, k, h in specs)
        params = sum(k * k * ci * co + co for ci, co, k, h in specs)
        if kind == "unet_forward":
            return {"bytes": 4.0 * (B * n * n * (case["in_ch"] + 1) + params), "flops": flops}
        return {"bytes": 4.0 * (B * n * n * (case["in_ch"] + 1) + 2 * params), "flops": 3 * flops}
    if kind == "prior":
        # one product with Xi and one with its preconditioner per field: 2-D real transforms of side 2n
        nf, M = case["nf"], 2 * n
        return {"bytes": 4.0 * 3 * nf * n * n, "flops": 2.0 * nf * 2 * M * M * 5 * math.log2(M)}
    K, M, nt = sum(_ks(case)), case["M"], case["nt"]
    side = n + 2 * pml_auto(n)
    # a step: twelve one-dimensional real transforms of every line (2.5 N log2 N each), 30 operations a cell
    step = K * side * side * (30.0 * math.log2(side) + 30.0)
    fields, traces = 4.0 * n * n * (K + len(_ks(case))), 4.0 * K * nt * M
    if kind == "forward":
        return {"bytes": fields + traces, "flops": step * (nt - 1)}
    if kind == "gradient":
        return {"bytes": 2 * fields + traces, "flops": 2 * step * (nt - 1)}
    if kind == "backproject":
        return {"bytes": 2 * fields + traces, "flops": 2 * step * (nt - 1)}
    # two levels: per iteration one objective and one gradient, and the first gradient
    evals = 2 + 3 * case["iters"]
    return {"bytes": 2 * fields + traces, "flops": evals * step * (nt - 1) * (1 + 1.0 / 8)}


# ---- the same in 64 bits --------------------------------------------------

def _net_exact(case, x, p, target=None):
    """The network (3x3 convolutions with ReLU, max pooling, nearest upsampling, skip connections, final
    1x1) in double precision: prediction, or loss and gradient in the library's parameter layout."""
    p = torch.as_tensor(p, device="cuda").double().requires_grad_(target is not None)
    specs = _conv_specs(case["levels"], case["base"], -(-case["in_ch"] // 8) * 8, case["n"])
    convs, o = [], 0
    for ci, co, k, _ in specs:
        w = p[o:o + co * k * k * ci].view(co, k, k, ci).permute(0, 3, 1, 2)
        o += co * k * k * ci
        convs.append((w, p[o:o + co], k // 2))
        o += co
    conv = lambda v, i: torch.nn.functional.conv2d(v, convs[i][0], convs[i][1], padding=convs[i][2])
    v = torch.nn.functional.pad(x.double(), (0, 0, 0, 0, 0, specs[0][0] - case["in_ch"]))
    i, skips, L = 0, [], case["levels"]
    with torch.set_grad_enabled(target is not None):
        for l in range(L):
            v = torch.relu(conv(torch.relu(conv(v, i)), i + 1))
            i += 2
            if l < L - 1:
                skips.append(v)
                v = torch.nn.functional.max_pool2d(v, 2)
        for l in range(L - 2, -1, -1):
            v = torch.cat([torch.nn.functional.interpolate(v, scale_factor=2, mode="nearest"), skips[l]], dim=1)
            v = torch.relu(conv(torch.relu(conv(v, i)), i + 1))
            i += 2
        out = conv(v, i)[:, 0]
        if target is None:
            return out
        loss = ((out - target.double()) ** 2).mean()
        loss.backward()
    return {"loss": float(loss), "grads": p.grad}


def exact(case, seed):
    kind = case["kind"]
    if kind in ("unet_forward", "unet_grads"):
        x, t, p = _net_inputs(case, seed)
        return _net_exact(case, x, p, t if kind == "unet_grads" else None)
    if kind == "prior":
        x, eta, sigma = _prior_inputs(case, seed)
        n, nf = case["n"], case["nf"]
        ax = (torch.arange(n, device="cuda", dtype=torch.float64) + 0.5) * DX
        gy, gx = torch.meshgrid(ax, ax, indexing="ij")
        pts = torch.stack([gx.flatten(), gy.flatten()], dim=1)
        xi = torch.cdist(pts, pts, compute_mode="donot_use_mm_for_euclid_dist").div_(-PRIOR_TAU).exp_()
        b = torch.stack([x[f].double().flatten() - eta[f] for f in range(nf)], dim=1)
        z = torch.cholesky_solve(b, torch.linalg.cholesky(xi)).T.reshape(nf, n, n)
        s2 = torch.as_tensor(sigma, device="cuda", dtype=torch.float64) ** 2
        value = float((0.5 * (b.T.reshape(nf, n, n) * z).sum(dim=(1, 2)) / s2).sum())
        return {"value": value, "grad": z / s2[:, None, None], "z": z, "iterations": None}
    if kind == "reconstruct":
        return None   # an optimiser's path has no 64-bit value of its own
    d = _sweep_inputs(case, seed)
    Ks = d["Ks"]
    m = _Scheme(case["n"], pml_auto(case["n"]), case["nt"], d["xy"], torch.float64)
    c, p0 = _by_set(d["c"], Ks).double(), d["p0"].double()
    if kind == "forward":
        return m.forward(c, p0)
    y, hist = m.forward(c, p0, keep=True)
    if kind == "backproject":
        return {"images": m.adjoint(c, p0, hist, d["y"].double())[0]}
    r = y - d["y"].double()
    w = d["w"].double()[:, None, None]
    gp, gc = m.adjoint(c, p0, hist, w * r)
    per = (0.5 * w * r * r).sum(dim=(1, 2)).split(Ks)
    return {"J": torch.stack([v.sum() for v in per]), "grad_p0": gp,
            "grad_c": torch.stack([v.sum(0) for v in gc.split(Ks)])}
