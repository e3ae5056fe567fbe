"""The work that this framework is timed on: calls of its public entry points, from the smallest
Monte Carlo run a program makes to the full gradient evaluation, in 2D and 3D, forward and adjoint,
single and batched, with the per-pixel steps around them and the U-Net denoiser.

``listed()`` names the cases, ``draw(rng)`` makes more of the same ranges, ``prepare`` builds the
inputs a program would hold on the GPU (maps, sources, run descriptors, a network), ``run`` makes one
pass, ``work`` states what a pass cannot do without, and ``exact`` gives the outputs in 64 bits where
plain torch can (the Monte Carlo itself has no such value: its packets' paths are the result).
"""
from __future__ import annotations

import math

import numpy as np
import torch
import torch.nn.functional as F

from paper_1608_05238_gb300 import mcr, mcr3
from paper_1608_05238_gb300.autograd import EpsFromH, EpsFromH3, HFromMu, HFromMu3, MCSpec, MCSpec3
from paper_1608_05238_gb300.denoiser import UNet, sample_scale

# Mean path of a packet in tissue-like media (mu_a 0.01, mu_s 10 /mm, g 0.9, some 10 mm across) from an
# edge source and from a volumetric (adjoint) source; a packet crosses about 1.27 pixels (1.5 voxels)
# per pixel side and collides mu_s times per mm.
_PATH_FORWARD, _PATH_ADJOINT = 11.4, 26.0


def listed():
    return [
        # the smallest configuration: a pencil beam into 32 x 32 pixels, 1e5 packets
        dict(name="pencil_32_k8", kind="forward", nz=32, nx=32, extent=8.0, K=8, packets=100_000, source="pencil"),
        # the low-count runs of a denoised reconstruction (1e5 packets per map): launch and latency count
        dict(name="low_forward_256_k16", kind="forward", nz=256, nx=256, extent=12.8, K=16, packets=100_000,
             source="line"),
        dict(name="low_adjoint_256_k16", kind="adjoint", nz=256, nx=256, extent=12.8, K=16, packets=100_000,
             source="volume"),
        # one gradient evaluation of the 4 mm reconstruction domain: two edge sources, K = 10
        dict(name="gradient_80_k10", kind="gradient", nz=80, nx=80, extent=4.0, K=10, packets=1_000_000,
             source="two_lines"),
        # the full gradient evaluation: 256 x 256, K = 32, 1e7 forward + 1e7 adjoint packets
        dict(name="gradient_256_k32", kind="gradient", nz=256, nx=256, extent=12.8, K=32, packets=10_000_000,
             source="line"),
        # a tally far larger than L2: 1024 x 1024, K = 64 (1.2 GB), one edge source
        dict(name="forward_1024_k64", kind="forward", nz=1024, nx=1024, extent=20.48, K=64, packets=1_000_000,
             source="line"),
        # many problems in one launch (wavelengths x sources, mixed grids), as training pairs are made
        dict(name="batch_32_k16", kind="batch", problems=32, extent=12.8, K=16, packets=200_000),
        # one 3D gradient evaluation: 96^3 voxels, L = 4
        dict(name="gradient3_96_l4", kind="gradient3", nz=96, ny=96, nx=96, dx=0.1, L=4, packets=4_000_000),
        # the highest 3D order on a ragged grid, isotropic point source
        dict(name="forward3_ragged_l8", kind="forward3", nz=53, ny=61, nx=75, dx=0.1, L=8, packets=1_000_000),
        # the per-pixel steps between and after the runs: H and eps, the adjoint source, the FP64 gradients
        dict(name="combine_1024_k64", kind="combine", nz=1024, nx=1024, K=64),
        # denoising one map in a reconstruction step, and one training step on a batch of maps
        dict(name="denoise_1x256", kind="denoise", batch=1, h=256, w=256, channels=33),
        dict(name="train_8x256", kind="train", batch=8, h=256, w=256, channels=33),
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["forward", "forward", "adjoint", "gradient", "tally", "batch", "forward3", "gradient3",
                       "combine", "denoise", "train"])
    if kind in ("forward", "adjoint", "gradient", "tally"):
        nz = int(_log_uniform(rng, 16, 1024))
        nx = max(16, min(1024, int(nz * _log_uniform(rng, 0.5, 2.0))))
        extent = _log_uniform(rng, 3.0, 15.0)
        K = rng.choice([0, 1, 4, 8, 10, 16, 16, 24, 32, 32, 48, 64])
        path = _PATH_FORWARD if kind in ("forward", "tally") else _PATH_ADJOINT + _PATH_FORWARD
        segments = path * (10.0 + 1.27 * nz / extent)
        packets = int(min(_log_uniform(rng, 1_000, 5_000_000), 6e8 / segments))
        source = {"adjoint": "volume", "gradient": rng.choice(["line", "two_lines"]),
                  "forward": rng.choice(["line", "pencil", "iso", "angular"]),
                  "tally": rng.choice(["line", "iso"])}[kind]
        c = dict(kind=kind, nz=nz, nx=nx, extent=extent, K=K, packets=packets, source=source)
        if kind == "tally":  # the alternatives to the harmonics: angular sectors, path-length bins
            c.update(K=0, sectors=0, time_bins=0)
            c[rng.choice(["sectors", "time_bins"])] = rng.choice([4, 16, 32, 50])
        return c
    if kind == "batch":
        return dict(kind=kind, problems=rng.randint(2, 48), extent=_log_uniform(rng, 6.0, 12.8),
                    K=rng.choice([4, 8, 16, 32]), packets=int(_log_uniform(rng, 2_000, 100_000)))
    if kind in ("forward3", "gradient3"):
        n = [int(_log_uniform(rng, 12, 96)) for _ in range(3)]
        return dict(kind=kind, nz=n[0], ny=n[1], nx=n[2], dx=_log_uniform(rng, 0.08, 0.2), L=rng.randint(0, 8),
                    packets=int(_log_uniform(rng, 1_000, 500_000)))
    if kind == "combine":
        return dict(kind=kind, nz=int(_log_uniform(rng, 16, 1024)), nx=int(_log_uniform(rng, 16, 1024)),
                    K=rng.choice([4, 8, 16, 31, 32, 64]))
    w = rng.choice([128, 256])
    return dict(kind=kind, batch=rng.randint(1, 8 if w == 256 else 16), h=rng.choice([64, 128, 192, 256]), w=w,
                channels=rng.choice([9, 17, 21, 33]))


# ---------------------------------------------------------------------------------------- inputs
def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) % (1 << 31))
    return g


def _f32(x):
    return float(np.float32(x))


def _phantom(shape, dx, rng, inclusions=3):
    """Background mu_a 0.01 / mu_s 10 with random round inclusions, on the GPU (2D or 3D)."""
    axes = torch.meshgrid(*[(torch.arange(n, device="cuda") + 0.5) * dx for n in shape], indexing="ij")
    mua = torch.full(shape, 0.01, device="cuda")
    mus = torch.full(shape, 10.0, device="cuda")
    for _ in range(inclusions):
        r = rng.uniform(0.05, 0.12) * min(shape) * dx
        inside = sum((a - rng.uniform(0.2, 0.8) * n * dx) ** 2 for a, n in zip(axes, shape)) <= r * r
        mua = torch.where(inside, rng.uniform(0.02, 0.2), mua)
        mus = torch.where(inside, rng.uniform(5.0, 20.0), mus)
    return mua.float().contiguous(), mus.float().contiguous()


def _sources(case, nz, nx, dx, rng):
    lx, lz = nx * dx, nz * dx
    top = mcr.Source(kind=mcr.LINE, x0=0.0, z0=0.0, x1=lx, z1=0.0, dir_x=0.0, dir_z=1.0)
    s = case["source"]
    if s == "line":
        return [top]
    if s == "two_lines":
        return [top, mcr.Source(kind=mcr.LINE, x0=lx, z0=0.0, x1=lx, z1=lz, dir_x=-1.0, dir_z=0.0)]
    x, z = rng.uniform(0.3, 0.7) * lx, rng.uniform(0.3, 0.7) * lz
    if s == "pencil":
        return [mcr.Source(kind=mcr.PENCIL, x0=x, z0=0.0, dir_x=rng.uniform(-0.3, 0.3), dir_z=1.0)]
    if s == "iso":
        return [mcr.Source(kind=mcr.ISO_POINT, x0=x, z0=z)]
    return [mcr.Source(kind=mcr.ANGULAR_POINT, x0=x, z0=z, ang_c=(0.3, 0.2), ang_s=(-0.2, 0.1, 0.1))]


def _signed_source(mua, gen):
    """A q* as a reconstruction meets it: decaying with depth, signed, noisy, in units of mu_a^2."""
    shape = mua.shape
    decay = torch.exp(-torch.linspace(0.0, 4.0, shape[0], device="cuda")).reshape(-1, *([1] * (mua.dim() - 1)))
    noise = torch.randn(shape, generator=gen, device="cuda")
    return (mua * decay * (1.0 + 0.7 * noise) * 1e-2).float().contiguous()


_LEVEL_CHANNELS = (32, 64, 128, 256)


def _unet_layers(channels):
    c0, c1, c2, c3 = _LEVEL_CHANNELS
    return [("e0a", channels, c0, 9), ("e0b", c0, c0, 9), ("e1a", c0, c1, 9), ("e1b", c1, c1, 9),
            ("e2a", c1, c2, 9), ("e2b", c2, c2, 9), ("ma", c2, c3, 9), ("mb", c3, c3, 9),
            ("d2a", c3 + c2, c2, 9), ("d2b", c2, c2, 9), ("d1a", c2 + c1, c1, 9), ("d1b", c1, c1, 9),
            ("d0a", c1 + c0, c0, 9), ("d0b", c0, c0, 9), ("out", c0, channels, 1)]


def _weights(channels, seed):
    """Weights [cout][taps][cin] and biases as a partly trained network has them (small residual head)."""
    g = _generator(seed + 77)
    out = {}
    for name, cin, cout, taps in _unet_layers(channels):
        std = 0.02 if name == "out" else math.sqrt(2.0 / (taps * cin))
        out[name] = (torch.randn(cout, taps, cin, generator=g, device="cuda") * std,
                     torch.randn(cout, generator=g, device="cuda") * 0.02)
    return out


def _maps(case, seed):
    """Low- and high-count harmonic maps [B][2K+1][H][W]: a decaying fluence, orders falling as 0.9^n."""
    B, C, H, W = case["batch"], case["channels"], case["h"], case["w"]
    g = _generator(seed)
    order = (torch.arange(C, device="cuda") + 1) // 2
    depth = torch.exp(-torch.linspace(0.0, 3.0, H, device="cuda")).reshape(1, 1, H, 1)
    amp = (0.9 ** order.float()).reshape(1, C, 1, 1) * depth
    smooth = F.interpolate(torch.randn(B, C, 8, 8, generator=g, device="cuda"), (H, W), mode="bilinear")
    clean = amp * (1.0 + 0.5 * smooth)
    noisy = clean + amp * 0.3 * torch.randn(B, C, H, W, generator=g, device="cuda")
    return (0.07 * noisy).contiguous(), (0.07 * clean).contiguous()


# ---------------------------------------------------------------------------------------- a pass
def prepare(case, seed):
    rng = np.random.default_rng(seed)
    kind = case["kind"]
    mc_seed = int(rng.integers(1 << 30))
    if kind in ("forward", "adjoint", "gradient", "tally"):
        nz, nx = case["nz"], case["nx"]
        dx, g = _f32(case["extent"] / nz), _f32(0.9)
        mua, mus = _phantom((nz, nx), dx, rng)
        if kind == "gradient":  # from the current estimate (a noisy map) against a measured H
            gen = _generator(seed)
            est = (0.01 * (1.0 + 0.1 * torch.randn(nz, nx, generator=gen, device="cuda"))).clamp_min(1e-3)
            spec = MCSpec(dx=dx, g=g, sources=_sources(case, nz, nx, dx, rng), K=case["K"],
                          n_packets=case["packets"], seed=mc_seed)
            depth = torch.exp(-torch.linspace(0.0, 3.0, nz, device="cuda")).reshape(nz, 1)
            return dict(case=case, mua=est.contiguous().requires_grad_(), mus=torch.full_like(mus, 10.0).requires_grad_(),
                        hmeas=(mua * depth * 0.2).contiguous(), spec=spec)
        med = mcr.Medium(mua, mus, dx, g)
        run_ = mcr.Run(K=case["K"], n_packets=case["packets"], seed=mc_seed, stream_id=1 if kind == "adjoint" else 0,
                       sectors=case.get("sectors", 0), time_bins=case.get("time_bins", 0),
                       time_bin_mm=_f32(case["extent"] / 8) if case.get("time_bins", 0) else 0.0)
        if kind == "adjoint":
            return dict(case=case, med=med, q=_signed_source(mua, _generator(seed)), run=run_)
        return dict(case=case, med=med, src=_sources(case, nz, nx, dx, rng)[0], run=run_)
    if kind == "batch":
        problems = []
        for i in range(case["problems"]):
            n = (128, 256, 512)[i % 3]
            dx = _f32(case["extent"] / n)
            mua, mus = _phantom((n, n), dx, rng)
            med = mcr.Medium((mua * (0.5, 1.0, 1.5, 2.0)[i % 4]).contiguous(),
                             (mus * (1.2, 1.0, 0.9, 0.8)[i % 4]).contiguous(), dx, _f32(0.9))
            ext = n * dx
            a, b = sorted(rng.uniform(0.0, ext, 2).tolist())
            lines = [(a, 0.0, b, 0.0, 0.0, 1.0), (a, ext, b, ext, 0.0, -1.0), (0.0, a, 0.0, b, 1.0, 0.0),
                     (ext, a, ext, b, -1.0, 0.0)]
            x0, z0, x1, z1, ux, uz = lines[(i // 4) % 4]
            src = mcr.Source(kind=mcr.LINE, x0=x0, z0=z0, x1=x1, z1=z1, dir_x=ux, dir_z=uz)
            problems.append(mcr.Problem(med, case["packets"], seed=mc_seed, stream_id=2 * i, source=src))
        return dict(case=case, problems=problems, common=mcr.Run(K=case["K"], n_packets=0))
    if kind in ("forward3", "gradient3"):
        shape, dx, g = (case["nz"], case["ny"], case["nx"]), _f32(case["dx"]), _f32(0.9)
        mua, mus = _phantom(shape, dx, rng)
        mid = [(n // 2 + 0.5) * dx for n in shape]
        if kind == "forward3":
            src = mcr3.Source3(mcr.ISO_POINT, x0=_f32(mid[2]), y0=_f32(mid[1]), z0=_f32(mid[0]))
            return dict(case=case, med=mcr3.Medium3(mua, mus, dx, g), src=src,
                        run=mcr.Run(K=case["L"], n_packets=case["packets"], seed=mc_seed))
        gen = _generator(seed)
        est = (0.01 * (1.0 + 0.1 * torch.randn(shape, generator=gen, device="cuda"))).clamp_min(1e-3)
        src = mcr3.Source3(mcr.PENCIL, x0=_f32(mid[2]), y0=_f32(mid[1]), z0=0.0)
        depth = torch.exp(-torch.linspace(0.0, 3.0, shape[0], device="cuda")).reshape(-1, 1, 1)
        return dict(case=case, mua=est.contiguous().requires_grad_(), mus=torch.full_like(mus, 10.0).requires_grad_(),
                    hmeas=(mua * depth * 0.02).contiguous(),
                    spec=MCSpec3(dx=dx, g=g, source=src, L=case["L"], n_packets=case["packets"], seed=mc_seed))
    if kind == "combine":
        return dict(case=case, **_combine_inputs(case, seed))
    net = UNet(in_ch=case["channels"], base=_LEVEL_CHANNELS[0], seed=0)
    net.set_state(_weights(case["channels"], seed))
    x, t = _maps(case, seed)
    return dict(case=case, net=net, x=x, t=t)


def _combine_inputs(case, seed):
    shape, C = (case["nz"], case["nx"]), 2 * case["K"] + 1
    g = _generator(seed)
    order = (torch.arange(C, device="cuda") + 1) // 2
    amp = (0.9 ** order.float()).reshape(C, 1, 1)
    coeff = amp * torch.randn((C,) + shape, generator=g, device="cuda")
    coeff[0] = coeff[0].abs() + 0.1
    adj = 1e-3 * amp * torch.randn((C,) + shape, generator=g, device="cuda")
    mua = 0.01 + 0.1 * torch.rand(shape, generator=g, device="cuda")
    hmeas = mua * (1.0 + 0.2 * torch.randn(shape, generator=g, device="cuda"))
    med = mcr.Medium(mua.contiguous(), torch.full_like(mua, 10.0), _f32(0.02), _f32(0.9))
    return dict(med=med, coeff=coeff.contiguous(), adj=adj.contiguous(), hmeas=hmeas.contiguous())


def run(state):
    s, kind = state, state["case"]["kind"]
    if kind in ("forward", "tally"):
        return mcr.forward(s["med"], s["src"], s["run"])
    if kind == "adjoint":
        return mcr.adjoint(s["med"], s["q"], s["run"])
    if kind == "gradient":
        H = HFromMu.apply(s["mua"], s["mus"], s["spec"])
        eps = EpsFromH.apply(H, s["hmeas"], s["spec"].dx)
        d_mua, d_mus = torch.autograd.grad(eps, (s["mua"], s["mus"]))
        return dict(H=H.detach(), eps=eps.detach(), d_mua=d_mua, d_mus=d_mus)
    if kind == "batch":
        return mcr.run_batch(s["problems"], s["common"])
    if kind == "forward3":
        return mcr3.forward(s["med"], s["src"], s["run"])
    if kind == "gradient3":
        H = HFromMu3.apply(s["mua"], s["mus"], s["spec"])
        eps = EpsFromH3.apply(H, s["hmeas"], s["spec"].dx)
        d_mua, d_mus = torch.autograd.grad(eps, (s["mua"], s["mus"]))
        return dict(H=H.detach(), eps=eps.detach(), d_mua=d_mua, d_mus=d_mus)
    if kind == "combine":
        H, v, eps = mcr.h_eps(s["med"], s["coeff"], s["hmeas"])
        q = mcr.adjoint_source(s["med"], v)
        d_mua, d_mus = mcr.gradient(s["med"], s["coeff"], s["adj"], v)
        return dict(H=H, v=v, eps=eps, q=q, d_mua=d_mua, d_mus=d_mus)
    net = s["net"]
    if kind == "denoise":
        return net.predict(s["x"], sample_scale(s["x"]))
    loss = net.train_step(s["x"], sample_scale(s["x"]), s["t"], 1e-4)
    return dict(loss=loss, weights={k: layer.w for k, layer in net.layers.items()},
                biases={k: layer.b for k, layer in net.layers.items()},
                weight_gradients={k: layer.gw for k, layer in net.layers.items()},
                bias_gradients=[layer.gb for layer in net.layers.values()][:8])


# ---------------------------------------------------------------------------------------- what a pass needs
def work(case):
    """Bytes: each input read once, each output written once.  Operations of a Monte Carlo pass: per
    pixel segment a track weight and one multiply-add per coefficient."""
    kind = case["kind"]
    if kind in ("forward", "adjoint", "gradient", "tally"):
        npix, C = case["nz"] * case["nx"], 2 * case["K"] + 1
        C = case.get("sectors", 0) or case.get("time_bins", 0) or C
        per_mm = 10.0 + 1.27 * case["nz"] / case["extent"]
        path = {"forward": _PATH_FORWARD, "tally": _PATH_FORWARD, "adjoint": _PATH_ADJOINT,
                "gradient": _PATH_ADJOINT + _PATH_FORWARD}[kind]
        sums = 2 if kind == "tally" else 2 * C
        n_src = 2 if case["source"] == "two_lines" else 1
        out = 4 * npix * (3 if kind == "gradient" else C)
        return dict(bytes=8 * npix + out + (4 * npix if kind != "forward" else 0),
                    flops=case["packets"] * n_src * path * per_mm * (20 + sums))
    if kind == "batch":
        npix = sum((128, 256, 512)[i % 3] ** 2 for i in range(case["problems"]))
        per_mm = 10.0 + 1.27 * 256 / case["extent"]
        C = 2 * case["K"] + 1
        return dict(bytes=8 * npix + 4 * npix * C,
                    flops=case["problems"] * case["packets"] * _PATH_FORWARD * per_mm * (20 + 2 * C))
    if kind in ("forward3", "gradient3"):
        nvox, C = case["nz"] * case["ny"] * case["nx"], (case["L"] + 1) ** 2
        segments = case["packets"] * (1 if kind == "forward3" else 2) * 13.0 * (10.0 + 1.5 / case["dx"])
        out = 4 * nvox * (C if kind == "forward3" else 3)
        return dict(bytes=8 * nvox + out, flops=segments * (30 + 2 * C))
    if kind == "combine":
        npix, C = case["nz"] * case["nx"], 2 * case["K"] + 1
        return dict(bytes=npix * (2 * 4 * C + 8 + 12 + 16), flops=npix * (4 * C + 10))
    B, H, W = case["batch"], case["h"], case["w"]
    level = {"e0a": 0, "e0b": 0, "e1a": 1, "e1b": 1, "e2a": 2, "e2b": 2, "ma": 3, "mb": 3, "d2a": 2, "d2b": 2,
             "d1a": 1, "d1b": 1, "d0a": 0, "d0b": 0, "out": 0}
    macs = sum(B * (H >> level[n]) * (W >> level[n]) * ci * co * taps for n, ci, co, taps in _unet_layers(case["channels"]))
    params = sum(ci * co * taps for _, ci, co, taps in _unet_layers(case["channels"]))
    maps = 4 * B * H * W * case["channels"]
    if kind == "denoise":
        return dict(bytes=2 * maps + 2 * params, flops=2 * macs)
    return dict(bytes=2 * maps + 2 * 16 * params, flops=6 * macs)


def _unet64(x0, w):
    def conv(x, name, relu=True):
        k, b = w[name]
        co, taps, ci = k.shape
        side = 3 if taps == 9 else 1
        y = F.conv2d(x, k.reshape(co, side, side, ci).permute(0, 3, 1, 2).contiguous(), b, padding=side // 2)
        return F.relu(y) if relu else y

    up = lambda t: t.repeat_interleave(2, dim=2).repeat_interleave(2, dim=3)
    s0 = conv(conv(x0, "e0a"), "e0b")
    s1 = conv(conv(F.avg_pool2d(s0, 2), "e1a"), "e1b")
    s2 = conv(conv(F.avg_pool2d(s1, 2), "e2a"), "e2b")
    m = conv(conv(F.avg_pool2d(s2, 2), "ma"), "mb")
    d2 = conv(conv(torch.cat([up(m), s2], 1), "d2a"), "d2b")
    d1 = conv(conv(torch.cat([up(d2), s1], 1), "d1a"), "d1b")
    d0 = conv(conv(torch.cat([up(d1), s0], 1), "d0a"), "d0b")
    return x0 + conv(d0, "out", relu=False)


def exact(case, seed):
    kind = case["kind"]
    if kind == "combine":
        s = _combine_inputs(case, seed)
        med, K = s["med"], case["K"]
        area, g = med.dx * med.dx, med.g
        c, a, mua, hm = (t.double() for t in (s["coeff"], s["adj"], med.mua, s["hmeas"]))
        H = mua * c[0]
        v = -area * (hm - H)
        pr = c[1:] * a[1:]
        order = torch.arange(1, K + 1, device="cuda", dtype=torch.float64).repeat_interleave(2).reshape(-1, 1, 1)
        d_mua = v * c[0] + area * (c[0] * a[0] / (2 * math.pi) + pr.sum(0) / math.pi)
        d_mus = area * ((1.0 - g ** order) * pr).sum(0) / math.pi
        return dict(H=H, v=v, eps=0.5 * area * ((hm - H) ** 2).sum(), q=-mua * v / area, d_mua=d_mua, d_mus=d_mus)
    if kind == "denoise":
        x, _ = _maps(case, seed)
        scale = 1.0 / x[:, 0].double().mean((1, 2))
        x0 = x.double() * scale.reshape(-1, 1, 1, 1)
        w = {k: (p.double(), b.double()) for k, (p, b) in _weights(case["channels"], seed).items()}
        return torch.cat([_unet64(x0[i:i + 1], w) for i in range(x0.shape[0])]) / scale.reshape(-1, 1, 1, 1)
    return None
