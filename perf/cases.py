"""What this framework's users have it do, as measurable cases.

A case is one of five kinds of call through the public Python binding
(paper_1304_2062_gb300.se2n):

inpaint   se2n_inpaint on images in device memory: the whole method.
host      se2n_inpaint_host: the same from pinned host buffers.
diffuse   se2n_diffuse on a transformed volume: the stage that a program
          with transforms of its own calls.
batch     se2n_batch_run: many uneven images through one handle.
unet      se2n_unet_forward or se2n_unet_backward: the learned surrogate.

`flag` is the diffusion the caller asks for: "prop" (S-step propagators),
"steps" (the default) or "fp64" (FP64 corner correction). `fresh` drops the
propagators before every pass, as a program does whose diffusion parameters
change from call to call; otherwise the plan keeps what it keeps. `bins`
"own" leaves the orientation to the library, "given" passes a bin map.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1304_2062_gb300 import se2n

BIN_FLAT = 255
BATCH_SIDES = (128, 256, 384, 512, 768, 1024)
FUSED_SIDES = (64, 128, 256, 384, 512, 768, 1024)
EPS, GUARD = 0.5, 0.1


def _inpaint(name, H, W, N, beta, T, steps, rounds, flag="prop", fresh=False, bins="given", proj=0, final_mix=0,
             reinject=0, kind="inpaint"):
    """T is the time of one restoration interval."""
    return dict(name=name, kind=kind, H=H, W=W, N=N, beta=beta, T=T, steps=steps, rounds=rounds, flag=flag,
                fresh=fresh, bins=bins, proj=proj, final_mix=final_mix, reinject=reinject)


def listed():
    return [
        # the smallest workload: one interval of a 64x64 thumbnail, where launches count
        _inpaint("small_64_N16", 64, 64, 16, 0.5, 1.0, 100, 1, bins="own"),
        # the default parameters on a 256x256 image, known pixels put back: how the surrogate's targets are made
        _inpaint("default_256_N32", 256, 256, 32, 0.5, 1.0, 100, 1, flag="steps", bins="own", reinject=1),
        # the headline workload, image after image through one plan
        _inpaint("headline_512_N32", 512, 512, 32, 0.25, 2.0, 500, 10, bins="own"),
        # the paper's angle count, with the propagators built in every call
        _inpaint("paper_512_N30_fresh", 512, 512, 30, 0.25, 2.0, 500, 10, fresh=True),
        # a photograph's size: sides that are no power of two
        _inpaint("photo_480x640_N32", 480, 640, 32, 0.25, 2.0, 100, 4),
        # a ragged size and an angle count without propagators, mean projection, one more restoration
        _inpaint("ragged_250x334_N24", 250, 334, 24, 0.3, 1.5, 60, 3, flag="steps", proj=1, final_mix=1),
        # the largest workload: a 2 GiB volume, 1000 steps, propagators built in every call
        _inpaint("large_2048_N64_fresh", 2048, 2048, 64, 0.25, 50.0, 1000, 1, fresh=True),
        # an application that holds its images in host memory
        _inpaint("host_768x1024_N16", 768, 1024, 16, 0.25, 2.0, 100, 2, bins="own", kind="host"),
        # the stage alone, in the stiff regime of the stress workload (beta dt = 10)
        dict(name="diffuse_stiff_512_N64", kind="diffuse", H=512, W=512, N=64, beta=10.0, T=100.0, steps=100,
             flag="steps"),
        # two dozen uneven images (sides and N of the batch workload) in one call
        dict(name="batch_24_uneven", kind="batch", count=24, pick=3, beta=0.25, T=2.0, steps=100, rounds=1),
        # the surrogate's inference batch and its training batch (loss and gradients)
        dict(name="unet_forward_64x256", kind="unet", count=64, H=256, W=256, backward=False),
        dict(name="unet_backward_32x256", kind="unet", count=32, H=256, W=256, backward=True),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _side(rng, lo=32, hi=1024):
    return 2 * max(1, round(_log(rng, lo, hi) / 2))


def draw(rng):
    kind = rng.choices(("inpaint", "host", "diffuse", "batch", "unet"), (10, 2, 3, 2, 2))[0]
    beta, T = round(_log(rng, 0.1, 0.5), 4), round(_log(rng, 0.5, 8.0), 3)
    steps = round(_log(rng, 12, 500) * max(1.0, T / 4))
    if kind in ("inpaint", "host"):
        N = rng.choice((16, 30, 32, 32, 64, 8, 24, 48))
        if rng.random() < 0.4:
            H, W = rng.choice(FUSED_SIDES), rng.choice(FUSED_SIDES)
        else:
            H, W = _side(rng), _side(rng)
        flag = "prop" if N in (16, 30, 32, 64) and rng.random() < 0.65 else "steps"
        return dict(kind=kind, H=H, W=W, N=N, beta=beta, T=T, steps=steps, rounds=rng.randint(1, 5), flag=flag,
                    fresh=flag == "prop" and rng.random() < 0.4, bins="own" if kind == "host" else "given",
                    proj=int(rng.random() < 0.2), final_mix=int(rng.random() < 0.2),
                    reinject=int(rng.random() < 0.3))
    if kind == "diffuse":
        N = rng.choice((4, 8, 12, 16, 24, 30, 32, 48, 64))
        flag = rng.choice(("steps", "steps", "fp64") + (("prop",) if N in (16, 30, 32, 64) else ()))
        if rng.random() < 0.25:   # stiff
            beta = round(_log(rng, 1.0, 10.0), 3)
            T, steps = float(round(_log(rng, 8, 80))), rng.randint(10, 80)
        return dict(kind=kind, H=_side(rng, 16, 640), W=_side(rng, 16, 640), N=N, beta=beta, T=T, steps=steps,
                    flag=flag)
    if kind == "batch":
        return dict(kind=kind, count=rng.randint(3, 20), pick=rng.randint(10, 10 ** 6), beta=beta, T=T, steps=steps,
                    rounds=rng.randint(1, 3))
    return dict(kind=kind, count=rng.randint(1, 32), H=8 * rng.randint(4, 32), W=8 * rng.randint(4, 32),
                backward=rng.random() < 0.5)


# ----------------------------------------------------------------------------
# inputs
# ----------------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) & 0x7FFFFFFF)
    return g


def _image(H, W, g, strokes=24):
    """Grey image in [0.05, 1]: smooth noise under random line strokes, float32 [H][W]."""
    u = torch.rand((1, 1, max(2, H // 16), max(2, W // 16)), generator=g, device="cuda")
    img = 0.05 + 0.15 * torch.nn.functional.interpolate(u, (H, W), mode="bicubic", align_corners=True)[0, 0].clamp(0, 1)
    y = torch.arange(H, device="cuda", dtype=torch.float32)[:, None]
    x = torch.arange(W, device="cuda", dtype=torch.float32)[None, :]
    for p in torch.rand((strokes, 6), generator=g, device="cuda").tolist():
        x0, y0, dx, dy = p[0] * W, p[1] * H, (p[2] - 0.5) * W, (p[3] - 0.5) * H
        t = (((x - x0) * dx + (y - y0) * dy) / max(dx * dx + dy * dy, 1e-6)).clamp(0, 1)
        d = torch.hypot(x - (x0 + t * dx), y - (y0 + t * dy))
        img = torch.maximum(img, (0.3 + 0.7 * p[5]) * (0.5 + 1.5 * p[4] + 0.5 - d).clamp(0, 1))
    return img.clamp(0.05, 1.0).contiguous()


def _mask(H, W, g, corrupted):
    """1 = known: random corruption and 4-pixel bars every 32 pixels (uint8)."""
    m = torch.rand((H, W), generator=g, device="cuda") >= corrupted
    bars = torch.arange(max(H, W), device="cuda") % 32 < 4
    return (m & ~bars[:H, None] & ~bars[None, :W]).to(torch.uint8).contiguous()


def _bins(f, mask, N, sigma=1.0, flat_tol=1e-4):
    """Direction bin of every pixel in 64 bits: tangent of the Gaussian-smoothed image."""
    H, W = f.shape
    F = torch.fft.fft2(f.double() * (mask != 0))
    k = torch.fft.fftfreq(H, device=f.device, dtype=torch.float64)[:, None]
    l = torch.fft.fftfreq(W, device=f.device, dtype=torch.float64)[None, :]
    F = F * torch.exp(-2.0 * math.pi ** 2 * sigma ** 2 * (k ** 2 + l ** 2))
    gx = torch.fft.ifft2(F * torch.where(l == -0.5, 0.0, l) * (2j * math.pi)).real
    gy = torch.fft.ifft2(F * torch.where(k == -0.5, 0.0, k) * (2j * math.pi)).real
    mag = torch.hypot(gx, gy)
    phi = torch.remainder(torch.atan2(gy, gx) + 0.5 * math.pi, math.pi)
    b = torch.remainder(torch.floor(phi * (N / math.pi) + 0.5), N)
    return torch.where(mag <= flat_tol * mag.max(), torch.full_like(b, BIN_FLAT), b).to(torch.uint8).contiguous()


def _flags(flag):
    return {"prop": se2n.SE2N_DIFFUSE_PROPAGATOR, "steps": 0, "fp64": se2n.SE2N_DIFFUSE_SM_FP64}[flag]


def _batch_shapes(case):
    """Sides and N of the batch's images, and each one's corrupted share."""
    r = np.random.default_rng(case["pick"])
    out = []
    for _ in range(case["count"]):
        side = int(r.choice(BATCH_SIDES))
        N = int(r.choice((16, 32, 64)))
        out.append((side, N, float(r.uniform(0.6, 0.9))))
    return out


def _volume(case, seed):
    """Spectrum with the decay of a lifted image's, complex64 [N][H][W]."""
    N, H, W = case["N"], case["H"], case["W"]
    v = torch.randn((N, H, W), generator=_gen(seed), device="cuda", dtype=torch.complex64)
    k = torch.fft.fftfreq(H, device="cuda")[:, None]
    l = torch.fft.fftfreq(W, device="cuda")[None, :]
    return (v / (0.02 + torch.hypot(k, l))).contiguous()


# 3x3 layers (input channels, output channels) of the surrogate, in the flat parameter vector's order
_LAYERS = ((8, 32), (32, 32), (32, 64), (64, 64), (64, 128), (128, 128), (128, 256), (256, 256), (384, 128),
           (128, 128), (192, 64), (64, 64), (96, 32), (32, 32))


def _unet_params(seed):
    """He-normal weights, small biases and head, float32 flat vector in host memory."""
    g = torch.Generator()
    g.manual_seed(int(seed) & 0x7FFFFFFF)
    parts = []
    for cin, cout in _LAYERS:
        fan = 9 * (2 if cin == 8 else cin)
        parts.append(torch.randn(cout * 9 * cin, generator=g) * math.sqrt(2.0 / fan))
        parts.append(torch.randn(cout, generator=g) * 0.05)
    parts.append(torch.randn(32, generator=g) * 0.05)
    parts.append(torch.full((1,), 0.01))
    return torch.cat(parts)


def _unet_inputs(case, seed):
    g = _gen(seed)
    n, H, W = case["count"], case["H"], case["W"]
    u = torch.rand((n, 1, max(2, H // 8), max(2, W // 8)), generator=g, device="cuda")
    clean = 0.05 + 0.95 * torch.nn.functional.interpolate(u, (H, W), mode="bilinear", align_corners=True)[:, 0]
    mask = (torch.rand((n, H, W), generator=g, device="cuda") >= 0.5).to(torch.uint8)
    return (clean * mask).contiguous(), mask, clean.contiguous()


# ----------------------------------------------------------------------------
# the cases
# ----------------------------------------------------------------------------

def _image_inputs(case, seed):
    g = _gen(seed)
    mask = _mask(case["H"], case["W"], g, 0.75)
    return (_image(case["H"], case["W"], g) * mask).contiguous(), mask


def _batch_inputs(case, seed):
    out = []
    for i, (side, N, share) in enumerate(_batch_shapes(case)):
        g = _gen(seed * 131 + i)
        mask = _mask(side, side, g, share)
        f = (_image(side, side, g, strokes=8) * mask).contiguous()
        out.append((f, mask, N, _bins(f, mask, N)))
    return out


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("inpaint", "host"):
        H, W, N = case["H"], case["W"], case["N"]
        f, mask = _image_inputs(case, seed)
        s = dict(case=case, plan=se2n.se2n_plan_create(H, W, N), prm=se2n.se2n_params_default(
            N=N, beta=case["beta"], T=case["T"] * case["rounds"], steps=case["steps"], rounds=case["rounds"],
            eps=EPS, guard=GUARD, proj=case["proj"], final_mix=case["final_mix"], reinject=case["reinject"],
            diffuse_flags=_flags(case["flag"])))
        if kind == "host":
            s.update(f=f.cpu().pin_memory(), mask=mask.cpu().pin_memory(), out=torch.empty((H, W)).pin_memory())
        else:
            s.update(f=f, mask=mask, out=torch.empty((H, W), device="cuda"),
                     vol=torch.empty((N, H, W), dtype=torch.complex64, device="cuda"),
                     bins=_bins(f, mask, N) if case["bins"] == "given" else None)
        return s
    if kind == "diffuse":
        return dict(case=case, plan=se2n.se2n_plan_create(case["H"], case["W"], case["N"]), src=_volume(case, seed),
                    vol=torch.empty((case["N"], case["H"], case["W"]), dtype=torch.complex64, device="cuda"))
    if kind == "batch":
        imgs = [(f, m, torch.empty_like(f), N, b) for f, m, N, b in _batch_inputs(case, seed)]
        prm = se2n.se2n_params_default(beta=case["beta"], T=case["T"] * case["rounds"], steps=case["steps"],
                                       rounds=case["rounds"], diffuse_flags=se2n.SE2N_DIFFUSE_PROPAGATOR)
        return dict(case=case, imgs=imgs, batch=se2n.se2n_batch_create(imgs, prm))
    f, mask, target = _unet_inputs(case, seed)
    u = se2n.se2n_unet_create(case["count"], case["H"], case["W"])
    params = _unet_params(seed)
    se2n.se2n_unet_set_params(u, params)
    return dict(case=case, unet=u, f=f, mask=mask, target=target, out=torch.empty_like(f),
                loss=torch.zeros(1, device="cuda"), grads=torch.empty(params.numel()).pin_memory())


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind in ("inpaint", "host"):
        if case["fresh"]:
            se2n.se2n_plan_drop_propagators(state["plan"])
        if kind == "host":
            se2n.se2n_inpaint_host(state["plan"], state["f"], state["mask"], state["prm"], state["out"])
        else:
            se2n.se2n_inpaint(state["plan"], state["f"], state["mask"], state["bins"], state["prm"], state["vol"],
                              state["out"])
        return state["out"]
    if kind == "diffuse":
        state["vol"].copy_(state["src"])   # the call works in place
        se2n.se2n_diffuse(state["plan"], state["vol"], case["beta"], case["T"], case["steps"], _flags(case["flag"]))
        return state["vol"]
    if kind == "batch":
        se2n.se2n_batch_run(state["batch"])
        return [img[2] for img in state["imgs"]]
    if case["backward"]:
        se2n.se2n_unet_backward(state["unet"], state["f"], state["mask"], state["target"], case["count"],
                                state["loss"])
        se2n.se2n_unet_get_grads(state["unet"], state["grads"])
        return dict(loss=state["loss"], grads=state["grads"])
    se2n.se2n_unet_forward(state["unet"], state["f"], state["mask"], case["count"], state["out"])
    return state["out"]


def _method_work(H, W, N, rounds):
    """One inpaint: the image, mask and result once; transforms at 5 n log2 n a plane and interval, and, for the
    diffusion, one N x N real map on complex vectors a frequency of the half spectrum."""
    half = H * (W // 2 + 1)
    fl = rounds * (2 * N * 2.5 * H * W * math.log2(H * W) + 4.0 * half * N * N)
    return 9 * H * W, fl


def work(case):
    kind = case["kind"]
    if kind in ("inpaint", "host"):
        b, fl = _method_work(case["H"], case["W"], case["N"], case["rounds"])
        return {"bytes": b, "flops": fl}
    if kind == "diffuse":
        n = case["N"] * case["H"] * case["W"]
        return {"bytes": 2 * 8 * n, "flops": 4.0 * n * case["N"]}
    if kind == "batch":
        parts = [_method_work(s, s, N, case["rounds"]) for s, N, _ in _batch_shapes(case)]
        return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}
    px, scale = case["count"] * case["H"] * case["W"], (1, 1, 4, 4, 16, 16, 64, 64, 16, 16, 4, 4, 1, 1)
    fl = sum(2.0 * 9 * (2 if cin == 8 else cin) * cout / s for (cin, cout), s in zip(_LAYERS, scale)) + 64.0
    weights = 4 * sum(9 * cin * cout + cout for cin, cout in _LAYERS)
    return {"bytes": (13 if case["backward"] else 9) * px + weights * (2 if case["backward"] else 1),
            "flops": px * fl * (3 if case["backward"] else 1)}


# ----------------------------------------------------------------------------
# the same in 64 bits
# ----------------------------------------------------------------------------

def _evolve(v, wy, wx, beta, T, steps):
    """S Crank-Nicolson steps of every frequency of v [N][rows][cols] (complex128, in place): the N x N step matrix
    raised to the power S. Frequencies whose sines are equal share one."""
    N = v.shape[0]
    th = math.pi * torch.arange(N, device=v.device, dtype=torch.float64) / N
    dt = T / steps
    eye = torch.eye(N, device=v.device, dtype=torch.float64)
    lap = torch.roll(eye, 1, 0) + torch.roll(eye, -1, 0) - 2.0 * eye
    uy, iy = torch.unique((wy * 2 ** 40).round(), return_inverse=True)
    ux, ix = torch.unique((wx * 2 ** 40).round(), return_inverse=True)
    uy, ux = uy / 2 ** 40, ux / 2 ** 40
    per = max(1, int(1.2e8 / (N * N * ux.numel())))
    order = torch.argsort(iy)
    starts = torch.searchsorted(iy[order].contiguous(), torch.arange(0, uy.numel() + per, per, device=v.device))
    for c, y0 in enumerate(range(0, uy.numel(), per)):
        y = uy[y0:y0 + per]
        a2 = (ux[None, :, None] * torch.cos(th) + y[:, None, None] * torch.sin(th)) ** 2
        A = torch.diag_embed(-a2).add_(beta * lap).reshape(-1, N, N)
        M = torch.linalg.solve(eye - 0.5 * dt * A, eye + 0.5 * dt * A)
        D, s = None, steps
        while s:
            if s & 1:
                D = M.clone() if D is None else D @ M
            s >>= 1
            if s:
                M = M @ M
        rows = order[starts[c]:starts[c + 1]]
        x = v[:, rows].permute(1, 2, 0)
        D = D.reshape(y.numel(), ux.numel(), N, N)
        out = torch.empty_like(x)
        for j in range(rows.numel()):
            Dj = D[iy[rows[j]] - y0][ix]
            out[j] = torch.complex((Dj @ x[j].real[..., None])[..., 0], (Dj @ x[j].imag[..., None])[..., 0])
        v[:, rows] = out.permute(2, 0, 1)
    return v


def _sines(n, m, device):
    return torch.sin(2.0 * math.pi * torch.arange(m, device=device, dtype=torch.float64) / n)


def _exact_method(f, mask, N, p, bins=None):
    """The image in 64 bits."""
    H, W = f.shape
    f = f.double()
    bins = _bins(f, mask, N) if bins is None else bins
    good = mask != 0
    f0 = f * good
    r = torch.arange(N, device=f.device)[:, None, None]
    on = (bins[None] == r) | (bins[None] == BIN_FLAT)
    v = torch.where(on, f0[None], torch.zeros((), dtype=torch.float64, device=f.device))
    h0 = torch.where(bins == BIN_FLAT, f0, f0.clamp(min=0.0))
    wy, wx = _sines(H, H, f.device), _sines(W, W // 2 + 1, f.device)
    for i in range(p["rounds"]):
        spec = torch.fft.rfft2(v)
        v = None
        v = torch.fft.irfft2(_evolve(spec, wy, wx, p["beta"], p["T"], p["steps"]), s=(H, W))
        if i + 1 < p["rounds"] or p.get("final_mix"):
            ht = v.max(dim=0).values
            scaled = good & (ht > GUARD * h0) & (ht > 0.0)
            sig = torch.where(scaled, (EPS * h0 + (1.0 - EPS) * ht) / torch.where(scaled, ht, 1.0), 1.0)
            lin = good & ~scaled
            v = torch.where(lin[None], EPS * torch.where(on, f0[None], 0.0) + (1.0 - EPS) * v, v * sig[None])
    out = v.mean(dim=0) if p.get("proj") else v.max(dim=0).values
    return torch.where(good, f, out) if p.get("reinject") else out


def _unet_exact(case, seed):
    """The network in 64 bits by torch's convolutions."""
    f, mask, target = _unet_inputs(case, seed)
    flat = _unet_params(seed).cuda().double().requires_grad_(case["backward"])
    Ws, o = [], 0
    for cin, cout in _LAYERS:
        n = cout * 9 * cin
        w = flat[o:o + n].reshape(cout, 3, 3, cin).permute(0, 3, 1, 2)
        Ws.append((w, flat[o + n:o + n + cout]))
        o += n + cout
    head, hb = flat[o:o + 32], flat[o + 32]
    outs, loss = [], 0.0
    step = 8
    for i in range(0, case["count"], step):
        m = (mask[i:i + step] != 0).double()
        x0 = f[i:i + step].double() * m
        x = torch.stack([x0, m] + [torch.zeros_like(m)] * 6, dim=1)

        def conv(x, k):
            return torch.relu(torch.nn.functional.conv2d(x, Ws[k][0], Ws[k][1], padding=1))

        skips = []
        for level in range(4):
            x = conv(conv(x if level == 0 else torch.nn.functional.avg_pool2d(x, 2), 2 * level), 2 * level + 1)
            skips.append(x)
        for k in range(3):
            up = torch.nn.functional.interpolate(x, scale_factor=2, mode="nearest")
            x = conv(conv(torch.cat([up, skips[2 - k]], dim=1), 8 + 2 * k), 9 + 2 * k)
        out = torch.einsum("bchw,c->bhw", x, head) + hb + x0
        if case["backward"]:
            part = ((out - target[i:i + step].double()) ** 2).sum() / target.numel()
            part.backward(retain_graph=True)
            loss += float(part.detach())
        else:
            outs.append(out)
    if not case["backward"]:
        return torch.cat(outs)
    return dict(loss=torch.tensor([loss], dtype=torch.float64), grads=flat.grad)


def exact(case, seed):
    kind = case["kind"]
    if kind == "inpaint" or kind == "host":
        f, mask = _image_inputs(case, seed)
        return _exact_method(f, mask, case["N"], case)
    if kind == "diffuse":
        v = _volume(case, seed).to(torch.complex128)
        return _evolve(v, _sines(case["H"], case["H"], v.device), _sines(case["W"], case["W"], v.device),
                       case["beta"], case["T"], case["steps"])
    if kind == "batch":
        return [_exact_method(f, m, N, case, b) for f, m, N, b in _batch_inputs(case, seed)]
    return _unet_exact(case, seed)
