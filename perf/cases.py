"""Performance cases of the eMAGPIE library: what a user's programs have it do.

Every case runs one pass through the package's public entry points on synthetic ptychography data
of the kind the tests and the benchmark use: an object with random amplitude and smooth random
phase, a disk probe with a Gaussian edge and quadratic phase, a jittered raster scan whose patches
may leave the object, and Poisson-counted far-field intensities.  Reconstructions start from a
state in mid-run: the true object and probe with some noise.  Inputs are made on the GPU with plain
torch from the seed alone.  ``exact`` restates the method in 64 bits with plain torch.
"""
import math
import random

import numpy as np
import torch

import paper_2511_01793_gb300 as emg
from paper_2511_01793_gb300 import autograd as emg_autograd

ALPHA = float(np.float32(0.05))
W_EPS = float(np.float32(1e-6))
# The most a drawn case may have: pixels of all diffraction patterns, minibatches of one pass.
MAX_PIXELS = 4096 * 256 * 256
MAX_MINIBATCHES = 128


def _epochs(name, **kw):
    return dict(dict(name=name, kind="epochs", prolong="bilinear", joint=1, dft="fft32", history=0, epochs=1), **kw)


def listed():
    return [
        # The smallest call: one position per step, as in the paper's sequential sweep, driven
        # from the caller's own loop.
        dict(name="step_m64_b1", kind="step", rows=256, cols=256, m=64, side_r=16, side_c=16, step=12, jitter=2,
             noise=0.02, levels=2, prolong="const", joint=1, dft="fft32", b=1),
        # The small parity configuration: a 10 x 10 noise-free scan with a 32-pixel probe, one
        # level, minibatches of 10; an interactive or test-sized reconstruction.
        _epochs("epoch_m32_b10", rows=128, cols=128, m=32, side_r=10, side_c=10, step=8, jitter=1, noise=0.0, levels=1,
                prolong="const", b=10),
        # A mid-sized scan that is watched: after the epoch the misfit history the stopping rules
        # read is computed and returned.
        _epochs("epoch_m64_watched", rows=512, cols=512, m=64, side_r=38, side_c=38, step=8, jitter=2, noise=0.02,
                levels=2, b=64, history=1),
        # The performance configuration (the benchmark's default workload).
        _epochs("epoch_m128_b64", rows=512, cols=512, m=128, side_r=30, side_c=30, step=12, jitter=2, noise=0.02, levels=3,
                b=64),
        # The precision configuration at full size with FP32 FFTs: the largest reconstruction.
        _epochs("epoch_m256_b256", rows=2048, cols=2048, m=256, side_r=64, side_c=64, step=28, jitter=3, noise=0.02,
                levels=3, b=256),
        # The same probe and minibatch with the DFT pair on the tensor cores, on a quarter of the scan.
        _epochs("epoch_m256_bf16x3", rows=1024, cols=1024, m=256, side_r=32, side_c=32, step=24, jitter=3, noise=0.02,
                levels=3, b=256, dft="bf16x3"),
        # End to end from pinned host buffers: new data and start state in, one epoch, state and
        # misfit back (the performance configuration).
        dict(name="host_m128_b64", kind="host", rows=512, cols=512, m=128, side_r=30, side_c=30, step=12, jitter=2,
             noise=0.02, levels=3, prolong="bilinear", joint=1, dft="fft32", b=64, epochs=1),
        # Gradient-based reconstruction: misfit and Wirtinger gradients at full size through
        # autograd, forward and backward (the differentiation configuration).
        dict(name="autograd_m256", kind="autograd", rows=1024, cols=1024, m=256, side_r=40, side_c=40, step=20, jitter=2,
             noise=0.02),
        # Misfit and gradients in one call on a mid-sized problem, as an outer optimiser asks for them.
        dict(name="gradient_m64", kind="gradient", rows=512, cols=512, m=64, side_r=38, side_c=38, step=8, jitter=2,
             noise=0.02),
        # Many uneven reconstructions advanced together, one epoch each.
        dict(name="batch_12", kind="batch", count=12, pick=3),
        # The forward model: simulated intensities of a scan.
        dict(name="simulate_m128", kind="simulate", rows=512, cols=512, m=128, side_r=30, side_c=30, step=12, jitter=2),
        # The quality of a finished reconstruction against a reference: the illuminated region and
        # the errors after the best alignment over it.
        dict(name="quality_n512", kind="quality", rows=512, cols=512, m=128, side_r=30, side_c=30, step=12, jitter=2),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_scan(rng, ms):
    m = rng.choice(ms)
    most = min(4096, MAX_PIXELS // (m * m))
    n_pos = _log_int(rng, 64, most)
    side_r = max(4, int(math.sqrt(n_pos) * rng.uniform(0.7, 1.4)))
    side_c = max(4, min(n_pos // side_r, most // side_r))
    step = max(2, int(m * rng.uniform(0.07, 0.3)))
    rows = min(2048, (side_r - 1) * step + m + rng.randint(-m // 4, m))
    cols = min(2048, (side_c - 1) * step + m + rng.randint(-m // 4, m))
    return dict(rows=rows, cols=cols, m=m, side_r=side_r, side_c=side_c, step=step, jitter=rng.randint(0, 3))


def _draw_params(rng, c):
    n_pos = c["side_r"] * c["side_c"]
    lo = max(1, n_pos // MAX_MINIBATCHES)
    return dict(noise=rng.choice([0.0, 0.01, 0.02]), levels=rng.choice([1, 2, 3, 3]) if c["m"] > 16 else rng.choice([1, 2]),
                prolong=rng.choice(["const", "bilinear", "bilinear"]), joint=rng.choice([1, 1, 1, 0]),
                dft="bf16x3" if c["m"] >= 128 and rng.random() < 0.25 else "fft32",
                b=min(n_pos, _log_int(rng, max(lo, 4), max(lo, 4, min(256, n_pos)))))


def draw(rng: random.Random):
    kind = rng.choice(["epochs", "epochs", "epochs", "epochs", "step", "host", "autograd", "gradient", "batch", "simulate",
                       "quality"])
    if kind == "batch":
        return dict(kind=kind, count=rng.randint(2, 12), pick=rng.randint(10, 10 ** 6))
    sizes = [16, 32, 64, 128, 256]
    if kind == "epochs":
        c = _draw_scan(rng, sizes)
        return dict(c, kind=kind, history=rng.choice([0, 0, 1]), epochs=1, **_draw_params(rng, c))
    if kind == "step":
        c = _draw_scan(rng, sizes)
        return dict(c, kind=kind, **dict(_draw_params(rng, c), b=_log_int(rng, 1, min(64, c["side_r"] * c["side_c"]))))
    if kind == "host":
        c = _draw_scan(rng, [32, 64, 128])
        # pinning host memory is slow: at most the performance configuration's data
        c["side_r"] = min(c["side_r"], 30)
        c["side_c"] = min(c["side_c"], 30)
        return dict(c, kind=kind, epochs=1, **dict(_draw_params(rng, c), dft="fft32"))
    if kind in ("autograd", "gradient"):
        c = _draw_scan(rng, sizes)
        while c["side_r"] * c["side_c"] * c["m"] ** 2 > 1600 * 256 * 256:
            c["side_r"] -= 1
        return dict(c, kind=kind, noise=rng.choice([0.0, 0.01, 0.02]))
    c = _draw_scan(rng, sizes if kind == "simulate" else [32, 64, 128, 256])
    while kind == "quality" and c["side_r"] * c["side_c"] > 1600:
        c["side_r"] -= 1
    return dict(c, kind=kind)


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------

def _batch_members(case):
    """Uneven problems: object side 256-1024, probe side 64-256 (at most half the object), 100-1600
    positions with a raster step of m / 8, two or three levels."""
    rng = random.Random(case["pick"])
    members, pixels = [], 0
    for _ in range(case["count"]):
        n = rng.choice([256, 512, 768, 1024])
        m = rng.choice([v for v in (64, 128, 256) if v <= n // 2])
        side = max(10, min(int(math.sqrt(rng.randint(100, 1600))), (n - m) // (m // 8) + 1))
        side = min(side, max(4, int(math.sqrt(max(1, (MAX_PIXELS // 2 - pixels) // (m * m))))))
        pixels += side * side * m * m
        members.append(dict(kind="epochs", rows=n, cols=n, m=m, side_r=side, side_c=side, step=m // 8, jitter=2,
                            noise=0.02, levels=rng.choice([2, 3]), prolong="bilinear", joint=1, dft="fft32",
                            b=min(64, side * side), epochs=1, history=0))
    return members


def _probe(m, device):
    radius = m / 3.2
    x = torch.arange(m, dtype=torch.float64, device=device) - (m - 1) / 2.0
    r = torch.sqrt(x[:, None] ** 2 + x[None, :] ** 2)
    amp = torch.where(r <= radius, torch.ones_like(r), torch.exp(-((r - radius) ** 2) / (2.0 * (m / 4.0) ** 2)))
    return torch.polar(amp, math.pi * (r / radius) ** 2).to(torch.complex64)


def _object(rows, cols, g):
    dev = g.device
    amp = 0.8 + 0.2 * torch.rand((rows, cols), generator=g, device=dev)
    white = torch.randn((rows, cols), generator=g, device=dev)
    fy, fx = torch.fft.fftfreq(rows, device=dev), torch.fft.fftfreq(cols, device=dev)
    low = torch.exp(-2.0 * math.pi ** 2 * 16.0 * (fy[:, None] ** 2 + fx[None, :] ** 2))
    s = torch.fft.ifft2(torch.fft.fft2(white) * low).real
    s = (s - s.min()) / (s.max() - s.min())
    return torch.polar(amp, math.pi * (2.0 * s - 1.0))


def _scan(case, g):
    r0 = (case["rows"] - (case["m"] + (case["side_r"] - 1) * case["step"])) // 2
    c0 = (case["cols"] - (case["m"] + (case["side_c"] - 1) * case["step"])) // 2
    r = r0 + case["step"] * torch.arange(case["side_r"], device=g.device)
    c = c0 + case["step"] * torch.arange(case["side_c"], device=g.device)
    pos = torch.stack(torch.meshgrid(r, c, indexing="ij"), dim=-1).reshape(-1, 2)
    j = case["jitter"]
    if j:
        pos = pos + torch.randint(-j, j + 1, pos.shape, generator=g, device=g.device)
    return pos.to(torch.int32).contiguous()


def _patches(z, pos, m):
    """z_k = P_k z (zero outside the object) and the flat object indices with their validity."""
    rows, cols = z.shape
    a = torch.arange(m, device=z.device)
    r = pos[:, 0].long()[:, None] + a
    c = pos[:, 1].long()[:, None] + a
    ok = ((r >= 0) & (r < rows))[:, :, None] & ((c >= 0) & (c < cols))[:, None, :]
    flat = r.clamp(0, rows - 1)[:, :, None] * cols + c.clamp(0, cols - 1)[:, None, :]
    return z.reshape(-1)[flat] * ok, flat, ok


def _chunks(n_pos, m):
    size = max(1, (1 << 24) // (m * m))
    return [(a, min(a + size, n_pos)) for a in range(0, n_pos, size)]


def _noise(x, rel, g):
    s = rel * float(x.abs().square().mean().sqrt()) / math.sqrt(2.0)
    return x + s * torch.complex(torch.randn(x.shape, generator=g, device=g.device),
                                 torch.randn(x.shape, generator=g, device=g.device))


def _inputs(case, seed, data=True):
    """Positions, intensities and the truth with noise (the state in mid-run), on the GPU."""
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    m = case["m"]
    z, q, pos = _object(case["rows"], case["cols"], g), _probe(m, g.device), _scan(case, g)
    d = None
    if data:
        d = torch.empty((len(pos), m, m), dtype=torch.float32, device=g.device)
        for a, b in _chunks(len(pos), m):
            d[a:b] = torch.fft.fft2(_patches(z, pos[a:b], m)[0] * q).abs().square()
            if case["noise"]:
                d[a:b] *= 1.0 + case["noise"] * torch.randn(d[a:b].shape, generator=g, device=g.device)
    return dict(z=z, q=q, pos=pos, d=d, z0=_noise(z, 0.03, g), q0=_noise(q, 0.03, g))


def _context(case, seed, x, **kw):
    p = emg.emg_default_params(
        alpha=ALPHA, levels=case.get("levels", 1), minibatch=case.get("b", min(64, len(x["pos"]))),
        prolong=emg.EMG_PROLONG_BILINEAR if case.get("prolong") == "bilinear" else emg.EMG_PROLONG_CONST,
        joint=case.get("joint", 1), w_eps=W_EPS, seed=int(seed) & 0xFFFF,
        dft=emg.EMG_DFT_BF16X3 if case.get("dft") == "bf16x3" else emg.EMG_DFT_FFT32)
    return emg.Context(x["pos"], x["d"], case["rows"], case["cols"], p, **kw)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        members = _batch_members(case)
        ctxs = []
        for i, c in enumerate(members):
            x = _inputs(c, seed * 64 + i)
            ctxs.append(_context(c, seed * 64 + i, x, obj=x["z0"], probe=x["q0"]))
            del ctxs[-1].intensity  # the library keeps its own amplitudes
        return dict(kind=kind, ctxs=ctxs, batch=_Batch(ctxs))
    x = _inputs(case, seed, data=kind not in ("simulate", "quality"))
    if kind in ("epochs", "step"):
        ctx = _context(case, seed, x, obj=x["z0"], probe=x["q0"])
        s = dict(kind=kind, ctx=ctx, epochs=case.get("epochs", 1), history=bool(case.get("history", 0)))
        if kind == "step":
            s["idx"] = _step_indices(case, seed)
        return s
    if kind == "host":
        ctx = _context(case, seed, x)
        pinned = {k: torch.empty(x[k].shape, dtype=x[k].dtype, pin_memory=True) for k in ("d", "z0", "q0")}
        for k, v in pinned.items():
            v.copy_(x[k])
        del ctx.intensity
        return dict(kind=kind, ctx=ctx, epochs=case["epochs"], pinned=pinned, **{k: v.numpy() for k, v in pinned.items()})
    if kind in ("autograd", "gradient"):
        ctx = _context(case, seed, x)
        s = dict(kind=kind, ctx=ctx, obj=x["z0"].contiguous(), probe=x["q0"].contiguous())
        if kind == "autograd":
            s["obj"].requires_grad_(True)
            s["probe"].requires_grad_(True)
        return s
    if kind == "simulate":
        return dict(kind=kind, z=x["z0"].contiguous(), q=x["q0"].contiguous(), pos=x["pos"])
    return dict(kind=kind, z=x["z0"].contiguous(), q=x["q0"].contiguous(), zr=x["z"].contiguous(), qr=x["q"].contiguous(),
                pos=x["pos"])


class _Batch:
    """The batch handle, destroyed with the state."""

    def __init__(self, ctxs):
        self.ctxs = ctxs  # outlive the handle
        self.handle = emg.emg_batch_create([c.ctx for c in ctxs])

    def __del__(self):
        emg.emg_batch_destroy(self.handle)


def _step_indices(case, seed):
    n_pos = case["side_r"] * case["side_c"]
    return np.random.default_rng(int(seed)).permutation(n_pos)[:case["b"]].astype(np.int32)


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------

def run(s):
    kind = s["kind"]
    if kind == "epochs":
        running, misfit = emg.emg_run_epochs(s["ctx"].ctx, s["epochs"], running=s["history"], misfit=s["history"])
        out = dict(object=s["ctx"].obj, probe=s["ctx"].probe)
        if s["history"]:
            out.update(running=[float(v) for v in running], misfit=[float(v) for v in misfit])
        return out
    if kind == "step":
        emg.emg_step_minibatch(s["ctx"].ctx, s["idx"])
        return dict(object=s["ctx"].obj, probe=s["ctx"].probe)
    if kind == "batch":
        emg.emg_batch_run_epochs(s["batch"].handle, 1, torch.cuda.current_stream().cuda_stream)
        return [dict(object=c.obj, probe=c.probe) for c in s["ctxs"]]
    if kind == "host":
        _, misfit = emg.emg_reconstruct_host(s["ctx"].ctx, s["d"], s["z0"], s["q0"], s["epochs"], misfit=True)
        return dict(object=s["z0"], probe=s["q0"], misfit=[float(v) for v in misfit])
    if kind == "autograd":
        loss = emg_autograd.misfit(s["obj"], s["probe"], s["ctx"])
        g_obj, g_probe = torch.autograd.grad(loss, (s["obj"], s["probe"]))
        return dict(misfit=float(loss.item()), g_obj=g_obj, g_probe=g_probe)
    if kind == "gradient":
        g_obj, g_probe = torch.empty_like(s["obj"]), torch.empty_like(s["probe"])
        phi = emg.emg_misfit_gradient(s["ctx"].ctx, s["obj"].data_ptr(), s["probe"].data_ptr(), g_obj.data_ptr(),
                                      g_probe.data_ptr())
        return dict(misfit=float(phi), g_obj=g_obj, g_probe=g_probe)
    stream = torch.cuda.current_stream().cuda_stream
    rows, cols = s["z"].shape
    m, n_pos = s["q"].shape[0], len(s["pos"])
    if kind == "simulate":
        d = torch.empty((n_pos, m, m), dtype=torch.float32, device=s["z"].device)
        emg.emg_simulate_intensity(s["z"].data_ptr(), rows, cols, s["q"].data_ptr(), m, s["pos"].data_ptr(), n_pos,
                                   d.data_ptr(), stream)
        return d
    region = torch.empty((rows, cols), dtype=torch.uint8, device=s["z"].device)
    emg.emg_illuminated_region(s["qr"].data_ptr(), m, s["pos"].data_ptr(), n_pos, rows, cols, 0.1, region.data_ptr(), stream)
    e = emg.emg_aligned_errors(s["z"].data_ptr(), s["zr"].data_ptr(), rows, cols, s["q"].data_ptr(), s["qr"].data_ptr(), m,
                               region.data_ptr(), stream)
    return dict(region=region, c_re=e["c"].real, c_im=e["c"].imag, object=e["object"], probe=e["probe"],
                phase_rms=e["phase_rms"])


# ---------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------

def work(case):
    if case["kind"] == "batch":
        w = [work(c) for c in _batch_members(case)]
        return {k: sum(v[k] for v in w) for k in ("bytes", "flops")}
    m, kind = case["m"], case["kind"]
    mm, n_pos, px = m * m, case["side_r"] * case["side_c"], case["rows"] * case["cols"]
    fft = 5 * mm * math.log2(mm)
    if kind == "step":
        n_pos = case["b"]
        px = min(px, n_pos * mm)
    if kind in ("epochs", "step", "host"):
        mg = 100 * mm * sum(4.0 ** -l for l in range(case["levels"]))
        one = n_pos * (2 * fft + mg)
        data = 4 * n_pos * mm
        flops = case.get("epochs", 1) * one
        if case.get("history") or kind == "host":
            flops += case["epochs"] * n_pos * (fft + 12 * mm)
        return {"bytes": data + 16 * (px + mm), "flops": flops}
    if kind in ("autograd", "gradient"):
        return {"bytes": 4 * n_pos * mm + 16 * (px + mm), "flops": n_pos * (2 * fft + 40 * mm)}
    if kind == "simulate":
        return {"bytes": 4 * n_pos * mm + 8 * (px + mm), "flops": n_pos * (fft + 9 * mm)}
    # the illumination as one correlation over the positions' patches, then the reductions
    return {"bytes": 17 * px + 24 * mm, "flops": 4.0 * n_pos * mm + 60 * px}


# ---------------------------------------------------------------------------
# The same in 64 bits with plain torch
# ---------------------------------------------------------------------------

def _schedule(seed, epoch, n):
    """SplitMix64 (Steele, Lea, Flood 2014) and Fisher-Yates: the default schedule of an epoch."""
    mask = (1 << 64) - 1
    s = (seed + epoch * 0x9E3779B97F4A7C15) & mask
    out = list(range(n))
    for i in range(n - 1, 0, -1):
        s = (s + 0x9E3779B97F4A7C15) & mask
        x = s
        x = ((x ^ (x >> 30)) * 0xBF58476D1CE4E5B9) & mask
        x = ((x ^ (x >> 27)) * 0x94D049BB133111EB) & mask
        j = (x ^ (x >> 31)) % (i + 1)
        out[i], out[j] = out[j], out[i]
    return out


def _ratio(num, den):
    return torch.where(den != 0, num / torch.where(den != 0, den, torch.ones_like(den)), torch.zeros_like(num))


def _restrict(x):
    return 0.25 * (x[..., 0::2, 0::2] + x[..., 1::2, 0::2] + x[..., 0::2, 1::2] + x[..., 1::2, 1::2])


def _prolong_axis(y, dim):
    n = y.shape[dim]
    i = torch.arange(n, device=y.device)
    lo = y.index_select(dim, (i - 1).clamp(min=0))
    hi = y.index_select(dim, (i + 1).clamp(max=n - 1))
    both = torch.stack([0.75 * y + 0.25 * lo, 0.75 * y + 0.25 * hi], dim=dim + 1 if dim >= 0 else y.dim() + dim + 1)
    shape = list(y.shape)
    shape[dim] = 2 * n
    return both.reshape(shape)


def _prolong(y, kind):
    if kind == "bilinear":
        return _prolong_axis(_prolong_axis(y, y.dim() - 2), y.dim() - 1)
    return y.repeat_interleave(2, -2).repeat_interleave(2, -1)


def _object_step(q, z, r, u, levels, kind):
    gain = _ratio(q.conj(), (u + q.abs().square()).to(q.dtype))
    if levels > 1:
        a2 = q.abs().square()
        ra2 = _restrict(a2)
        s = _prolong(ra2, kind)
        qh = _restrict(q)
        wz = _ratio(a2, s)
        wr = _ratio(_prolong(qh, kind) * q.conj(), s.to(q.dtype))
        uh = _ratio(qh.abs().square(), ra2) * _restrict(u)
        zh = _restrict(wz * z)
        z = z + _prolong(_object_step(qh, zh, _restrict(wr * r), uh, levels - 1, kind) - zh, kind)
    return z + gain * (r - q * z)


def _joint(x, xp):
    root = torch.sqrt(x * xp)
    return torch.where((root * x.conj()).real < 0, -root, root)


def _revised(psi, a):
    """R_k and the misfit of each position."""
    big = torch.fft.fft2(psi)
    mod = big.abs()
    phase = torch.where(mod > 0, big / torch.where(mod > 0, mod, torch.ones_like(mod)), torch.ones_like(big))
    return torch.fft.ifft2(a * phase), 0.5 * (mod - a).square().sum(dim=(1, 2)) / (psi.shape[-1] ** 2)


def _minibatch(case, z, q, pos, a):
    m, kind = case["m"], case["prolong"]
    zk, flat, ok = _patches(z, pos, m)
    r, phi = _revised(q * zk, a)
    a2 = q.abs().square()
    mq = a2.max()
    zt = _object_step(q, zk, r, ALPHA * (mq - a2), case["levels"], kind)
    mu = zk.abs().square().amax(dim=(1, 2))
    live = mu > 0
    qt = q + zk.conj() / torch.where(live, mu, torch.ones_like(mu))[:, None, None] * (r - q * zk)
    if case["joint"]:
        zt, qt = _joint(zk, zt), _joint(q.expand_as(qt), qt)
    w = (a2 + W_EPS * mq) * ok
    num = torch.zeros(z.numel(), dtype=z.dtype, device=z.device).index_add_(0, flat.reshape(-1), (w * zt).reshape(-1))
    den = torch.zeros(z.numel(), dtype=torch.float64, device=z.device).index_add_(0, flat.reshape(-1), w.reshape(-1))
    cover = torch.zeros(z.numel(), dtype=torch.float64, device=z.device).index_add_(
        0, flat.reshape(-1), ok.reshape(-1).to(torch.float64))
    z = torch.where((cover > 0).reshape(z.shape), _ratio(num, den.to(num.dtype)).reshape(z.shape), z)
    if bool(live.any()):
        q = qt[live].mean(dim=0)
    return z, q, float(phi.sum())


def _amplitudes(d):
    return d.double().clamp(min=0).sqrt()


def _misfit(z, q, pos, d):
    m, total = q.shape[0], 0.0
    for a, b in _chunks(len(pos), m):
        total += float(_revised(q * _patches(z, pos[a:b], m)[0], _amplitudes(d[a:b]))[1].sum())
    return total


def _exact_epochs(case, seed):
    x = _inputs(case, seed)
    z, q, pos = x["z0"].to(torch.complex128), x["q0"].to(torch.complex128), x["pos"]
    n_pos, b = len(pos), case["b"]
    running, misfit = [], []
    for e in range(case["epochs"]):
        order = torch.tensor(_schedule(int(seed) & 0xFFFF, e, n_pos), device=pos.device)
        total = 0.0
        for a in range(0, n_pos, b):
            k = order[a:a + b]
            z, q, phi = _minibatch(case, z, q, pos[k], _amplitudes(x["d"][k]))
            total += phi
        running.append(total)
        if case.get("history") or case["kind"] == "host":
            misfit.append(_misfit(z, q, pos, x["d"]))
    out = dict(object=z, probe=q)
    if case["kind"] == "host":
        out.update(misfit=misfit)
    elif case.get("history"):
        out.update(running=running, misfit=misfit)
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return [_exact_epochs(c, seed * 64 + i) for i, c in enumerate(_batch_members(case))]
    if kind in ("epochs", "host"):
        out = _exact_epochs(case, seed)
        if kind == "host":
            out = {k: v.cpu().numpy() if isinstance(v, torch.Tensor) else v for k, v in out.items()}
        return out
    x = _inputs(case, seed, data=kind not in ("simulate", "quality"))
    z, q, pos, m = x["z0"].to(torch.complex128), x["q0"].to(torch.complex128), x["pos"], case["m"]
    if kind == "step":
        k = torch.from_numpy(_step_indices(case, seed)).long().to(pos.device)
        z, q, _ = _minibatch(case, z, q, pos[k], _amplitudes(x["d"][k]))
        return dict(object=z, probe=q)
    if kind == "simulate":
        d = torch.empty((len(pos), m, m), dtype=torch.float64, device=z.device)
        for a, b in _chunks(len(pos), m):
            d[a:b] = torch.fft.fft2(_patches(z, pos[a:b], m)[0] * q).abs().square()
        return d
    if kind in ("autograd", "gradient"):
        gz, gq, total = torch.zeros(z.numel(), dtype=z.dtype, device=z.device), torch.zeros_like(q), 0.0
        for a, b in _chunks(len(pos), m):
            zk, flat, ok = _patches(z, pos[a:b], m)
            r, phi = _revised(q * zk, _amplitudes(x["d"][a:b]))
            e = q * zk - r
            total += float(phi.sum())
            gz.index_add_(0, flat.reshape(-1), (q.conj() * e * ok).reshape(-1))
            gq += (zk.conj() * e).sum(dim=0)
        return dict(misfit=total, g_obj=gz.reshape(z.shape), g_probe=gq)
    zr, qr = x["z"].to(torch.complex128), x["q"].to(torch.complex128)
    illum = torch.zeros(z.numel(), dtype=torch.float64, device=z.device)
    for a, b in _chunks(len(pos), m):
        _, flat, ok = _patches(z, pos[a:b], m)
        illum.index_add_(0, flat.reshape(-1), (qr.abs().square() * ok).reshape(-1))
    region = (illum >= 0.1 * illum.max()).reshape(z.shape)
    a, b = z[region], zr[region]
    c = (a.conj() * b).sum() / a.abs().square().sum()
    norm = lambda v: v.abs().square().sum().sqrt()  # noqa: E731
    return dict(region=None, c_re=float(c.real), c_im=float(c.imag), object=float(norm(c * a - b) / norm(b)),
                probe=float(norm(q / c - qr) / norm(qr)),
                phase_rms=float(torch.angle(c * a * b.conj()).square().mean().sqrt()))
