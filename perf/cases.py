"""The work that a user of this library has it do, as cases to be timed.

Kinds of a case ("kind"):
  plain    Plan.reconstruct / reconstruct_f64: frames of one pupil on one grid
           (powers of two, or the even windows that leave a few lenslets of
           padding around the pupil), slopes and phase resident on the GPU
  host     Plan.reconstruct_host: the same from pinned host buffers
  ragged   Batch.run: frames of several pupils and grids in one launch
  linear   LinearWarmStart.reconstruct: low-rank warm start, then the loop
  unet     Net.forward, then Plan.reconstruct from that warm start
  train    Net.gradients: forward, loss and backward pass of the network

Inputs are seeded von Karman slopes (D = 8 m, r0 = 0.15 m, L0 = 25 m, white
noise of 0.02 to 0.1 rad), the statistics of synth.py, made on the GPU.
"""

import math
import os

import numpy as np
import torch

from paper_1705_04298_gb300 import fwr, synth

R0, L0 = 0.15, 25.0
WEIGHTS = os.path.join("paper_1705_04298_gb300", "weights", "warmstart_w16_n40.npz")
RAGGED = ((40, 128), (64, 128), (80, 256), (128, 256))  # lenslets across, grid


def plain(n, N, frames, iters, **kw):
    c = {"kind": "plain", "n": n, "N": N, "frames": frames, "iters": iters, "filter": "lsq", "sigma": 0.05,
         "periodic": 0, "f64": False, "extended": False}
    c.update(kw)
    return c


def listed():
    return [
        # one frame of a small sensor, the converged loop: latency
        dict(plain(16, 32, 1, 10), name="one_16_32"),
        # the same in double precision, the path users check the others with
        dict(plain(16, 32, 1, 10, f64=True), name="one_16_32_f64"),
        # one step of a closed loop of a 40 x 40 system: a frame, few iterations
        dict(plain(40, 128, 1, 2, sigma=0.02, periodic=1), name="loop_40_128"),
        # the paper's system, a batch of telemetry frames (the benchmark's workload)
        dict(plain(40, 128, 1000, 10, filter="wiener", sigma=0.1), name="batch_40_128"),
        # the same frames from and to host memory
        dict(plain(40, 128, 1000, 10, filter="wiener", sigma=0.1, kind="host"), name="host_40_128"),
        # a long sequence of a larger sensor (the precision study's grid)
        dict(plain(128, 256, 1000, 10), name="batch_128_256"),
        # ELT scale: a short burst of frames
        dict(plain(200, 512, 16, 10), name="elt_200_512"),
        # the paper's small window: three lenslets of padding on each side
        dict(plain(40, 46, 1000, 10, filter="wiener", sigma=0.1), name="window_40_46"),
        # frames of four sensors in one launch
        {"kind": "ragged", "frames": 1024, "iters": 5, "name": "ragged_1024"},
        # linear warm start and one iteration in place of ten
        {"kind": "linear", "n": 40, "N": 128, "rank": 256, "frames": 1000, "iters": 1, "name": "linear_40_128"},
        # the network's warm start and one iteration
        {"kind": "unet", "frames": 1000, "iters": 1, "name": "unet_40_128"},
        # a training step's gradients at the training batch
        {"kind": "train", "frames": 256, "name": "train_256"},
    ]


# ------------------------------------------------------------------- draws --

def _log(rng, a, b):
    return max(a, min(b, int(round(math.exp(rng.uniform(math.log(a), math.log(b + 0.999)))))))


def _frames(rng, n, N, iters, most):
    """Frame counts from 1 to `most`, no more work than 1000 frames of 256^2, k = 10."""
    cap = int(_plain_flops(256, 10) * 1000 / _plain_flops(N, iters))
    return _log(rng, 1, max(1, min(most, cap)))


def draw(rng):
    kind = rng.choice(("plain",) * 6 + ("window", "window", "f64", "host", "ragged", "linear", "unet", "train"))
    iters = rng.choice((0, 1, 2, 3, 5, 10))
    opt = {"filter": rng.choice(("lsq", "wiener")), "sigma": rng.choice((0.02, 0.05, 0.1)),
           "periodic": rng.choice((0, 0, 0, 1, 2))}
    if kind in ("plain", "host"):
        N = rng.choice((16, 32, 64, 64, 128, 128, 256, 256, 512))
        n = _log(rng, max(8, N // 4), min(N - 2, 200))
        F = _frames(rng, n, N, iters, 1000 if N <= 256 else 150)
        if kind == "plain" and N <= 128 and rng.random() < 0.15:
            opt["extended"] = True  # training targets: the extended slopes too
        return plain(n, N, F, iters, kind=kind, **opt)
    if kind == "window":
        n = rng.randint(14, 56)
        N = min(64, n + n % 2 + 2 * rng.choice((1, 2, 3, 3, 4, 6)))
        if N & (N - 1) == 0:
            N -= 2
        n = min(n, N - 2)
        return plain(n, N, _log(rng, 1, 1000), iters, f64=rng.random() < 0.15, **opt)
    if kind == "f64":
        N = rng.choice((16, 32, 64))
        n = _log(rng, max(8, N // 4), N - 2)
        return plain(n, N, _log(rng, 1, 64), iters, f64=True, **opt)
    if kind == "ragged":
        return {"kind": "ragged", "frames": _log(rng, 8, 1500), "iters": iters}
    if kind == "linear":
        N = rng.choice((64, 128))
        n = rng.randint(N // 4, N // 2)
        return {"kind": "linear", "n": n, "N": N, "rank": rng.choice((128, 256, 512)),
                "frames": _log(rng, 1, 1000), "iters": rng.choice((1, 1, 2))}
    if kind == "unet":
        return {"kind": "unet", "frames": _log(rng, 1, 1000), "iters": rng.choice((1, 2))}
    return {"kind": "train", "frames": _log(rng, 4, 256)}


# ------------------------------------------------------------------ inputs --

def make_slopes(n, F, seed, sigma, dtype=torch.float32):
    """(F, 2, n, n) slopes of independent von Karman screens, zero outside the
    pupil: screens by the FFT method at half a pitch, slopes by trapezoidal
    means along the lenslet edges, white noise."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    M = 1 << max(1, (4 * n - 1).bit_length())
    d = synth.TELESCOPE_D / n
    f = torch.fft.fftfreq(M, d=d / 2, device="cuda", dtype=torch.float64)
    psd = 0.023 * R0 ** (-5.0 / 3.0) * (f[None, :] ** 2 + f[:, None] ** 2 + L0 ** -2.0) ** (-11.0 / 6.0)
    psd[0, 0] = 0.0
    amp = (psd.sqrt() * (M * M / (M * d / 2))).float()
    mask = torch.from_numpy(synth.pupil_mask(n)).cuda()
    out = torch.empty((F, 2, n, n), dtype=dtype, device="cuda")
    step = max(1, (1 << 25) // (M * M))
    w = (0.25, 0.5, 0.25)
    for a in range(0, F, step):
        b = min(F, a + step)
        z = torch.view_as_complex(torch.randn((b - a, M, M, 2), generator=g, device="cuda"))
        s = torch.fft.ifft2(z * amp).real
        sx = sum(w[r] * (s[:, r:r + 2 * n:2, 2:2 * n + 1:2] - s[:, r:r + 2 * n:2, 0:2 * n:2]) for r in range(3))
        sy = sum(w[r] * (s[:, 2:2 * n + 1:2, r:r + 2 * n:2] - s[:, 0:2 * n:2, r:r + 2 * n:2]) for r in range(3))
        v = torch.stack((sx, sy), 1)
        v = v + sigma * torch.randn(v.shape, generator=g, device="cuda")
        out[a:b] = torch.where(mask, v, torch.zeros_like(v)).to(dtype)
    return out


def make_plan(n, N, filt="lsq", sigma=0.0, periodic=0):
    r0, l0 = synth.pitch_units(n, R0, L0)
    return fwr.Plan(synth.pupil_mask(n), N / n, fwr.WIENER if filt == "wiener" else fwr.LSQ, sigma ** 2, r0, l0,
                    periodic, grid=N)


def linear_factors(n, N, rank):
    """Factors of the size and scale of a fitted operator, smooth in neither
    index: (2 n_valid, rank) and (2 N^2, rank)."""
    g = torch.Generator(device="cuda").manual_seed(11)
    k = 2 * int(synth.pupil_mask(n).sum())
    A = torch.randn((k, rank), generator=g, device="cuda") / math.sqrt(k)
    V = torch.randn((2 * N * N, rank), generator=g, device="cuda") / math.sqrt(rank)
    return A, V


def train_targets(F, seed):
    """Smooth extended slopes outside the pupil, (F, 2, 128, 128)."""
    g = torch.Generator(device="cuda").manual_seed(seed + 5)
    z = torch.randn((F, 2, 12, 12), generator=g, device="cuda")
    return torch.nn.functional.interpolate(z, size=(128, 128), mode="bicubic", align_corners=False).contiguous()


def ragged_plan_of(case, seed):
    """Which sensor each frame is of: equal counts, shuffled."""
    return np.random.default_rng(seed).permutation(np.arange(case["frames"]) % len(RAGGED))


def prepare(case, seed):
    kind, F = case["kind"], case.get("frames")
    st = {"case": case}
    if kind in ("plain", "host"):
        n, N = case["n"], case["N"]
        dt = torch.float64 if case["f64"] else torch.float32
        st["plan"] = make_plan(n, N, case["filter"], case["sigma"], case["periodic"])
        st["slopes"] = make_slopes(n, F, seed, case["sigma"], dt)
        if kind == "host":
            st["slopes"] = st["slopes"].cpu().pin_memory()
            st["phase"] = torch.empty((F, N, N), dtype=dt, pin_memory=True)
            st["plan"].reserve(F)
        else:
            st["phase"] = torch.empty((F, N, N), dtype=dt, device="cuda")
            if case["extended"]:
                st["ext"] = torch.empty((F, 2, N, N), dtype=dt, device="cuda")
    elif kind == "ragged":
        st["plans"] = [make_plan(n, N) for n, N in RAGGED]
        which = ragged_plan_of(case, seed)
        st["slopes"], st["phase"] = [], []
        ins, outs = [None] * F, [None] * F
        for p, (n, N) in enumerate(RAGGED):
            at = np.flatnonzero(which == p)
            s = make_slopes(n, len(at), seed + p, 0.05)
            o = torch.empty((len(at), N, N), device="cuda")
            st["slopes"].append(s)
            st["phase"].append(o)
            for i, f in enumerate(at):
                ins[f], outs[f] = s[i], o[i]
        st["in_ptrs"], st["out_ptrs"] = fwr.Batch.pointer_table(ins), fwr.Batch.pointer_table(outs)
        st["batch"] = fwr.Batch(st["plans"], which, case["iters"])
    elif kind == "linear":
        n, N = case["n"], case["N"]
        st["plan"] = make_plan(n, N, "wiener", 0.05)
        A, V = linear_factors(n, N, case["rank"])
        st["warm"] = fwr.LinearWarmStart(st["plan"], A.cpu().numpy(), V.cpu().numpy(), F)
        st["slopes"] = make_slopes(n, F, seed, 0.05)
        st["phase"] = torch.empty((F, N, N), device="cuda")
    else:
        d = np.load(WEIGHTS)
        st["net"] = fwr.Net(int(d["width"]), F, d["weights"])
        st["slopes"] = make_slopes(40, F, seed, 0.05)
        if kind == "unet":
            st["plan"] = make_plan(40, 128, "wiener", 0.05)
            st["ext"] = torch.empty((F, 2, 128, 128), device="cuda")
            st["phase"] = torch.empty((F, 128, 128), device="cuda")
        else:
            st["plan"] = make_plan(40, 128)
            st["target"] = train_targets(F, seed)
    return st


# --------------------------------------------------------------------- run --

def run(st):
    c = st["case"]
    kind = c["kind"]
    if kind == "plain":
        call = st["plan"].reconstruct_f64 if c["f64"] else st["plan"].reconstruct
        phase = call(st["slopes"], c["iters"], st["phase"], ext_out=st.get("ext"))
        return (phase, st["ext"]) if "ext" in st else phase
    if kind == "host":
        return st["plan"].reconstruct_host(st["slopes"], c["iters"], st["phase"])
    if kind == "ragged":
        st["batch"].run(st["in_ptrs"], st["out_ptrs"])
        return st["phase"]
    if kind == "linear":
        return st["warm"].reconstruct(st["slopes"], c["iters"], st["phase"])
    if kind == "unet":
        ext = st["net"].forward(st["plan"], st["slopes"], st["ext"])
        return ext, st["plan"].reconstruct(st["slopes"], c["iters"], st["phase"], ext_init=ext)
    loss, grad = st["net"].gradients(st["plan"], st["slopes"], st["target"])
    return {"loss": loss, "grad": grad}


# -------------------------------------------------------------------- work --

def _plain_flops(N, iters):
    """(2k + 1.5) complex N^2 transforms a frame, 5 N^2 log2(N^2) each."""
    return (2 * iters + 1.5) * 5.0 * N * N * math.log2(N * N)


def _plain_work(n, N, F, iters, size=4):
    return {"bytes": float(F) * (2 * n * n + N * N) * size, "flops": F * _plain_flops(N, iters)}


def _unet_macs(w=16):
    """Multiply-adds of one image through the network."""
    at = {32: (3 * w + w * w + 3 * w * w + w * w), 16: (2 * w * w + 4 * w * w + 12 * w * w + 4 * w * w),
          8: (8 * w * w + 16 * w * w + 32 * w * w + 16 * w * w), 4: 32 * w * w}
    return sum(9 * H * H * c for H, c in at.items()) + 32 * 32 * 2 * w


def work(case):
    kind = case["kind"]
    if kind in ("plain", "host"):
        w = _plain_work(case["n"], case["N"], case["frames"], case["iters"], 8 if case["f64"] else 4)
        if case["extended"]:
            w["bytes"] *= 2
        return w
    if kind == "ragged":
        parts = [_plain_work(n, N, len(range(p, case["frames"], len(RAGGED))), case["iters"])
                 for p, (n, N) in enumerate(RAGGED)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    F = case["frames"]
    if kind == "linear":
        n, N, r = case["n"], case["N"], case["rank"]
        w = _plain_work(n, N, F, case["iters"])
        k = 2 * int(synth.pupil_mask(n).sum())
        w["bytes"] += 2.0 * r * (k + 2 * N * N)
        w["flops"] += 2.0 * F * r * (k + 2 * N * N)
        return w
    if kind == "unet":
        w = _plain_work(40, 128, F, case["iters"])
        return {"bytes": w["bytes"] + 4.0 * F * 2 * 128 * 128, "flops": w["flops"] + 2.0 * F * _unet_macs()}
    return {"bytes": 4.0 * F * (2 * 40 * 40 + 2 * 128 * 128), "flops": 6.0 * F * _unet_macs()}


# ------------------------------------------------------------------- exact --
# What run() returns, in 64 bits, from the equations alone.

def _filters(n, N, filt, sigma):
    k = torch.arange(N, dtype=torch.float64, device="cuda")
    u = torch.where(k < N // 2, k, k - N) / N
    a = torch.exp(2j * math.pi * u) - 1
    t = torch.sinc(u) * torch.exp(1j * math.pi * u)
    t[N // 2] = 0
    gx, gy = t[:, None] * a[None, :], a[:, None] * t[None, :]
    g2 = gx.abs() ** 2 + gy.abs() ** 2
    ok = g2 >= 1e-14
    zero = torch.zeros_like(g2)
    lsq = torch.where(ok, 1 / torch.where(ok, g2, zero + 1), zero)
    last = lsq
    if filt == "wiener":
        r0, l0 = synth.pitch_units(n, R0, L0)
        w = 0.023 * r0 ** (-5.0 / 3.0) * (u[None, :] ** 2 + u[:, None] ** 2 + l0 ** -2.0) ** (-11.0 / 6.0)
        last = torch.where(ok, 1 / (g2 + sigma ** 2 / w), zero)
    return gx, gy, lsq, last


def exact_plain(slopes, n, N, iters, filt, sigma, periodic, ext=None):
    """(phases, extended slopes) of (F, 2, n, n) slopes, in 64 bits."""
    gx, gy, lsq, last = _filters(n, N, filt, sigma)
    off = (N - n) // 2
    mask = torch.zeros((N, N), dtype=torch.bool, device="cuda")
    mask[off:off + n, off:off + n] = torch.from_numpy(synth.pupil_mask(n)).cuda()
    phases, exts = [], []
    step = max(1, (1 << 22) // (N * N))

    def fill(s):
        s[:, 0, :, N - 1] = -s[:, 0, :, :N - 1].sum(2)
        s[:, 1, N - 1, :] = -s[:, 1, :N - 1, :].sum(1)

    for f in range(0, slopes.shape[0], step):
        m = torch.zeros((min(step, slopes.shape[0] - f), 2, N, N), dtype=torch.float64, device="cuda")
        m[:, :, off:off + n, off:off + n] = slopes[f:f + step].to(device="cuda", dtype=torch.float64)
        s = torch.where(mask, m, ext[f:f + step].double()) if ext is not None else torch.where(mask, m, m * 0)
        for it in range(iters + 1):
            if periodic == 0 or (periodic == 1 and it == iters):
                fill(s)
            t = torch.fft.fft2(s)
            p = gx.conj() * t[:, 0] + gy.conj() * t[:, 1]
            if it < iters:
                p = p * lsq
                s = torch.where(mask, m, torch.fft.ifft2(torch.stack((gx * p, gy * p), 1)).real)
            else:
                phases.append(torch.fft.ifft2(p * last).real)
                exts.append(s)
    return torch.cat(phases), torch.cat(exts)


def _bf16(x):
    """Rounded to BF16, with the gradient of the identity."""
    return x + (x.detach().to(torch.bfloat16).to(x.dtype) - x.detach())


def exact_net(flat, width, slopes):
    """The network's (F, 2, 32, 32) output in 64 bits: BF16 weights and stored
    activations are part of its definition, FP32 biases too. Returns the
    output and the leaves (weights, bias per layer) for gradients."""
    F = slopes.shape[0]
    mask = torch.zeros((128, 128), dtype=torch.float64, device="cuda")
    mask[44:84, 44:84] = torch.from_numpy(synth.pupil_mask(40)).cuda().double()
    x = torch.zeros((F, 3, 128, 128), dtype=torch.float64, device="cuda")
    x[:, :2, 44:84, 44:84] = 0.5 * slopes.double()
    x[:, 2] = 1.0
    x = _bf16(torch.nn.functional.avg_pool2d(x * mask, 4))
    w1, w2, w3 = width, 2 * width, 4 * width
    sizes = [(3, w1), (w1, w1), (w1, w2), (w2, w2), (w2, w3), (w3, w3), (w3, w3), (w3, w3), (2 * w3, w3), (w3, w3),
             (w3 + w2, w2), (w2, w2), (w2 + w1, w1), (w1, w1), (w1, 2)]
    leaves, at = [], 0
    for i, (ci, co) in enumerate(sizes):
        k = 1 if i == 14 else 3
        W = flat[at:at + co * k * k * ci].to(torch.bfloat16).double().view(co, k, k, ci)
        at += W.numel()
        b = flat[at:at + co].double()
        at += co
        leaves.append((W.requires_grad_(), b.requires_grad_()))

    def conv(i, x):
        W, b = leaves[i]
        k = W.shape[1]
        B, C, H, _ = x.shape
        cols = torch.nn.functional.unfold(x, k, padding=k // 2)             # B, C k k, H H
        y = torch.matmul(W.permute(0, 3, 1, 2).reshape(W.shape[0], -1), cols) + b[:, None]
        y = y.view(B, -1, H, H)
        return _bf16(torch.relu(y)) if i < 14 else y

    def pool(x):
        return _bf16(torch.nn.functional.avg_pool2d(x, 2))

    def up(x, skip):
        return torch.cat((x.repeat_interleave(2, 2).repeat_interleave(2, 3), skip), 1)

    s1 = conv(1, conv(0, x))
    s2 = conv(3, conv(2, pool(s1)))
    s3 = conv(5, conv(4, pool(s2)))
    y = conv(7, conv(6, pool(s3)))
    y = conv(9, conv(8, up(y, s3)))
    y = conv(11, conv(10, up(y, s2)))
    y = conv(13, conv(12, up(y, s1)))
    return conv(14, y), leaves


def exact_train(flat, width, slopes, target):
    """Loss and flat gradient in 64 bits, images in chunks."""
    t = torch.nn.functional.avg_pool2d(0.5 * target.double(), 4)
    pupil = torch.zeros((1, 1, 128, 128), dtype=torch.float64, device="cuda")
    pupil[0, 0, 44:84, 44:84] = torch.from_numpy(synth.pupil_mask(40)).cuda().double()
    lm = (torch.nn.functional.max_pool2d(pupil, 4) == 0).double()
    lm[:, :, 31, :] = 0
    lm[:, :, :, 31] = 0
    cnt = 2 * slopes.shape[0] * float(lm.sum())
    loss, grad = 0.0, 0
    for f in range(0, slopes.shape[0], 16):
        out, leaves = exact_net(flat, width, slopes[f:f + 16])
        part = (((out - t[f:f + 16]) * lm) ** 2).sum() / cnt
        g = torch.autograd.grad(part, [v for pair in leaves for v in pair])
        grad = grad + torch.cat([v.reshape(-1) for v in g])
        loss += float(part)
    return loss, grad


def exact(case, seed):
    kind, F = case["kind"], case.get("frames")
    if kind in ("plain", "host"):
        n, N = case["n"], case["N"]
        s = make_slopes(n, F, seed, case["sigma"], torch.float64 if case["f64"] else torch.float32)
        phase, ext = exact_plain(s, n, N, case["iters"], case["filter"], case["sigma"], case["periodic"])
        return (phase, ext) if case["extended"] else phase
    if kind == "ragged":
        which = ragged_plan_of(case, seed)
        return [exact_plain(make_slopes(n, int((which == p).sum()), seed + p, 0.05), n, N, case["iters"], "lsq", 0.05,
                            0)[0] for p, (n, N) in enumerate(RAGGED)]
    if kind == "linear":
        n, N = case["n"], case["N"]
        A, V = linear_factors(n, N, case["rank"])
        s = make_slopes(n, F, seed, 0.05)
        cells = torch.from_numpy(np.flatnonzero(synth.pupil_mask(n).ravel())).cuda()
        X = s.view(F, 2, n * n)[:, :, cells].reshape(F, -1)
        r = lambda v: v.to(torch.bfloat16).double()  # noqa: E731  (the factors and products are stored in BF16)
        ext = r(r(r(X) @ r(A)) @ r(V).T).view(F, 2, N, N)
        return exact_plain(s, n, N, case["iters"], "wiener", 0.05, 0, ext)[0]
    d = np.load(WEIGHTS)
    flat = torch.from_numpy(np.asarray(d["weights"], np.float32)).cuda()
    s = make_slopes(40, F, seed, 0.05)
    if kind == "unet":
        with torch.no_grad():
            out = torch.cat([exact_net(flat, int(d["width"]), s[f:f + 16])[0] for f in range(0, F, 16)])
        ext = (out / 0.5).repeat_interleave(4, 2).repeat_interleave(4, 3)
        return ext, exact_plain(s, 40, 128, case["iters"], "wiener", 0.05, 0, ext.float())[0]
    loss, grad = exact_train(flat, int(d["width"]), s, train_targets(F, seed))
    return {"loss": loss, "grad": grad}
