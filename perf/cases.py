"""Performance cases of the hologram-rendering library: what its users have it do.

Every case goes through the public binding (paper_2508_03911_gb300.hv and .af) as a
program does: a handle is opened and its settings applied once (prepare), then each
pass pushes a batch of raw frames and renders every complete window (run). All work
is queued on one stream, as in a program that owns one GPU stream.

Streams with overlapping windows keep the last frames of a batch in the time queue;
prepare pushes the batch once beforehand, so every pass sees the same frames before
its own (the batch's own tail) and renders the same number of windows.
"""
import math

import numpy as np
import torch

from paper_2508_03911_gb300 import af, autofocus, hv

LAM, PITCH = 852e-9, 20e-6
MOMENTS = ("M0", "M1", "M2", "M1N", "M2N")
NZ = 64  # distances of the plain focus sweep

# ------------------------------------------------------------------ cases


def _stft(name, width, height, bits, spatial, T, S, nw, **kw):
    """A stream rendered by STFT: nw windows of T frames, S apart, per pass."""
    c = dict(kind="stft", width=width, height=height, bits=bits, spatial=spatial, T=T, S=S, nw=nw,
             z=0.30 if spatial == "asp" else 0.25, fs=71400.0, klo=max(1, T // 64), khi=max(1, (T * 49) // 100),
             moments="M0+M1+M2", tuned=1, highpass=0.0, conv=0, renorm=0, accumulate=1, host=0)
    c.update(kw)
    if name:
        c["name"] = name
    return c


def _pca(name, side, spatial, T, nw, groups, precision):
    c = dict(kind="pca", width=side, height=side, bits=16, spatial=spatial, T=T, S=T, nw=nw,
             z=0.40 if spatial == "asp" else 0.25, fs=20000.0, groups=groups, precision=precision, tuned=1)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # one preview image from 64 frames of an 8-bit camera, default settings: a
        # single short window, bound by launches and latency
        _stft("preview_asp_64", 256, 256, 8, "asp", 64, 64, 1, fs=20000.0, klo=4, khi=28, moments="M0", tuned=0),
        # live view: a camera's 12-bit frames in page-locked host memory, one window
        # in, its images back on the host before the next
        _stft("live_host_128", 256, 256, 16, "fresnel", 128, 128, 1, host=1),
        # offline rendering of a recording with separate windows (512/512)
        _stft("record_asp_512", 256, 256, 16, "asp", 512, 512, 8),
        # the sliding window of a long recording: 512 frames every 64
        _stft("stream_fresnel_512_64", 256, 256, 16, "fresnel", 512, 64, 64),
        # a wide sensor region with every output and the display chain: high-pass,
        # ragged stride, 5 x 5 Gaussian, re-normalised, mean of the last 4 images
        _stft("display_1024x512_128_48", 1024, 512, 16, "asp", 128, 48, 9, moments="M0+M1+M2+M1N+M2N",
              highpass=0.02, conv=5, renorm=1, accumulate=4),
        # propagated fields themselves (no temporal analysis), 8-bit frames, default form
        dict(name="fields_fresnel_512", kind="fields", width=512, height=512, bits=8, spatial="fresnel", z=0.25,
             n=96, tuned=0),
        # eigen-decomposition of short windows, many per pass
        _pca("pca_fresnel_256_t32", 256, "fresnel", 32, 128, 7, "fp32"),
        # eigen-decomposition of long windows of large frames, tensor-core covariance
        _pca("pca_asp_512_t256", 512, "asp", 256, 2, 31, "split_bf16"),
        # eight cameras of uneven sizes stepped together, four windows each
        dict(name="group_uneven_8", kind="group", nw=4, fs=71400.0,
             members="128:32:fresnel,128:128:asp,256:512:asp,256:32:fresnel,512:128:asp,512:32:fresnel,"
                     "1024:128:asp,1024:32:fresnel"),
        # plain autofocus: 64 distances for each hologram of a batch
        dict(name="focus_sweep_64", kind="sweep", side=256, n=64, nz=NZ),
        # learned autofocus, inference: log-spectra of a batch, then the network
        dict(name="autofocus_infer_512", kind="infer", n=512),
        # learned autofocus, training: loss and gradients of a batch
        dict(name="autofocus_grad_256", kind="grad", n=256),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_stft(rng):
    w, h = rng.choice([64, 128, 256, 256, 512, 1024]), rng.choice([64, 128, 256, 256, 512, 1024])
    if rng.random() < 0.5:
        h = w
    T = rng.choice([8, 16, 32, 64, 128, 256, 512, 1024])
    most = max(1, (1 << 26) // (w * h))  # frames of a pass
    while T > most:
        T //= 2
    S = T if rng.random() < 0.4 else rng.randint(max(1, T // 8), min(2 * T, most))
    lo = -(-T // S)
    nw = _log_int(rng, lo, max(lo, most // S))
    spatial = rng.choice(["asp", "asp", "fresnel", "none"])
    klo = rng.randint(0, T // 2)
    kw = dict(fs=rng.choice([20000.0, 71400.0]), klo=klo, khi=rng.randint(klo, T - 1 if rng.random() < 0.3 else max(klo, T // 2)),
              moments="+".join(m for m in MOMENTS if rng.random() < 0.5) or "M0", tuned=rng.randint(0, 1))
    if spatial == "asp" and rng.random() < 0.3:
        kw["highpass"] = round(rng.uniform(0.005, 0.1), 4)
    lag = -(-T // S) - 1  # windows of a pass that begin in the batch before
    if rng.random() < 0.4:
        kw.update(conv=rng.choice([0, 3, 5, 9]), renorm=rng.randint(0, 1),
                  accumulate=rng.randint(1, max(1, min(8, nw - lag))))
    if w * h * nw * S <= 1 << 24 and rng.random() < 0.3:
        kw["host"] = 1
    return _stft(None, w, h, rng.choice([8, 16]), spatial, T, S, nw, **kw)


def draw(rng):
    kind = rng.choice(["stft", "stft", "stft", "stft", "pca", "fields", "group", "sweep", "infer", "grad"])
    if kind == "stft":
        return _draw_stft(rng)
    if kind == "pca":
        T = rng.choice([32, 32, 64, 128, 256])
        side = rng.choice([128, 256, 512])
        groups = rng.randint(3, T // 8) if T > 32 else rng.randint(2, 7)
        prec = "fp32" if T < 128 else rng.choice(["fp32", "split_bf16"])
        nw = _log_int(rng, 1, max(1, min(128, (1 << 27) // (T * side * side)))) if T <= 64 else 1
        return _pca(None, side, rng.choice(["asp", "fresnel"]), T, nw, groups, prec)
    if kind == "fields":
        w, h = rng.choice([64, 128, 256, 512, 1024]), rng.choice([64, 128, 256, 512, 1024])
        spatial = rng.choice(["asp", "fresnel"])
        return dict(kind="fields", width=w, height=h, bits=rng.choice([8, 16]), spatial=spatial,
                    z=0.30 if spatial == "asp" else 0.25, n=_log_int(rng, 1, (1 << 26) // (w * h)),
                    tuned=rng.randint(0, 1))
    if kind == "group":
        m = []
        for _ in range(rng.randint(2, 6)):
            side = rng.choice([128, 256, 512])
            m.append("%d:%d:%s" % (side, rng.choice([32, 64, 128]), rng.choice(["asp", "fresnel"])))
        return dict(kind="group", nw=rng.randint(1, 4), fs=71400.0, members=",".join(m))
    if kind == "sweep":
        side = rng.choice([128, 256, 256, 512])
        return dict(kind="sweep", side=side, n=_log_int(rng, 1, (1 << 22) // (side * side)), nz=rng.randint(8, NZ))
    if kind == "infer":
        return dict(kind="infer", n=_log_int(rng, 1, 512))
    return dict(kind="grad", n=_log_int(rng, 1, 256))


# ----------------------------------------------------------------- inputs

_STREAM = None


def _stream():
    """The program's one stream."""
    global _STREAM
    if _STREAM is None:
        _STREAM = torch.cuda.Stream()
    return _STREAM


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _points(gen, n, height, width, z, count, radius, cx=0.0, cy=0.0):
    """n sensor fields (n, H, W) of `count` point scatterers each, paraxial spherical
    waves converging at distance z (n,): the phase separates in x and y, so a field
    is a product of two thin matrices."""
    dev = "cuda"
    rad = radius * torch.sqrt(torch.rand((n, count), generator=gen, device=dev, dtype=torch.float64))
    ang = 2 * math.pi * torch.rand((n, count), generator=gen, device=dev, dtype=torch.float64)
    amp = (0.25 + 0.75 * (torch.rand((n, count), generator=gen, device=dev) < 0.3)).to(torch.complex64)
    amp = amp * torch.exp(2j * math.pi * torch.rand((n, count), generator=gen, device=dev))
    c = (math.pi * PITCH * PITCH / (LAM * z)).reshape(-1, 1, 1)

    def axis(size, pos):
        d = torch.arange(size, device=dev, dtype=torch.float64).reshape(1, 1, -1) - size / 2 - pos.unsqueeze(-1)
        ph = torch.remainder(c * d * d, 2 * math.pi).to(torch.float32)
        return torch.polar(torch.ones_like(ph), -ph)

    ax = axis(width, cx + rad * torch.cos(ang))
    ay = axis(height, cy + rad * torch.sin(ang))
    return torch.matmul((ay * amp.unsqueeze(-1)).transpose(1, 2), ax)


def _carrier(height, width):
    c = torch.arange(width, device="cuda").reshape(1, -1) + torch.arange(height, device="cuda").reshape(-1, 1)
    return math.sqrt(10.0) * torch.exp(0.5j * math.pi * (c % 4))  # |R|^2 = 10 <|O|^2>, at a quarter of the band


def _record(inten, gen, bits):
    """Shot noise and the camera's pixel type: uint8, or 12-bit values in 16 bits."""
    full = 255 if bits == 8 else 4095
    v = torch.poisson(inten, generator=gen).clamp_(0, full)
    return v.to(torch.uint8 if bits == 8 else torch.int16)


def _frames(seed, n, height, width, bits, z, bins, T):
    """n frames of an off-axis recording: a static speckle object and one group of
    scatterers turning at bin b of T frames for every b of `bins`."""
    gen = _gen(seed)
    zz = torch.full((1,), z, device="cuda", dtype=torch.float64)
    side = min(height, width)
    static = _points(gen, 1, height, width, zz, 96, side / 4)[0]
    moving = torch.cat([_points(gen, 1, height, width, zz, 16, side / 8, side / 10, side / 10) for _ in bins])
    static = static / static.abs().square().mean().sqrt()
    moving = moving / moving.abs().square().mean((1, 2), keepdim=True).sqrt() / math.sqrt(len(bins))
    base = (_carrier(height, width) + static * math.sqrt(0.5)).reshape(1, -1)
    moving = (moving * math.sqrt(0.5)).reshape(len(bins), -1)
    gain = 0.30 * (255 if bits == 8 else 4095) / 11.0
    out = torch.empty((n, height, width), dtype=torch.uint8 if bits == 8 else torch.int16, device="cuda")
    turn = 2 * math.pi / T * torch.tensor([float(b) for b in bins], device="cuda", dtype=torch.float64)
    step = max(1, (1 << 25) // (height * width))
    for a in range(0, n, step):
        b = min(n, a + step)
        ph = torch.remainder(torch.arange(a, b, device="cuda", dtype=torch.float64).reshape(-1, 1) * turn,
                             2 * math.pi).to(torch.float32)
        u = torch.polar(torch.ones_like(ph), ph) @ moving + base
        out[a:b] = _record(gain * (u.real.square() + u.imag.square()), gen, bits).reshape(b - a, height, width)
    return out


def _bins(case):
    """Doppler lines of a recording, as bins of its window (fractions allowed)."""
    T = case["T"]
    if case["kind"] == "pca":  # evenly spaced lines: the sub-basis 2 .. 1 + 2 groups ends at a clear gap
        return [float(b) * (T // 2 // (case["groups"] + 1)) for b in range(1, case["groups"] + 1)]
    return [T * f for f in (0.03, 0.07, 0.13, 0.22, 0.31)]


def _holograms(seed, n, side):
    """n holograms (12-bit) of 24 point scatterers at a distance of their own, and the distances."""
    gen = _gen(seed)
    z = 0.10 + 0.50 * torch.rand(n, generator=gen, device="cuda", dtype=torch.float64)
    out = torch.empty((n, side, side), dtype=torch.int16, device="cuda")
    ref = _carrier(side, side)
    for a in range(0, n, 128):
        b = min(n, a + 128)
        f = _points(gen, b - a, side, side, z[a:b], 24, 32.0)
        f = f / f.abs().square().mean((1, 2), keepdim=True).sqrt()
        inten = (ref + f).abs().square()
        out[a:b] = _record(inten * (0.30 * 4095 / 11.0), gen, 16)
    return out, z.to(torch.float32)


def _net_inputs(seed, n):
    """Network inputs as training sees them: standardised log-spectra of holograms,
    here smooth random images with their statistics, and target distances."""
    gen = _gen(seed)
    x = torch.randn((n, 1, 128, 128), generator=gen, device="cuda")
    x = 0.8 * x + 0.6 * torch.randn((n, 1, 128, 1), generator=gen, device="cuda")
    z = 0.10 + 0.50 * torch.rand(n, generator=gen, device="cuda")
    return x.to(torch.bfloat16), z


def _net_params(seed):
    """He-uniform weights and small biases (a network some steps into training)."""
    p = autofocus.he_uniform(int(seed) & 0x7FFFFFFF)
    rng = np.random.default_rng(int(seed) & 0x7FFFFFFF)
    for name, o, n, _ in _tensors():
        if name[0] == "b" or name.endswith("b"):
            p[o:o + n] = rng.uniform(-0.05, 0.05, n)
    return p.astype(np.float32)


def _tensors():
    shapes = [("w1", (16, 1, 3, 3)), ("b1", (16,)), ("w2", (32, 16, 3, 3)), ("b2", (32,)), ("w3", (64, 32, 3, 3)),
              ("b3", (64,)), ("w4", (64, 64, 3, 3)), ("b4", (64,)), ("f1w", (32, 64)), ("f1b", (32,)),
              ("f2w", (1, 32)), ("f2b", (1,))]
    o, out = 0, []
    for name, s in shapes:
        n = int(np.prod(s))
        out.append((name, o, n, s))
        o += n
    return out


def _members(case):
    return [(int(a), int(b), c) for a, b, c in (m.split(":") for m in case["members"].split(","))]


# ---------------------------------------------------------------- prepare


def _renderer(width, height, bits, cap):
    return hv.Renderer(width, height, bits, cap, stream=_stream().cuda_stream)


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("stft", "pca"):
        w, h, T, S, n = case["width"], case["height"], case["T"], case["S"], case["nw"] * case["S"]
        frames = _frames(seed, n, h, w, case["bits"], case["z"], _bins(case), T)
        r = _renderer(w, h, case["bits"], n + T + S)
        kw = dict(spatial=case["spatial"], z=case["z"], T=T, stride=S, fs=case["fs"], tuned=case["tuned"])
        if kind == "pca":
            r.set_params(w, h, temporal="pca", pca=(2, 1 + 2 * case["groups"]), precision=case["precision"], **kw)
            nout = 1
        else:
            m = tuple(case["moments"].split("+"))
            r.set_params(w, h, band=(case["klo"], case["khi"]), moments=m, highpass=case["highpass"], **kw)
            nout = len(m)
            if case["conv"] or case["renorm"] or case["accumulate"] > 1:
                hv.hv_set_postprocess(r.h, kernel_size=case["conv"], sigma=case["conv"] / 5.0,
                                      renormalize=bool(case["renorm"]), accumulate=case["accumulate"])
        host = bool(case.get("host"))
        if host:
            frames = frames.cpu().pin_memory()
        out = torch.zeros((case["nw"], nout, h, w), dtype=torch.float32)
        out = out.pin_memory() if host else out.cuda()
        torch.cuda.synchronize()
        s = dict(kind="render", r=r, frames=frames, out=out, host=host)
        run(s)  # settings applied (and the tuned kernels chosen), the time queue filled
    elif kind == "fields":
        w, h, n = case["width"], case["height"], case["n"]
        frames = _frames(seed, n, h, w, case["bits"], case["z"], [3.0, 7.0], 32)
        r = _renderer(w, h, case["bits"], n)
        r.set_params(w, h, spatial=case["spatial"], z=case["z"], temporal="none", tuned=case["tuned"])
        out = torch.zeros((n, h, w, 2), dtype=torch.float32, device="cuda")
        torch.cuda.synchronize()
        s = dict(kind="render", r=r, frames=frames, out=out, host=False)
        run(s)
    elif kind == "group":
        rs, frames, outs = [], [], []
        for i, (side, T, spatial) in enumerate(_members(case)):
            z = 0.30 if spatial == "asp" else 0.25
            n = case["nw"] * T
            r = _renderer(side, side, 16, n)
            r.set_params(side, side, spatial=spatial, z=z, T=T, stride=T, fs=case["fs"],
                         band=(max(1, T // 64), T // 2 - 1), moments=("M0", "M1", "M2"), tuned=1)
            rs.append(r)
            frames.append(_frames(int(seed) * 101 + i, n, side, side, 16, z, [0.1 * T, 0.3 * T], T))
            outs.append(torch.zeros((case["nw"], 3, side, side), dtype=torch.float32, device="cuda"))
        torch.cuda.synchronize()
        s = dict(kind="group", rs=rs, frames=frames, outs=outs,
                 g=_Group(hv.hv_group_open([r.h for r in rs], stream=_stream().cuda_stream, use_graph=True), rs))
        run(s)
    elif kind in ("sweep", "infer"):
        n = case["n"]
        side = case.get("side", 256)
        frames, _ = _holograms(seed, n, side)
        r = _renderer(side, side, 16, n)
        r.set_params(side, side, spatial="asp", z=0.3, T=16, stride=16, band=(1, 7))
        if kind == "sweep":
            zs = np.linspace(0.10, 0.60, case["nz"])
            s = dict(kind="sweep", r=r, frames=frames, zs=zs, metric=torch.zeros((n, case["nz"]), device="cuda"))
        else:
            net = af.Autofocus(n, stream=_stream().cuda_stream)
            net.set_params(_net_params(seed))
            s = dict(kind="infer", r=r, frames=frames, net=net,
                     feats=torch.zeros((n, 1, 128, 128), dtype=torch.bfloat16, device="cuda"),
                     z=torch.zeros(n, device="cuda"))
        torch.cuda.synchronize()
        run(s)  # settings applied, the sweep's transfer functions built
    else:
        n = case["n"]
        x, z = _net_inputs(seed, n)
        net = af.Autofocus(n, stream=_stream().cuda_stream)
        net.set_params(_net_params(seed))
        s = dict(kind="grad", net=net, x=x, z=z, loss=torch.zeros(1, device="cuda"),
                 grad=torch.zeros(af.NPARAMS, device="cuda"))
    torch.cuda.synchronize()
    return s


class _Group:
    """A group handle closed before its members."""

    def __init__(self, g, members):
        self.g, self.members = g, members

    def __del__(self):
        hv.hv_group_close(self.g)
        for r in self.members:
            r.close()


# -------------------------------------------------------------------- run


def run(s):
    kind = s["kind"]
    if kind == "render":
        r, out = s["r"], s["out"]
        # host frames are copied in and the images read back; device frames, complete
        # already, are read in place
        if r.push(s["frames"], async_=not s["host"]) != hv.HV_OK:
            raise RuntimeError("input queue full")
        r.render(out)
        return out
    if kind == "group":
        hv.hv_render_group(s["g"].g, s["frames"], s["outs"])
        return s["outs"]
    if kind == "sweep":
        hv.hv_focus_sweep(s["r"].h, s["frames"], s["zs"], s["metric"])
        return s["metric"]
    if kind == "infer":
        hv.hv_af_features(s["r"].h, s["frames"], s["feats"])
        s["net"].forward(s["feats"], s["z"])
        return {"features": s["feats"], "z": s["z"]}
    s["net"].loss_grad(s["x"], s["z"], s["loss"], s["grad"])
    return {"loss": s["loss"], "grad": s["grad"]}


# ------------------------------------------------------------------- work


def _spatial_flops(spatial, hw):
    fft2 = 5.0 * hw * math.log2(hw)
    # ASP: the transform of a real frame (half a complex one), the product, the inverse
    return 1.5 * fft2 + 6.0 * hw if spatial == "asp" else (fft2 + 4.0 * hw if spatial == "fresnel" else 0.0)


# multiply-adds of the network per image: four convolutions, two dense layers
_NET_MACS = [9 * 1 * 16 * 64 * 64, 9 * 16 * 32 * 32 * 32, 9 * 32 * 64 * 16 * 16, 9 * 64 * 64 * 8 * 8, 64 * 32 + 32]


def work(case):
    kind = case["kind"]
    if kind in ("stft", "pca"):
        hw, T, S, nw = case["width"] * case["height"], case["T"], case["S"], case["nw"]
        used = nw * min(S, T)  # frames of the batch that some window needs
        nout = len(case["moments"].split("+")) if kind == "stft" else 1
        b = used * hw * (case["bits"] // 8) + 4.0 * nw * nout * hw
        f = used * _spatial_flops(case["spatial"], hw)
        if kind == "stft":
            f += nw * hw * (5.0 * T * math.log2(T) + 7.0 * (case["khi"] - case["klo"] + 1))
            f += nw * nout * hw * (2.0 * case["conv"] ** 2 + case["accumulate"])
        else:
            # Hermitian covariance and projection onto the sub-basis, per pixel
            f += nw * hw * (4.0 * T * T + 8.0 * T * 2 * case["groups"])
        return {"bytes": b, "flops": f}
    if kind == "fields":
        hw = case["width"] * case["height"]
        return {"bytes": case["n"] * hw * (case["bits"] // 8 + 8.0),
                "flops": case["n"] * _spatial_flops(case["spatial"], hw)}
    if kind == "group":
        b = f = 0.0
        for side, T, spatial in _members(case):
            hw, n = side * side, case["nw"] * T
            b += n * hw * 2.0 + case["nw"] * 3 * hw * 4.0
            f += n * _spatial_flops(spatial, hw) + case["nw"] * hw * (5.0 * T * math.log2(T) + 3.5 * T)
        return {"bytes": b, "flops": f}
    if kind == "sweep":
        hw, n, nz = case["side"] ** 2, case["n"], case["nz"]
        fft2 = 5.0 * hw * math.log2(hw)
        return {"bytes": n * hw * 2.0 + n * nz * 4.0, "flops": n * (0.5 * fft2 + nz * (fft2 + 10.0 * hw))}
    n = case["n"]
    if kind == "infer":
        return {"bytes": n * (65536 * 2.0 + 16384 * 2.0 + 4.0),
                "flops": n * (2.5 * 65536 * 16 + 2.0 * sum(_NET_MACS))}
    # forward, and backward's weight gradients (all layers) and input gradients (all but the first)
    return {"bytes": n * 16384 * 2.0 + 3 * 4.0 * af.NPARAMS,
            "flops": n * 2.0 * (3 * sum(_NET_MACS) - _NET_MACS[0])}


# -------------------------------------------------------------- tolerance


def tolerance(case):
    """About four times the largest error against exact() over listed and drawn cases."""
    kind = case["kind"]
    if kind == "fields":
        return {"rel": 1e-6}  # 1.8e-7: float32 transforms
    if kind == "group":
        return {"rel": 2e-6}  # 3e-7
    if kind == "sweep":
        return {"rel": 2e-7}  # 4e-8: ratios of float64 sums of float32 amplitudes
    if kind == "infer":
        return {"rel": 7e-3}  # 1.7e-3: the features' rounding to bfloat16
    if kind == "grad":
        return {"rel": 1e-3}  # 2.2e-4: activations that round to the other bfloat16 neighbour
    if kind == "pca":
        return {"rel": 3e-6}  # 5.4e-7
    # 1.1e-6 for a band of one bin of shot noise beside a static part a thousand times larger
    return {"rel": 5e-6}


# ------------------------------------------------------------------ exact


def _pixels(frames):
    """Raw frames as float64."""
    return frames.cuda().to(torch.float64)


def _propagate(frames, spatial, z, highpass=0.0):
    """The field of every frame in complex128, one frame group at a time."""
    n, h, w = frames.shape
    dev = frames.device
    if spatial == "none":
        return _pixels(frames).to(torch.complex128)
    fx = torch.fft.fftfreq(w, device=dev, dtype=torch.float64)
    fy = torch.fft.fftfreq(h, device=dev, dtype=torch.float64)
    out = torch.empty((n, h, w), dtype=torch.complex128, device=dev)
    if spatial == "asp":
        k = 2 * math.pi / LAM
        kx, ky = 2 * math.pi / PITCH * fx.reshape(1, -1), 2 * math.pi / PITCH * fy.reshape(-1, 1)
        kz2 = k * k - kx * kx - ky * ky
        ph = z * torch.sqrt(kz2.clamp(min=0.0))
        keep = (kz2 >= 0) & ((fx.reshape(1, -1) ** 2 + fy.reshape(-1, 1) ** 2 >= highpass * highpass) | (highpass <= 0))
        H = torch.polar(keep.to(torch.float64), ph)
    else:
        c = math.pi * PITCH * PITCH / (LAM * z)
        x = (torch.arange(w, device=dev, dtype=torch.float64) - w / 2).reshape(1, -1)
        y = (torch.arange(h, device=dev, dtype=torch.float64) - h / 2).reshape(-1, 1)
        ph = c * (x * x + y * y)
        H = torch.polar(torch.ones_like(ph), ph)
    step = max(1, (1 << 24) // (h * w))
    for a in range(0, n, step):
        u = _pixels(frames[a:a + step])
        if spatial == "asp":
            out[a:a + step] = torch.fft.ifft2(torch.fft.fft2(u) * H)
        else:
            out[a:a + step] = torch.fft.fftshift(torch.fft.fft2(u * H), dim=(1, 2))
    return out


def _moments(u, T, klo, khi, fs, names):
    """The outputs of one window u (T, H, W), stacked."""
    S = torch.fft.fft(u, dim=0)[klo:khi + 1]
    P = S.real.square() + S.imag.square()
    k = torch.arange(klo, khi + 1, device=u.device, dtype=torch.float64)
    f = (torch.where(k < T // 2, k, k - T) * (fs / T / 1000.0)).reshape(-1, 1, 1)
    m0, m1, m2 = P.sum(0), (f * P).sum(0), (f * f * P).sum(0)
    d = torch.where(m0 > 0, m0, torch.ones_like(m0))
    zero = torch.zeros_like(m0)
    got = {"M0": m0, "M1": m1, "M2": m2, "M1N": torch.where(m0 > 0, m1 / d, zero),
           "M2N": torch.where(m0 > 0, torch.sqrt((m2 / d).clamp(min=0)), zero)}
    return torch.stack([got[m] for m in MOMENTS if m in names])


def _postprocess(img, case):
    """Convolution (periodic, Gaussian), division by the mean, mean of the last images;
    the images before a pass's first are the last ones of the pass before, the same."""
    K = case["conv"]
    if K:
        d = torch.arange(K, device=img.device, dtype=torch.float64) - K // 2
        s = float(np.float32(K / 5.0))
        k = torch.exp(-(d.reshape(-1, 1) ** 2 + d.reshape(1, -1) ** 2) / (2 * s * s))
        k = k / k.sum()
        acc = torch.zeros_like(img)
        for a in range(K):
            for b in range(K):
                acc += k[a, b] * torch.roll(img, (K // 2 - a, K // 2 - b), dims=(2, 3))
        img = acc
    if case["renorm"]:
        mean = img.mean((2, 3), keepdim=True)
        img = torch.where(mean != 0, img / torch.where(mean != 0, mean, torch.ones_like(mean)), torch.zeros_like(img))
    A = case["accumulate"]
    if A > 1:
        n = img.shape[0]
        img = torch.stack([sum(img[(i - j) % n] for j in range(A)) / A for i in range(n)])
    return img


def _exact_stft(case, frames):
    T, S, nw = case["T"], case["S"], case["nw"]
    before = S * (-(-T // S) - 1)  # frames of the batch before that this pass's windows still hold
    u = _propagate(frames.cuda(), case["spatial"], case["z"], case.get("highpass", 0.0))
    names = case["moments"].split("+")
    out = []
    for i in range(nw):
        at = torch.arange(i * S, i * S + T, device=u.device) - before
        out.append(_moments(u[at % u.shape[0]], T, case["klo"], case["khi"], case["fs"], names))
    out = torch.stack(out)
    return _postprocess(out, case) if "conv" in case else out


def _exact_pca(case, frames):
    T, nw, m = case["T"], case["nw"], 1 + 2 * case["groups"]
    out = []
    for i in range(nw):
        u = _propagate(frames[i * T:(i + 1) * T], case["spatial"], case["z"])
        X = u.reshape(T, -1)
        C = X.conj() @ X.T  # C[a, b] = sum over pixels of conj(X_a) X_b
        lam, V = torch.linalg.eigh(C.cpu())
        V = V.to(u.device)[:, torch.argsort(lam, descending=True).to(u.device)][:, 1:m]
        y = X.T @ V
        out.append((y.real.square() + y.imag.square()).sum(1).reshape(1, case["height"], case["width"]))
    return torch.stack(out)


def _exact_sweep(case, frames):
    out = torch.zeros((case["n"], case["nz"]), dtype=torch.float64, device="cuda")
    for j, z in enumerate(np.linspace(0.10, 0.60, case["nz"])):
        for a in range(0, case["n"], 32):
            f = _pixels(frames[a:a + 32])
            amp = _propagate(f - f.mean((1, 2), keepdim=True), "asp", float(z)).abs()
            mu, sd = amp.mean((1, 2)), amp.std((1, 2), unbiased=False)
            out[a:a + 32, j] = torch.where(mu > 0, torch.sqrt(sd / torch.where(mu > 0, mu, torch.ones_like(mu))), mu)
    return out


def _exact_features(frames):
    out = []
    for a in range(0, frames.shape[0], 64):
        f = _pixels(frames[a:a + 64])
        F = torch.fft.fftshift(torch.fft.fft2(f - f.mean((1, 2), keepdim=True)), dim=(1, 2)).abs()
        n, h, w = F.shape
        v = torch.log1p(F.reshape(n, h // 2, 2, w // 2, 2).mean((2, 4)))
        out.append((v - v.mean((1, 2), keepdim=True)) / v.std((1, 2), unbiased=False, keepdim=True))
    return torch.cat(out).unsqueeze(1)


def _bf16(x):
    """The value the method keeps in bfloat16, its gradient passed through."""
    return x + (x.detach().to(torch.float32).to(torch.bfloat16).to(torch.float64) - x.detach())


def _exact_net(x, flat):
    """The network's normalised output; weights and activations rounded where the method keeps bfloat16."""
    p = {name: flat[o:o + n].reshape(s) for name, o, n, s in _tensors()}
    a = x
    for layer in range(1, 5):
        w = _bf16(p["w%d" % layer])
        n, ci, h, _ = a.shape
        cols = torch.nn.functional.unfold(a, 3, padding=1, stride=2)
        y = w.reshape(w.shape[0], -1) @ cols + p["b%d" % layer].reshape(-1, 1)
        a = _bf16(torch.relu(y).reshape(n, w.shape[0], h // 2, h // 2))
    g = a.mean((2, 3))
    hid = torch.relu(g @ p["f1w"].T + p["f1b"])
    return (hid @ p["f2w"].T + p["f2b"]).reshape(-1)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("stft", "pca"):
        n = case["nw"] * case["S"]
        frames = _frames(seed, n, case["height"], case["width"], case["bits"], case["z"], _bins(case), case["T"])
        return _exact_stft(case, frames) if kind == "stft" else _exact_pca(case, frames)
    if kind == "fields":
        frames = _frames(seed, case["n"], case["height"], case["width"], case["bits"], case["z"], [3.0, 7.0], 32)
        return torch.view_as_real(_propagate(frames, case["spatial"], case["z"]))
    if kind == "group":
        out = []
        for i, (side, T, spatial) in enumerate(_members(case)):
            z, n = 0.30 if spatial == "asp" else 0.25, case["nw"] * T
            frames = _frames(int(seed) * 101 + i, n, side, side, 16, z, [0.1 * T, 0.3 * T], T)
            c = dict(T=T, S=T, nw=case["nw"], spatial=spatial, z=z, fs=case["fs"], klo=max(1, T // 64),
                     khi=T // 2 - 1, moments="M0+M1+M2")
            out.append(_exact_stft(c, frames).to(torch.float64))
        return out
    if kind == "sweep":
        return _exact_sweep(case, _holograms(seed, case["n"], case["side"])[0])
    flat = torch.from_numpy(_net_params(seed)).cuda().to(torch.float64)
    if kind == "infer":
        feats = _exact_features(_holograms(seed, case["n"], 256)[0])
        with torch.no_grad():
            x = feats.to(torch.float32).to(torch.bfloat16).to(torch.float64)
            z = torch.cat([0.35 + 0.25 * _exact_net(x[a:a + 64], flat) for a in range(0, case["n"], 64)])
        return {"features": feats, "z": z}
    x, z = _net_inputs(seed, case["n"])
    flat.requires_grad_(True)
    loss = torch.zeros(1, dtype=torch.float64, device="cuda")
    for a in range(0, case["n"], 64):
        t = (z[a:a + 64].to(torch.float64) - 0.35) / 0.25
        part = (_exact_net(x[a:a + 64].to(torch.float64), flat) - t).square().sum() / case["n"]
        part.backward()
        loss += part.detach()
    return {"loss": loss, "grad": flat.grad}
