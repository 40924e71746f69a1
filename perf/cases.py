"""The work that users of this framework have it do, as measurable cases.

A case names a call (or a short sequence of calls) of the public entry points in
paper_1904_09409_gb300.funnel with its sizes; prepare() makes what a program has
in hand before the call (synthetic line images on the GPU or in pinned host
memory, a plan, output buffers), run() is one pass, exact() the same result in
64 bits with plain torch.  Images are the package's synthetic workload: straight
ridges and step edges at random slopes and intercepts, partly occluded, with
additive noise.

Map lengths must be even and of the form 2^a 3^b, so an image of any other size
is given the next such lengths (480 x 640 -> a 486 x 648 map); images whose
sides are such lengths already use them unchanged.
"""
import math
import random

import torch

from paper_1904_09409_gb300 import funnel, synth

LENGTHS = sorted(2 ** a * 3 ** b for a in range(1, 14) for b in range(9) if 2 ** a * 3 ** b <= funnel.FT_MAX_LENGTH)


def next_length(n):
    """The smallest supported map length >= n."""
    return next(v for v in LENGTHS if v >= n)


def listed():
    return [
        # one small photograph or camera frame at a time, where latency and
        # launches count: the single-image workload of the package (top-3)
        dict(name="detect_256", kind="detect", H=256, W=256, Hp=256, S=256, batch=1, interp="linear",
             space="regular", top_k=3, lines=3, noise=0.1),
        # a few VGA camera frames: neither side is a supported length, and the
        # next ones (486 x 648) are not among the powers of two
        dict(name="detect_vga", kind="detect", H=480, W=640, Hp=486, S=648, batch=8, interp="linear",
             space="regular", top_k=8, lines=8, noise=0.2),
        # the benchmark batch: 64 images of 1024 x 1024, maps only
        dict(name="forward_1024", kind="forward", H=1024, W=1024, Hp=1024, S=1024, batch=64, interp="linear",
             space="regular", lines=10, noise=0.2),
        # the same images arriving as consecutive batches, each with its peaks
        dict(name="stream_1024", kind="stream", H=1024, W=1024, Hp=1024, S=1024, batch=16, batches=4,
             interp="linear", space="regular", top_k=8, lines=10, noise=0.2),
        # one step of fitting by gradient: forward, loss against a target map and
        # the gradient with respect to the images, 32 x 512 x 512
        dict(name="train_512", kind="train", H=512, W=512, Hp=512, S=512, batch=32, interp="linear",
             space="regular", lines=8, noise=0.2),
        # the transform as a layer of a torch model on full-HD frames, with the
        # smoother interpolator: forward and backward through autograd
        dict(name="layer_fullhd_cubic", kind="layer", H=1080, W=1920, Hp=1152, S=1944, batch=2, interp="cubic",
             space="regular", lines=12, noise=0.1),
        # the paper's own band-limited interpolator on a batch of 1024 x 1024
        dict(name="forward_1024_fourier", kind="forward", H=1024, W=1024, Hp=1024, S=1024, batch=16,
             interp="fourier", space="regular", lines=10, noise=0.2),
        # the same interpolator in both directions where the map is longer than
        # the image and no length is a power of two
        dict(name="layer_576_fourier", kind="layer", H=432, W=576, Hp=432, S=648, batch=4, interp="fourier",
             space="regular", lines=6, noise=0.2),
        # steep lines (|k| > 1): the inverse space on 720p frames, with the
        # detected lines verified against the images
        dict(name="inverse_720p", kind="detect", H=720, W=1280, Hp=1296, S=768, batch=4, interp="linear",
             space="inverse", top_k=8, lines=8, noise=0.1, verify=True),
        # large scans with many lines
        dict(name="detect_4096", kind="detect", H=4096, W=4096, Hp=4096, S=4096, batch=4, interp="linear",
             space="regular", top_k=100, lines=100, noise=0.2),
        # a batch of images of uneven sizes (sides from the package's list)
        dict(name="mixed_sizes", kind="mixed", batch=96, sides="all", interp="linear", top_k=8, shape_seed=1),
        # from host memory to the list of lines, copies included
        dict(name="host_1024", kind="host", H=1024, W=1024, Hp=1024, S=1024, batch=16, interp="linear",
             space="regular", top_k=8, lines=10, noise=0.2),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A case of the same ranges: any image size from 64 to 4096 on a side, sides
    of any value (odd heights too), each call, interpolator and space."""
    kind = rng.choice(["detect", "detect", "detect", "forward", "stream", "train", "layer", "layer", "mixed", "host"])
    if kind == "mixed":
        return dict(kind="mixed", batch=rng.randint(16, 96), sides=rng.choice(["all", "small"]),
                    interp=rng.choice(["linear", "linear", "cubic"]), top_k=rng.randint(1, 8),
                    shape_seed=rng.randint(2, 1 << 20))
    interp = rng.choice(["linear", "linear", "cubic", "fourier"]) if kind in ("detect", "forward", "layer") else "linear"
    space = rng.choice(["regular", "regular", "regular", "inverse"]) if kind in ("detect", "layer") else "regular"
    top = 1024 if interp == "fourier" else 4096
    H, W = _log_int(rng, 64, top), _log_int(rng, 64, top)
    style = rng.choice(["own", "length", "power"])
    if interp == "fourier" and style == "own":
        style = "length"                                  # its image widths must be supported lengths
    if style == "length":
        H, W = next_length(H), next_length(W)
    elif style == "power":
        H, W = 1 << round(math.log2(H)), 1 << round(math.log2(W))
    W += W & 1                                            # the transform's width is even
    if space == "inverse":
        H += H & 1
        Hp, S = next_length(W), next_length(H)
    else:
        Hp, S = next_length(H), next_length(W)
    pixels = 12e6 if interp == "fourier" else 24e6
    batch = _log_int(rng, 1, max(1.0, min(64.0, pixels / (Hp * S))))
    c = dict(kind=kind, H=H, W=W, Hp=Hp, S=S, batch=batch, interp=interp, space=space,
             lines=rng.randint(2, 12), noise=round(rng.uniform(0.05, 0.3), 3))
    if kind in ("detect", "stream", "host"):
        c["top_k"] = rng.randint(1, 8)
    if kind == "stream":
        c["batches"] = rng.randint(2, 4)
        c["batch"] = max(1, batch // c["batches"])
    if kind == "detect":
        c["verify"] = rng.random() < 0.3
    return c


# ------------------------------------------------------------------- inputs
def _image(rng, gen, H, W, lines, noise):
    """One image: ridges and steps of random slope and intercept, parts of them
    occluded, background and noise (the package's synthetic content, drawn on the
    GPU).  In the inverse space the caller passes the transposed sizes."""
    dev = gen.device
    bg = rng.gauss(0.2, 0.05)
    img = torch.full((H, W), bg, dtype=torch.float32, device=dev)
    rows = torch.arange(H, dtype=torch.float32, device=dev)[:, None]
    cols = torch.arange(W, dtype=torch.float32, device=dev)[None, :]
    boxes = []
    for _ in range(lines):
        k, b = rng.uniform(-1.0, 1.0), rng.uniform(0.0, H)
        d = rows - (cols * k + b)
        if rng.random() < 0.5:
            sigma = rng.uniform(1.0, 3.0)
            img += torch.exp(d * d * (-0.5 / (sigma * sigma * (1.0 + k * k))))
        else:
            img += (d > 0) * rng.uniform(0.3, 1.0)
        c0 = rng.uniform(0.0, W)
        c1 = min(W - 1.0, c0 + rng.uniform(0.0, 0.3) * W)
        r0, r1 = sorted((k * c0 + b, k * c1 + b))
        boxes.append((max(0, int(r0) - 3), min(H, int(r1) + 4), max(0, int(c0) - 3), min(W, int(c1) + 4)))
    for r0, r1, c0, c1 in boxes:
        if r0 < r1 and c0 < c1:
            img[r0:r1, c0:c1] = bg
    return img + noise * torch.randn((H, W), generator=gen, dtype=torch.float32, device=dev)


def _images(case, seed, n):
    rng = random.Random(seed)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    inv = case["space"] == "inverse"
    H, W = (case["W"], case["H"]) if inv else (case["H"], case["W"])
    out = torch.empty((n, case["H"], case["W"]), dtype=torch.float32, device="cuda")
    for i in range(n):
        img = _image(rng, gen, H, W, case["lines"], case["noise"])
        out[i] = img.t() if inv else img
    return out, gen


def _target(case, gen, n):
    """Target maps of the gradient workload: Gaussian blobs (2 cells) at the
    cells of some lines, the blobs of one map drawn at random."""
    Hp, S = case["Hp"], case["S"]
    t = torch.arange(Hp, dtype=torch.float32, device="cuda")
    s = torch.arange(S, dtype=torch.float32, device="cuda")
    out = torch.zeros((n, Hp, S), dtype=torch.float32, device="cuda")
    for _ in range(case["lines"]):
        tc = torch.rand(n, generator=gen, device="cuda") * Hp
        sc = torch.rand(n, generator=gen, device="cuda") * S
        dt = (t[None] - tc[:, None] + Hp / 2) % Hp - Hp / 2
        ds = (s[None] - sc[:, None] + S / 2) % S - S / 2
        out += torch.exp(dt * dt / -8.0)[:, :, None] * torch.exp(ds * ds / -8.0)[:, None, :]
    return out


def _shapes(case):
    rng = random.Random(case["shape_seed"])
    sides = synth.VARLEN_SIDES if case["sides"] == "all" else [v for v in synth.VARLEN_SIDES if v <= 768]
    return [(rng.choice(sides), rng.choice(sides)) for _ in range(case["batch"])]


def _loss_scale(case):
    return 2.0 / case["W"]


def prepare(case, seed):
    st = dict(kind=case["kind"], case=case)
    if case["kind"] == "mixed":
        b = funnel.Batch(_shapes(case), interp=case["interp"])
        rng = random.Random(seed)
        gen = torch.Generator(device="cuda")
        gen.manual_seed(seed)
        st["x"] = torch.empty(b.img_total, dtype=torch.float32, device="cuda")
        for j, i in enumerate(b.order):
            h, w = b.shapes[i]
            o = int(b.img_off[j])
            st["x"][o:o + h * w] = _image(rng, gen, h, w, rng.randint(1, 12), 0.2).reshape(-1)
        st["batch"] = b
        st["map"] = torch.empty(b.map_total, dtype=torch.float32, device="cuda")
        n = b.n
    else:
        st["plan"] = funnel.Plan(case["H"], case["W"], case["S"], case["Hp"], case["interp"], case["space"])
        n = case["batch"] * case.get("batches", 1)
        x, gen = _images(case, seed, n)
        maps = (case["batch"], case["Hp"], case["S"])
        if case["kind"] == "host":
            st["x"] = x.cpu().pin_memory()
        elif case["kind"] == "stream":
            st["x"] = list(x.split(case["batch"]))
        elif case["kind"] == "layer":
            st["x"] = x.requires_grad_(True)
            st["g"] = torch.randn(maps, generator=gen, dtype=torch.float32, device="cuda")
        else:
            st["x"] = x
        if case["kind"] not in ("host", "layer"):
            st["map"] = torch.empty(maps, dtype=torch.float32, device="cuda")
        if case["kind"] == "train":
            st["target"] = _target(case, gen, n)
            st["loss"] = torch.empty(n, dtype=torch.float32, device="cuda")
            st["grad"] = torch.empty_like(x)
    if "top_k" in case:
        place = dict(pin_memory=True) if case["kind"] == "host" else dict(device="cuda")
        st["out"] = torch.empty(n * case["top_k"] * funnel.PEAK_DTYPE.itemsize, dtype=torch.uint8, **place)
        st["count"] = torch.empty(n, dtype=torch.int32, **place)
    return st


# ---------------------------------------------------------------------- run
def _peaks(st):
    """The peak records as their fields: cells (t, s), and value, k, b."""
    k = st["case"]["top_k"]
    rec = st["out"].view(torch.int32).view(-1, k, 5)
    return dict(count=st["count"], cell=rec[..., :2], line=st["out"].view(torch.float32).view(-1, k, 5)[..., 2:])


def run(st):
    c, kind = st["case"], st["kind"]
    if kind == "forward":
        funnel.ft_forward(st["plan"], st["x"], st["map"])
        return dict(map=st["map"])
    if kind == "detect":
        funnel.ft_detect(st["plan"], st["x"], st["map"], c["top_k"], out=st["out"], count=st["count"])
        r = dict(map=st["map"], **_peaks(st))
        if c.get("verify"):
            r["profile"], r["length"], r["verdict"] = funnel.ft_verify(st["plan"], st["x"], st["out"], st["count"],
                                                                       c["top_k"])
        return r
    if kind == "stream":
        funnel.ft_detect_batches(st["plan"], st["x"], st["map"], c["top_k"], out=st["out"], count=st["count"])
        return dict(map=st["map"], **_peaks(st))
    if kind == "train":
        funnel.ft_forward(st["plan"], st["x"], st["map"])
        funnel.ft_abs_mse_backward(st["plan"], st["map"], st["target"], _loss_scale(c), loss=st["loss"],
                                   grad_img=st["grad"])
        return dict(map=st["map"], loss=st["loss"], grad=st["grad"])
    if kind == "layer":
        st["x"].grad = None
        y = funnel.funnel_transform(st["x"], st["plan"])
        y.backward(st["g"])
        return dict(map=y.detach(), grad=st["x"].grad)
    if kind == "mixed":
        st["batch"].run(st["x"], st["map"], c["top_k"], out=st["out"], count=st["count"])
        return dict(map=st["map"], **_peaks(st))
    if kind == "host":
        funnel.ft_detect_host(st["plan"], st["x"], c["top_k"], out_host=st["out"], count_host=st["count"])
        return _peaks(st)
    raise ValueError(kind)


# --------------------------------------------------------------------- work
def _one_forward(H, W, Hp, S, interp, top_k=0):
    """Bytes and operations of one image: the image in and the map out (and the
    peaks), the real transforms of the columns, the interpolated rows and their
    transforms."""
    L = Hp // 2 + 1
    taps = {"linear": 8.0, "cubic": 28.0, "fourier": 0.0}[interp]
    flops = 2.5 * Hp * math.log2(Hp) * (W + S) + L * (taps * S + 5.0 * S * math.log2(S))
    if interp == "fourier":
        M = W + S
        flops += L * (5.0 * W * math.log2(W) + 10.0 * M * math.log2(M) + 6.0 * (W + S + M))
    return 4.0 * H * W + 4.0 * Hp * S + 20.0 * top_k, flops


def work(case):
    k = case.get("top_k", 0)
    if case["kind"] == "mixed":
        both = [_one_forward(h, w, h, w, case["interp"], k) for h, w in _shapes(case)]
        return dict(bytes=sum(b for b, _ in both), flops=sum(f for _, f in both))
    inv = case["space"] == "inverse"
    H, W = (case["W"], case["H"]) if inv else (case["H"], case["W"])
    b, f = _one_forward(H, W, case["Hp"], case["S"], case["interp"], k)
    image, cells = 4.0 * case["H"] * case["W"], 4.0 * case["Hp"] * case["S"]
    if case["kind"] == "train":          # the target in and the gradient out; the map is already in hand
        b, f = b + cells + image, 2.0 * f
    elif case["kind"] == "layer":        # the map's gradient in and the image's out
        b, f = b + cells + image, 2.0 * f
    elif case["kind"] == "stream":       # the maps are scratch: the last batch's are an output
        b = image + 20.0 * k + cells / case["batches"]
    elif case["kind"] == "host":
        b = image + 20.0 * k
    n = case["batch"] * case.get("batches", 1)
    return dict(bytes=n * b, flops=n * f)


# -------------------------------------------------------------------- exact
def _parity(n):
    return 1.0 - 2.0 * (torch.arange(n, device="cuda") % 2).double()


def _interpolate(F, S, Hp, interp):
    """Every row l >= 1 of F [L][W] (complex128, x centred) at x' H' / (2 l), x' =
    -S/2 .. S/2-1, zero outside the image columns; row 0 zero."""
    L, W = F.shape
    xp = torch.arange(S, device="cuda") - S // 2
    out = [torch.zeros((1, S), dtype=F.dtype, device="cuda")]
    step = max(1, (1 << 23) // S)
    if interp == "fourier":
        sgn = _parity(W)
        Fh = torch.fft.fft(F, dim=1) * sgn[None] / W       # coefficient of exp(2 pi j u x / W), u mod W
        u = torch.arange(-(W // 2), W // 2 + 1, device="cuda")
        wt = torch.ones(W + 1, dtype=torch.float64, device="cuda")
        wt[0] = wt[-1] = 0.5                               # the Nyquist term as a cosine
        C = Fh[:, u % W] * wt[None]
        for l in range(1, L):
            num, den = xp * Hp, 2 * l
            ok = (num >= -(W // 2) * den) & (num <= (W // 2 - 1) * den)
            r = (u[:, None] * num[None, ok]) % (den * W)   # the phase u p / W, reduced exactly
            th = r.double() * (2.0 * math.pi / (den * W))
            row = torch.zeros(S, dtype=F.dtype, device="cuda")
            row[ok] = C[l] @ torch.polar(torch.ones_like(th), th)
            out.append(row[None])
        return torch.cat(out)
    for l0 in range(1, L, step):
        l = torch.arange(l0, min(L, l0 + step), device="cuda")[:, None]
        num, den = xp[None] * Hp, 2 * l
        i0 = torch.div(num, den, rounding_mode="floor")
        fr = (num - i0 * den).double() / den.double()
        if interp == "linear":
            taps = [(0, 1.0 - fr), (1, fr)]
        else:                                              # Keys' kernel, a = -1/2
            near = lambda s: (1.5 * s - 2.5) * s * s + 1.0                # noqa: E731  |s| <= 1
            far = lambda s: ((-0.5 * s + 2.5) * s - 4.0) * s + 2.0        # noqa: E731  1 < |s| < 2
            taps = [(-1, far(1.0 + fr)), (0, near(fr)), (1, near(1.0 - fr)), (2, far(2.0 - fr))]
        acc = 0.0
        for d, w in taps:
            col = i0 + d + W // 2
            ok = (col >= 0) & (col < W)
            acc = acc + torch.gather(F[l0:l0 + l.shape[0]], 1, col.clamp(0, W - 1)) * (w * ok)
        out.append(acc)
    return torch.cat(out)


def _forward64(img, Hp, S, interp):
    """The transform of one image (float64, the transform's own frame)."""
    H, W = img.shape
    top = (Hp - H) // 2
    p = torch.nn.functional.pad(img, (0, 0, top, Hp - H - top))
    F = torch.fft.rfft(p, dim=0) * _parity(Hp // 2 + 1)[:, None]
    V = _interpolate(F, S, Hp, interp)
    m = torch.arange(S, device="cuda") - S // 2
    G = (S * torch.fft.ifft(V, dim=1))[:, m % S] * (1.0 - 2.0 * (m % 2).double())[None]
    return torch.fft.irfft(G * _parity(Hp // 2 + 1)[:, None], n=Hp, dim=0)


def exact(case, seed):
    """The maps (and loss and gradients) in 64 bits; peak records have no value
    here (their cells are whole numbers, and their values are cells of the map)."""
    st = prepare(case, seed)
    kind = case["kind"]
    if kind == "host":
        return None
    if kind == "mixed":
        b = st["batch"]
        out = torch.empty(b.map_total, dtype=torch.float64, device="cuda")
        for j, i in enumerate(b.order):
            h, w = b.shapes[i]
            o, q = int(b.img_off[j]), int(b.map_off[j])
            img = st["x"][o:o + h * w].view(h, w).double()
            out[q:q + h * w] = _forward64(img, h, w, case["interp"]).reshape(-1)
        return dict(map=out, count=None, cell=None, line=None)
    inv = case["space"] == "inverse"
    x = st["x"][-1] if kind == "stream" else st["x"]
    maps, grads, losses = [], [], []
    for i in range(x.shape[0]):
        img = x[i].detach().double()
        img.requires_grad_(kind in ("train", "layer"))
        P = _forward64(img.t() if inv else img, case["Hp"], case["S"], case["interp"])
        if kind == "train":
            loss = ((P.abs() * _loss_scale(case) - st["target"][i].double()) ** 2).mean()
            losses.append(loss.detach())
            grads.append(torch.autograd.grad(loss / x.shape[0], img)[0])
        elif kind == "layer":
            grads.append(torch.autograd.grad(P, img, st["g"][i].double())[0])
        maps.append(P.detach())
    r = dict(map=torch.stack(maps))
    if kind == "train":
        r.update(loss=torch.stack(losses), grad=torch.stack(grads))
    elif kind == "layer":
        r.update(grad=torch.stack(grads))
    elif kind in ("detect", "stream"):
        r.update(count=None, cell=None, line=None)
        if case.get("verify"):
            r.update(profile=None, length=None, verdict=None)
    return r
