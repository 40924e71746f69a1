"""Child process of tests/test_gpu_debug_wide.py: loads the bounds-checked build
(FT_DEBUG=1 before the binding is imported) and runs the kernels of the wide radices
(12, 18, 24 and 36 samples per thread) with ragged tile bands, the fused loss and its
adjoint, the three peak passes, the chirp-z rows and the grouped mixed-size kernels;
compares with the generic kernels of the same build and the oracle's peak list, and
prints OK when every result matches and no device index check fired."""
import os
import sys

import numpy as np

os.environ["FT_DEBUG"] = "1"
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import torch                                            # noqa: E402

import oracle                                           # noqa: E402
from paper_1904_09409_gb300 import funnel as f          # noqa: E402

assert f.LIB_PATH.endswith("libfunnel_debug.so"), f.LIB_PATH
assert f.ft_debug_build()
assert f.ft_debug_flags() == 0

rng = np.random.default_rng(17)
bad, flags = [], 0


def rel(a, b):
    return float((a.double() - b.double()).norm() / b.double().norm())


def gpu(*shape):
    return torch.from_numpy(rng.standard_normal(shape).astype(np.float32)).cuda()


def results(plan, x, g, t):
    m, gi = torch.empty_like(g), torch.empty_like(x)
    f.ft_forward(plan, x, m)
    f.ft_backward(plan, g, gi)
    loss, gl = f.ft_abs_mse_backward(plan, g, t, 0.5)
    torch.cuda.synchronize()
    return m, gi, loss, gl


# (H, W, S, H', interp): E = 18 with a ragged last band, 18 / 12, 24 and 36, the
# shortest lengths, register-resident chirp-z rows (the last block partly empty)
CASES = [(150, 96, 108, 162, "linear"), (470, 320, 324, 486, "cubic"), (1000, 200, 216, 1152, "linear"),
         (300, 60, 64, 3888, "cubic"), (150, 570, 576, 162, "linear"), (90, 2590, 2592, 96, "linear"),
         (70, 72, 72, 72, "linear"), (96, 486, 486, 96, "fourier"), (97, 128, 128, 128, "fourier"),
         (64, 576, 576, 64, "fourier")]
for H, W, S, Hp, interp in CASES:
    x, g, t = gpu(3, H, W), gpu(3, Hp, S), gpu(3, Hp, S)
    lists = {}
    for mode in ("multi", "sparse", "dense"):
        os.environ["FT_PEAKS"] = mode
        with f.Plan(H, W, S, Hp, interp) as plan:
            m = torch.empty_like(g)
            for _ in range(2):
                out, cnt = f.ft_detect(plan, x, m, 20)
            torch.cuda.synchronize()
            lists[mode] = [(int(p["t"]), int(p["s"])) for p in f.peaks_to_numpy(out, cnt, 20)[1]]
            if mode == "multi":
                fast = results(plan, x, g, t)
                f.ft_plan_set_variant(plan, 1)
                slow = results(plan, x, g, t)
                err = [rel(a, b) for a, b in zip(fast, slow)]
                if not max(err) <= 2e-6:
                    bad.append((H, W, S, Hp, interp, err))
    want = [(a, b) for a, b, _ in oracle.peaks_ref(np.abs(fast[0][1].cpu().numpy()).astype(np.float64), 20)]
    if any(v != want for v in lists.values()):
        bad.append((H, W, S, Hp, interp, lists, want))
    now = f.ft_debug_flags()
    flags |= now
    print((H, W, S, Hp, interp), "flags", now, "errors", err)

shapes = [(128, 192), (1536, 128), (192, 384), (256, 256)]
os.environ.pop("FT_PEAKS")
with f.Batch(shapes) as b:
    imgs = [rng.standard_normal(s).astype(np.float32) for s in shapes]
    xb = torch.from_numpy(b.pack(imgs)).cuda()
    for c2r in (256, 512):
        b.set_config(512, 128, c2r)
        mb = torch.zeros(b.map_total, device="cuda")
        out = torch.empty(b.n * 8 * f.PEAK_DTYPE.itemsize, dtype=torch.uint8, device="cuda")
        cnt = torch.empty(b.n, dtype=torch.int32, device="cuda")
        b.run(xb, mb, 8, out=out, count=cnt)
        torch.cuda.synchronize()
        for (H, W), img, m in zip(shapes, imgs, b.unpack_maps(mb.cpu().numpy())):
            with f.Plan(H, W, W, H) as plan:
                ref = torch.empty((1, H, W), device="cuda")
                f.ft_forward(plan, torch.from_numpy(img[None]).cuda(), ref)
                torch.cuda.synchronize()
                e = rel(torch.from_numpy(m), ref[0].cpu())
                if not e <= 2e-6:
                    bad.append(("batch", H, W, c2r, e))
now = f.ft_debug_flags()
flags |= now
print("batch flags", now)
print("flags", flags, "mismatches", bad)
print("OK" if flags == 0 and not bad else "FAIL")
