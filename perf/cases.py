"""Performance cases of the DoG blob detector.

Each case is one pass of a call that users of this package make, through its
Python entry points (`Detector`, `DoGSoftHist`, `stretch`, `render_spheres`).
Inputs are synthetic frames drawn on the GPU from a seed: PLIF-shaped blob
fields as in `synth.plif_frame_u16`, blob frames as in
`synth.small_blob_frame`, and rendered spheres.

Kinds of case:
  detect   one frame through `Detector.detect` (a live camera frame)
  batch    many frames through `Detector.detect_batched` (frames of an
           acquisition, analysed together)
  soft     one training step of the sigma ladder: `DoGSoftHist` forward, a
           squared loss against a target histogram, and its gradients
  cube     `Detector.debug_dog`: the scale-normalised DoG cube of a frame
  stretch  contrast stretch of a 12-bit frame on its own
  render   evaluation frames of rendered spheres
The detector reports blobs in no particular order: `detect` puts them on a
map of the frame, `batch` sorts them on the device, as a program that tracks
or compares them does.
"""
import math
import random

import torch

from paper_2010_08486_gb300 import _lib, autotune, dog, synth

DEV = "cuda"
# ladders of this repository: (min_sigma, ratio, levels, threshold)
LADDERS = {
    "small": (1.0, 1.6, 6, 0.1),      # dog.small_frame_config
    "plif": (0.8, 1.1, 25, 0.05),     # dog.plif_config
    "spheres": (2.0, 1.15, 14, 0.05), # the sphere frames' ladder
    "grad": (1.0, 1.25, 12, 0.05),    # dog.grad_config
}
CAP = 8192     # blobs a frame may have
SAT = 0.0035   # contrast-stretch saturation of the paper


def listed():
    return [
        # the smallest call: one 256 x 256 frame, a handle as it comes
        dict(name="detect_small", kind="detect", h=256, w=256, dtype="f32", ladder="small"),
        # one camera frame at a time, latency-bound: PLIF frame at 25 scales,
        # the call captured once in a CUDA graph and replayed
        dict(name="detect_plif", kind="detect", h=1024, w=1024, dtype="u16", ladder="plif", tiled=True, graph=True),
        # a cropped region of interest: odd sizes, single precision
        dict(name="detect_ragged", kind="detect", h=701, w=933, dtype="f32", ladder="plif", tiled=True, graph=True),
        # few wide kernels, where the FFT backend is the right choice
        dict(name="detect_fft", kind="detect", h=1024, w=1024, dtype="u16", ladder="0.8:14:6", backend="fft",
             graph=True),
        # the headline workload: an acquisition of 12-bit frames at 25 scales
        dict(name="batch_plif", kind="batch", n=96, h=1024, w=1024, dtype="u16", ladder="plif"),
        # frames of several cameras and crops in one call, single precision
        dict(name="batch_uneven", kind="batch", n=64, h=0, w=0, dtype="f32", ladder="plif"),
        # the paper's evaluation frames, contrast stretched at ingest
        dict(name="batch_spheres", kind="batch", n=8, h=1000, w=1000, dtype="u16", ladder="spheres", sat=SAT),
        # one step of tuning the ladder on a batch of full frames
        dict(name="soft_train", kind="soft", n=16, h=1024, w=1024, ladder="grad"),
        # the same on two small crops of odd size
        dict(name="soft_crop", kind="soft", n=2, h=251, w=333, ladder="grad"),
        # the DoG cube of a crop, for plots and parity
        dict(name="cube", kind="cube", h=509, w=517, dtype="f32", ladder="plif"),
        # preprocessing on its own: limits and stretched frame
        dict(name="stretch", kind="stretch", h=1024, w=1280),
        # evaluation frames: eight renders of 100 spheres
        dict(name="render", kind="render", n=8, h=1000, w=1000, spheres=100),
    ]


def _size(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["detect", "detect", "batch", "batch", "soft", "cube", "stretch", "render"])
    h, w = _size(rng, 128, 1024), _size(rng, 128, 1280)
    # the repository's own ladders, or one of its sweep: sigma 0.8 to s_max in K levels
    ladder = rng.choice(["small", "plif", "spheres", "grad",
                         "0.8:%g:%d" % (rng.choice([2.0, 4.0, 8.0]), rng.choice([6, 12, 25]))])
    dtype = rng.choice(["u16", "f32"])
    sat = rng.choice([0.0, 0.0, SAT]) if dtype == "u16" else 0.0
    if kind == "detect":
        return dict(kind=kind, h=h, w=w, dtype=dtype, ladder=ladder, sat=sat, tiled=rng.random() < 0.7,
                    graph=rng.random() < 0.7, backend=rng.choice(["direct", "direct", "direct", "fft"]))
    if kind == "batch":
        if rng.random() < 0.3:
            return dict(kind=kind, n=_size(rng, 8, 128), h=0, w=0, dtype=dtype, ladder=ladder, sat=sat)
        return dict(kind=kind, n=max(2, min(_size(rng, 4, 256), 96 * 1024 * 1024 // (h * w))), h=h, w=w,
                    dtype=dtype, ladder=ladder, sat=sat)
    if kind == "soft":
        return dict(kind=kind, n=_size(rng, 1, 16), h=h, w=min(w, 1024), ladder=rng.choice(["grad", "grad", "small"]))
    if kind == "cube":
        return dict(kind=kind, h=h, w=w, dtype=dtype, ladder=ladder)
    if kind == "stretch":
        return dict(kind=kind, h=h, w=w)
    return dict(kind=kind, n=rng.randint(1, 8), h=h, w=w, spheres=rng.randint(20, 200))


# ------------------------------------------------------------------- inputs
def _ladder(case):
    name = case["ladder"]
    if name in LADDERS:
        return LADDERS[name]
    lo, hi, k = name.split(":")
    return float(lo), (float(hi) / float(lo)) ** (1.0 / (int(k) - 1)), int(k), 0.05


def _radii(case):
    s0, ratio, k, _ = _ladder(case)
    return [int(math.floor(4.0 * s0 * ratio ** i + 0.5)) for i in range(k)]


def _shapes(case, seed):
    if case["h"]:
        return [(case["h"], case["w"])] * case.get("n", 1)
    # frame sizes of several cameras, a third of them cropped to odd sizes;
    # the same for every seed, as a program's cameras are
    r = random.Random(case["n"])
    out = []
    for _ in range(case["n"]):
        h, w = r.choice(synth.BATCH_SIZES)
        out.append((h - r.randint(1, 40), w - r.randint(1, 40)) if r.random() < 1 / 3 else (h, w))
    return out


def _gen(seed):
    return torch.Generator(DEV).manual_seed(int(seed))


def _uniform(g, lo, hi, n):
    return lo + (hi - lo) * torch.rand(n, generator=g, device=DEV)


def _blobs(img, cx, cy, s, amp):
    ys = torch.arange(img.shape[0], device=DEV, dtype=torch.float32)[None] - cy[:, None]
    xs = torch.arange(img.shape[1], device=DEV, dtype=torch.float32)[None] - cx[:, None]
    q = (-0.5 / (s * s))[:, None]
    img += (torch.exp(ys * ys * q) * amp[:, None]).t() @ torch.exp(xs * xs * q)


def _frame(g, h, w, kind):
    """One frame: 12-bit counts as int16 ("u16"), counts / 4095 ("f32") or a
    small blob frame with Gaussian noise ("small")."""
    img = torch.zeros((h, w), device=DEV)
    if kind == "small":
        n = 20 * max(1, h * w // 65536)
        _blobs(img, _uniform(g, 0, w, n), _uniform(g, 0, h, n), _uniform(g, 1, 8, n), _uniform(g, 0.3, 1, n))
        return (img + 0.02 * torch.randn((h, w), generator=g, device=DEV)).clamp(0, 1)
    n = max(1, synth.plif_blob_count(h, w))
    cx, cy, amp = _uniform(g, 0, w, n), _uniform(g, 0, h, n), _uniform(g, 0.3, 1, n)
    s = torch.exp(math.log(3.0) + 0.5 * torch.randn(n, generator=g, device=DEV)).clamp(0.8, 20)
    ys = torch.arange(h, device=DEV, dtype=torch.float32)[:, None] - h / 2
    xs = torch.arange(w, device=DEV, dtype=torch.float32)[None] - w / 2
    img += 0.25 * torch.exp(-(ys * ys) / (2 * 300.0 ** 2)) * torch.exp(-(xs * xs) / (2 * 120.0 ** 2))
    _blobs(img, cx, cy, s, amp)
    counts = torch.poisson(4095.0 * img.clamp(0, 1), generator=g).clamp(max=4095.0)
    return counts.to(torch.int16) if kind == "u16" else counts / 4095.0


def _frames(case, seed):
    g = _gen(seed)
    kind = "small" if case.get("ladder") == "small" and case.get("dtype") == "f32" else case.get("dtype", "f32")
    return [_frame(g, h, w, kind) for h, w in _shapes(case, seed)]


def _spheres(case, seed, f):
    return torch.from_numpy(synth.sphere_table(seed * 1000 + f, n=case["spheres"], h=case["h"], w=case["w"],
                                               r_range=(4.0, 16.0))).to(DEV)


def _detector(case, shapes, cap):
    s0, ratio, k, thr = _ladder(case)
    return dog.Detector(dog.DetectorConfig(
        min_sigma=s0, ratio=ratio, n_levels=k, threshold=thr, max_h=max(h for h, _ in shapes),
        max_w=max(w for _, w in shapes), blob_cap=cap, stretch_sat=case.get("sat", 0.0),
        backend=_lib.BACKEND_FFT if case.get("backend") == "fft" else _lib.BACKEND_DIRECT))


def _tile(det, shape):
    """Row bands as the tuner's model ranks them first (no timing)."""
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    det.set_tiling(autotune.candidate_bands([shape], det.radii, n_sm)[0])


def prepare(case, seed):
    kind = case["kind"]
    st = {"kind": kind, "case": case, "seed": seed}
    if kind == "render":
        st["spheres"] = [_spheres(case, seed, f) for f in range(case["n"])]
        return st
    if kind == "stretch":
        st["img"] = _frame(_gen(seed), case["h"], case["w"], "u16")
        return st
    st["frames"] = frames = _frames(case, seed)
    shapes = [tuple(f.shape) for f in frames]
    if kind == "detect":
        st["det"] = det = _detector(case, shapes, CAP)
        if case.get("tiled"):
            _tile(det, shapes[0])
        st["out"] = dog.BlobList(torch.zeros((CAP, 5), dtype=torch.int32, device=DEV),
                                 torch.zeros((), dtype=torch.int32, device=DEV))
        st["hist"] = torch.zeros(det.nbins_out, dtype=torch.int32, device=DEV)
        st["slots"] = torch.arange(CAP, device=DEV)
        if case.get("graph"):
            side = torch.cuda.Stream()
            side.wait_stream(torch.cuda.current_stream())
            with torch.cuda.stream(side):
                _detect(st)
            torch.cuda.current_stream().wait_stream(side)
            st["graph"] = torch.cuda.CUDAGraph()
            with torch.cuda.graph(st["graph"]):
                st["got"] = _detect(st)
    elif kind == "batch":
        st["det"] = det = _detector(case, shapes, CAP)
        st["table"] = det.frame_table(frames, CAP)
        st["out"] = torch.zeros((len(frames) * CAP, 5), dtype=torch.int32, device=DEV)
        st["counts"] = torch.zeros(len(frames), dtype=torch.int32, device=DEV)
        st["hists"] = torch.zeros((len(frames), det.nbins_out), dtype=torch.int32, device=DEV)
    elif kind == "cube":
        st["det"] = _detector(case, shapes, CAP)
        _tile(st["det"], shapes[0])
    else:
        st["frames"] = torch.stack(frames).requires_grad_(True)
        st["det"] = det = _detector(case, shapes, CAP)
        _tile(det, shapes[0])
        st["sigmas"], st["target"] = _training(case, seed)
        st["sigmas"].requires_grad_(True)
    return st


def _training(case, seed):
    """A ladder in the middle of its tuning and the histogram it is tuned to."""
    s0, ratio, k, _ = _ladder(case)
    g = _gen(seed + 77)
    sig = torch.tensor([s0 * ratio ** i for i in range(k)], device=DEV) * _uniform(g, 0.98, 1.02, k)
    return sig.float(), _uniform(g, 0.0, 200.0, 32) * case["n"] * case["h"] * case["w"] / 2 ** 20


# --------------------------------------------------------------------- runs
def _sorted_blobs(out, counts):
    """Every frame's slots as (x, y, level) and (sigma, response), ordered by
    (level, y, x); slots past a frame's count are 0."""
    b = out.view(counts.shape[0], -1, 5)
    used = torch.arange(b.shape[1], device=out.device)[None] < counts[:, None]
    key = torch.where(used, (b[..., 2] << 22 | b[..., 1] << 11 | b[..., 0]), 2 ** 31 - 1)
    order = key.sort(dim=1).indices
    b = torch.where(used[..., None], b.gather(1, order[..., None].expand(-1, -1, 5)), 0)
    return b[..., :3], b[..., 3:].contiguous().view(torch.float32)


def _detect(state):
    """Detection of the state's frame; the blobs as a map of the frame: the
    record of the blob centred at a pixel, zeros elsewhere (two blobs never
    share a centre: concentric discs overlap and are coalesced)."""
    h, w = state["frames"][0].shape
    blobs, hist, _ = state["det"].detect(state["frames"][0], out=state["out"], hist=state["hist"])
    at = torch.add(blobs.raw[:, 0], blobs.raw[:, 1], alpha=w)
    at = torch.where(state["slots"] < blobs.count, at, h * w).long()
    m = torch.zeros((h * w + 1, 5), dtype=torch.int32, device=DEV).index_copy_(0, at, blobs.raw)[:h * w]
    return {"where": m[:, :3], "size": m.view(torch.float32)[:, 3:], "count": blobs.count, "hist": hist}


def run(state):
    kind = state["kind"]
    if kind == "detect":
        if "graph" in state:
            state["graph"].replay()
            return state["got"]
        return _detect(state)
    if kind == "batch":
        out, counts, hists = state["det"].detect_batched(None, table=state["table"], out=state["out"],
                                                         counts=state["counts"], hists=state["hists"])
        where, size = _sorted_blobs(out, counts)
        return {"where": where, "size": size, "counts": counts, "hists": hists}
    if kind == "soft":
        hist = dog.DoGSoftHist.apply(state["frames"], state["sigmas"], state["det"])
        loss = ((hist - state["target"]) ** 2).sum()
        g_frames, g_sigmas = torch.autograd.grad(loss, (state["frames"], state["sigmas"]))
        return {"hist": hist.detach(), "g_frames": g_frames, "g_sigmas": g_sigmas}
    if kind == "cube":
        return {"cube": state["det"].debug_dog(state["frames"][0])}
    if kind == "stretch":
        lohi = dog.stretch_limits(state["img"], SAT)
        return {"lohi": lohi, "frame": dog.stretch(state["img"], lohi)}
    got = [dog.render_spheres(s, state["case"]["h"], state["case"]["w"], seed=state["seed"] * 1000 + f,
                              with_intensity=True) for f, s in enumerate(state["spheres"])]
    return {"counts": [c for c, _ in got], "intensity": [i for _, i in got]}


# --------------------------------------------------------------------- work
def work(case):
    kind = case["kind"]
    shapes = _shapes(case, 0)
    px = sum(h * w for h, w in shapes)
    src = 2 if case.get("dtype") == "u16" else 4
    if kind == "render":
        # each sphere's disc (mean area of R in U[4, 16], frame edges aside) is sampled 16 times a pixel
        disc = math.pi * (16.0 ** 3 - 4.0 ** 3) / (3 * 12.0)
        return {"bytes": px * 6, "flops": case["n"] * case["spheres"] * disc * 16 * 8 + px * 100}
    if kind == "stretch":
        return {"bytes": px * 6, "flops": px * 4}
    taps = sum(2 * r + 1 for r in _radii(case))
    k = len(_radii(case))
    blur = 4.0 * taps * px          # separable passes of every level, 2 flop a tap
    test = 6.0 * (k - 1) * px       # differences, scaling, separable 3x3x3 maximum
    if kind == "cube":
        return {"bytes": px * (src + 4 * (k - 1)), "flops": blur + 2.0 * (k - 1) * px}
    if kind == "soft":
        # forward, and the adjoint blur of every level; frames read twice, gradients written
        return {"bytes": px * 12, "flops": 2 * blur + test}
    if case.get("backend") == "fft":
        n = sum((h + 2 * max(_radii(case))) * (w + 2 * max(_radii(case))) for h, w in shapes)
        return {"bytes": px * src, "flops": 2.5 * n * math.log2(n) * (k + 1) + 2.0 * n * k + test}
    return {"bytes": px * src, "flops": blur + test}


# -------------------------------------------------------------------- exact
def _reflect(n, r):
    i = torch.arange(-r, n + r, device=DEV) % (2 * n)
    return torch.where(i >= n, 2 * n - 1 - i, i)


def _blur64(img, sigma, r):
    """Separable Gaussian with half-sample symmetric reflection, 64 bits; img (..., H, W)."""
    j = torch.arange(-r, r + 1, device=DEV, dtype=torch.float64)
    w = torch.exp(-j * j / (2 * sigma * sigma))
    w = w / w.sum()
    for dim in (-1, -2):
        n = img.shape[dim]
        x = img.index_select(dim, _reflect(n, r))
        img = sum(w[t] * x.narrow(dim, t, n) for t in range(2 * r + 1))
    return img


def _cube64(img, sigmas, radii):
    """The DoG cube (P, H, W) with the finite-difference normalisation."""
    levels = [_blur64(img, s, r) for s, r in zip(sigmas, radii)]
    return torch.stack([s / (t - s) * (a - b)
                        for a, b, s, t in zip(levels, levels[1:], sigmas, sigmas[1:])])


def _soft64(case, seed):
    s0, ratio, k, thr = _ladder(case)
    frames, radii, nbins, temp = _frames(case, seed), _radii(case), 32, 0.01
    sig, target = _training(case, seed)
    sig = sig.double().requires_grad_(True)
    lo, hi = math.log(s0), math.log(s0 * ratio ** (k - 2))
    bins = torch.arange(nbins, device=DEV, dtype=torch.float64) + 0.5

    def hist(img):
        cube = _cube64(img, list(sig), radii)
        d = cube.detach()[None, None]
        mask = torch.nn.functional.max_pool3d(d, 3, 1, 1)[0, 0] == d[0, 0]
        t = ((torch.log(sig[:-1]) - lo) / (hi - lo)).clamp(0.5 / nbins, 1 - 0.5 / nbins)
        kappa = (1 - (nbins * t[:, None] - bins[None]).abs()).clamp(min=0)
        s = torch.stack([torch.sigmoid((cube[p][mask[p]] - thr) / temp).sum() for p in range(k - 1)])
        return s @ kappa

    imgs = [f.double().requires_grad_(True) for f in frames]
    with torch.no_grad():
        total = sum(hist(i) for i in imgs)
    g_hist = 2 * (total - target.double())
    g_sig, g_frames = torch.zeros_like(sig), []
    for i in imgs:   # one frame's graph at a time
        a, b = torch.autograd.grad((hist(i) * g_hist).sum(), (i, sig))
        g_frames.append(a)
        g_sig += b
    return {"hist": total, "g_frames": torch.stack(g_frames), "g_sigmas": g_sig}


def _intensity64(sph, h, w, ss=4, bg=0.05):
    off = (2 * torch.arange(ss, device=DEV, dtype=torch.float64) + 1) / (2 * ss) - 0.5
    ys = (torch.arange(h, device=DEV, dtype=torch.float64)[:, None] + off).reshape(-1)
    xs = (torch.arange(w, device=DEV, dtype=torch.float64)[:, None] + off).reshape(-1)
    img = torch.full((h, w), bg, device=DEV, dtype=torch.float64)
    for cx, cy, r, a in sph.double().cpu().tolist():
        y0, y1 = max(0, int(cy - r) - 2), min(h, int(cy + r) + 3)
        x0, x1 = max(0, int(cx - r) - 2), min(w, int(cx + r) + 3)
        dy, dx = ys[y0 * ss:y1 * ss] - cy, xs[x0 * ss:x1 * ss] - cx
        q = (1 - (dx[None] ** 2 + dy[:, None] ** 2) / (r * r)).clamp(min=0).sqrt()
        img[y0:y1, x0:x1] += a * q.reshape(y1 - y0, ss, x1 - x0, ss).mean(dim=(1, 3))
    return img


def exact(case, seed):
    kind = case["kind"]
    if kind == "cube":
        s0, ratio, k, _ = _ladder(case)
        img = _frames(case, seed)[0].double()
        img = img / 4095.0 if case["dtype"] == "u16" else img
        return {"cube": _cube64(img, [s0 * ratio ** i for i in range(k)], _radii(case))}
    if kind == "soft":
        return _soft64(case, seed)
    if kind == "stretch":
        img = _frame(_gen(seed), case["h"], case["w"], "u16").double()
        n = img.numel()
        k = min(int(math.floor(SAT / 2 * n)), (n - 1) // 2)
        v = img.reshape(-1).sort().values
        lo, hi = v[k], v[n - 1 - k]
        return {"lohi": None, "frame": ((img - lo) / (hi - lo)).clamp(0, 1)}
    if kind == "render":
        return {"counts": None, "intensity": [_intensity64(_spheres(case, seed, f), case["h"], case["w"])
                                              for f in range(case["n"])]}
    # a detection's sigmas and responses belong to maxima that single precision
    # decides: near ties the list in 64 bits is another list
    return None
