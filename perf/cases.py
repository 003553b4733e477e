"""The work whose speed this library is measured by, one case per way of using it.

A case is a dict of plain values: what kind of call it is, the volume (X, Y, Z), the
views and their PSFs, and the options. ``listed()`` gives the named ones, ``draw``
more of the same ranges; ``prepare`` builds what a program holds before the call,
``run`` makes the call once, ``work`` says what it cannot do without, and ``exact``
computes its outputs with plain torch in 64 bits.

Inputs are synthetic light-sheet data made on the device: small soft objects of random
place and intensity, blurred periodically with each view's Gaussian PSF, Poisson noise.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1308_0730_gb300 import autograd, mvd

# light-sheet PSFs: lateral and axial sigma, and the box (Kx, Ky, Kz) of the unrotated view
SPIM = dict(sxy=1.2, sax=4.0, bx=15, by=15, bz=41)
SPIM_LARGE = dict(sxy=1.5, sax=5.0, bx=19, by=19, bz=51)


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------

def _iterate(name, dims, views, iters, psf, **more):
    c = {"name": name, "kind": "iterate", "X": dims[0], "Y": dims[1], "Z": dims[2], "views": views, "iters": iters,
         "layout": "spim", "precision": "precise", "boundary": "periodic", "lam": 0.0, "weights": False,
         "combined": False, "background": 0.0, "peak": 100.0}
    c.update(psf)
    c.update(more)
    return c


def listed():
    small = dict(sxy=1.0, sax=2.5, bx=7, by=7, bz=13)
    return [
        # an acquisition loop that may not allocate: one pass over three views of a small
        # region of interest, launch latency and little work
        dict(_iterate("noalloc-32", (32, 32, 32), 3, 1, small, layout="axes", background=1.0), kind="noalloc"),
        # the small volume of the tests and the smoke run: 10 iterations, direct engine
        _iterate("blobs-32", (32, 32, 32), 3, 10, small, layout="axes", background=1.0),
        # a cropped region whose lengths are not {2,3,5}-smooth: only the direct engine takes it
        _iterate("odd-97x83x61", (97, 83, 61), 2, 1, dict(sxy=1.2, sax=2.5, bx=9, by=9, bz=15), background=1.0),
        # the four-view volume of the benchmark (power-of-two lengths), default precision
        _iterate("mid-256x256x128", (256, 256, 128), 4, 2, SPIM),
        # the large specimen's grid and PSFs, two of its views
        _iterate("specimen-1024x1024x512", (1024, 1024, 512), 2, 1, SPIM_LARGE, background=5.0, peak=200.0),
        # mixed-radix lengths: one volume of the benchmark's batch
        _iterate("smooth-300x180x150", (300, 180, 150), 3, 1, SPIM, background=1.0, peak=150.0),
        # many independent volumes of uneven size advanced by one graph launch
        dict(_iterate("batch-6", (120, 100, 72), 3, 2, SPIM, background=1.0), kind="batch", volumes=6),
        # the camera sees nothing outside the grid, with the paper's usual lambda: a padded grid
        _iterate("zero-256x256x128", (256, 256, 128), 2, 1, SPIM, boundary="zero", lam=0.006, background=1.0),
        # all-FP32 arithmetic, partially overlapping views
        _iterate("fast-256x256x128", (256, 256, 128), 4, 2, SPIM, precision="fast", weights=True, background=1.0),
        # the kernels of a new set of seven PSFs (set-up of an experiment)
        dict(_iterate("kernels-7views", (96, 64, 96), 7, 1, SPIM_LARGE, background=1.0), kind="kernels",
             variant="efficient"),
        # one PSF-calibration step: unrolled iterations and their gradient
        dict(_iterate("grad-128x128x96", (128, 128, 96), 4, 8, SPIM, background=1.0), kind="grad"),
        # the next time point of a recording: views from pinned host memory, result to the host
        dict(_iterate("series-256x256x128", (256, 256, 128), 4, 5, SPIM, background=1.0), kind="series"),
    ]


def _smooth(n):
    """The nearest {2,3,5}-smooth integer."""
    for d in range(n):
        for m in (n - d, n + d):
            k = m
            for p in (2, 3, 5):
                while k % p == 0:
                    k //= p
            if m >= 8 and k == 1:
                return m
    return 8


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: sizes over the whole range of each kind, odd ones among them."""
    kind = rng.choice(["noalloc", "direct", "odd", "pow2", "pow2", "large", "smooth", "smooth", "batch", "bounded",
                       "fast", "kernels", "grad", "series"])
    sxy, sax = rng.uniform(0.9, 1.5), rng.uniform(2.5, 5.0)
    more = dict(background=rng.choice([1.0, 2.0, 5.0]), peak=round(rng.uniform(50, 300), 1))
    spim = dict(sxy=round(sxy, 3), sax=round(sax, 3), bx=15, by=15, bz=rng.choice([31, 41]))

    def box(kz):
        return dict(sxy=round(sxy, 3), sax=round(0.6 * sax, 3), bx=rng.choice([5, 7, 9]), by=rng.choice([5, 7, 9]),
                    bz=rng.choice(kz))

    if kind in ("noalloc", "direct"):
        dims = [_log(rng, 20, 72) for _ in range(3)]
        c = _iterate("", dims, rng.randint(1, 3), rng.randint(1, 6) if kind == "direct" else 1, box([9, 11, 13]),
                     layout="axes", **more)
        return _unnamed(dict(c, kind="noalloc") if kind == "noalloc" else c)
    if kind == "odd":
        dims = [_log(rng, 40, 180) for _ in range(3)]
        dims[rng.randrange(3)] = rng.choice([47, 59, 67, 71, 89, 97, 113, 131])
        return _unnamed(_iterate("", dims, rng.randint(1, 3), 1, box([9, 13, 17]), **more))
    pow2 = [rng.choice([64, 128, 256, 512]), rng.choice([64, 128, 256, 512]), rng.choice([64, 128, 256])]
    smooth = [_smooth(_log(rng, 48, 320)), _smooth(_log(rng, 48, 320)), _smooth(_log(rng, 48, 192))]
    if kind == "pow2":
        return _unnamed(_iterate("", pow2, rng.randint(2, 6), rng.randint(1, 4), spim,
                                 precision=rng.choice(["precise", "precise", "mixed"]),
                                 combined=rng.random() < 0.25, **more))
    if kind == "large":
        return _unnamed(_iterate("", (1024, 512, rng.choice([128, 256, 512])), rng.randint(1, 2), 1, SPIM_LARGE, **more))
    if kind == "smooth":
        return _unnamed(_iterate("", smooth, rng.randint(2, 6), rng.randint(1, 3), spim, weights=rng.random() < 0.3,
                                 lam=rng.choice([0.0, 0.0, 0.006]), **more))
    if kind == "batch":
        dims = [_smooth(_log(rng, 60, 160)) for _ in range(3)]
        return _unnamed(dict(_iterate("", dims, rng.randint(2, 4), rng.randint(1, 3), spim, **more), kind="batch",
                             volumes=rng.randint(3, 8)))
    if kind == "bounded":
        dims = [_log(rng, 60, 256), _log(rng, 60, 256), _log(rng, 60, 128)]
        return _unnamed(_iterate("", dims, rng.randint(2, 4), rng.randint(1, 2), spim,
                                 boundary=rng.choice(["zero", "mirror"]), lam=rng.choice([0.0, 0.006]), **more))
    if kind == "fast":
        return _unnamed(_iterate("", rng.choice([pow2, smooth]), rng.randint(2, 6), rng.randint(1, 3), spim,
                                 precision="fast", **more))
    if kind == "kernels":
        b = dict(spim, bx=rng.choice([11, 15, 19]), bz=rng.choice([31, 41, 51]))
        b["by"] = b["bx"]
        return _unnamed(dict(_iterate("", (72, 60, 64), rng.randint(2, 7), 1, b, **more), kind="kernels",
                             variant=rng.choice(["efficient", "opt1"])))
    if kind == "grad":
        dims = [_smooth(_log(rng, 48, 128)) for _ in range(3)]
        return _unnamed(dict(_iterate("", dims, rng.randint(2, 4), rng.randint(2, 6), spim, **more), kind="grad"))
    dims = rng.choice([[256, 256, 64], [_smooth(_log(rng, 96, 256)), _smooth(_log(rng, 96, 256)), 96]])
    return _unnamed(dict(_iterate("", dims, rng.randint(2, 4), rng.randint(2, 10), spim, **more), kind="series"))


def _unnamed(c):
    return {k: v for k, v in c.items() if k != "name"}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _psf(sxy, sax, box, angle, axis):
    """Gaussian PSF sampled on the odd bounding box of ``box`` rotated about y; float32 [Kz][Ky][Kx]."""
    t = math.radians(angle)
    R = np.array([[math.cos(t), 0.0, math.sin(t)], [0.0, 1.0, 0.0], [-math.sin(t), 0.0, math.cos(t)]])
    half = np.abs(R) @ np.array([(b - 1) / 2 for b in box])
    K = [int(2 * math.floor(h + 1e-9) + 1) for h in half]
    var = [sxy ** 2] * 3
    var["xyz".index(axis)] = sax ** 2
    Si = np.linalg.inv(R @ np.diag(var) @ R.T)
    z, y, x = np.meshgrid(*[np.arange(k) - (k - 1) / 2 for k in reversed(K)], indexing="ij")
    d = np.stack([x, y, z], -1)
    p = np.exp(-0.5 * np.einsum("...i,ij,...j->...", d, Si, d))
    return (p / p.sum()).astype(np.float32)


def _psfs(c):
    box, out = (c["bx"], c["by"], c["bz"]), []
    for v in range(c["views"]):
        if c["layout"] == "axes":  # elongated along x, y, z in turn
            a = (2 - v) % 3
            b = [box[0], box[1]]
            b.insert(a, box[2])
            out.append(_psf(c["sxy"], c["sax"], b, 0.0, "xyz"[a]))
        else:  # rotated about y, as a sample rotated in the light sheet
            out.append(_psf(c["sxy"], c["sax"], box, v * 360.0 / c["views"], "z"))
    # a rotated box may not exceed the volume: trim it symmetrically
    dims = (c["Z"], c["Y"], c["X"])
    trimmed = []
    for p in out:
        cut = [slice((k - min(k, (n - 1) | 1 if n % 2 else n - 1)) // 2, None) for k, n in zip(p.shape, dims)]
        p = p[tuple(slice(s.start, p.shape[i] - s.start) for i, s in enumerate(cut))]
        trimmed.append(np.ascontiguousarray(p / p.sum(dtype=np.float64), dtype=np.float32))
    return trimmed


def _measured(c, seed):
    """A set of kernels is built for measured PSFs: their widths differ from one experiment to the next."""
    if c["kind"] != "kernels":
        return c
    f = np.random.default_rng(int(seed)).uniform(0.9, 1.1, 2)
    return dict(c, sxy=c["sxy"] * f[0], sax=c["sax"] * f[1])


def _spectrum(p, shape, dtype, device):
    """rfftn of a centred kernel placed on the periodic grid ``shape``."""
    if not isinstance(p, torch.Tensor):
        p = torch.from_numpy(np.asarray(p)).to(device)
    p = p.to(dtype)
    big = torch.zeros(shape, dtype=dtype, device=device)
    big = _insert(big, p)
    return torch.fft.rfftn(big)


def _insert(big, p):
    full = torch.nn.functional.pad(p, [q for k, n in zip(reversed(p.shape), reversed(big.shape)) for q in (0, n - k)])
    return big + torch.roll(full, [-(k // 2) for k in p.shape], dims=(0, 1, 2))


def _volumes(c, psfs, seed):
    """Views on the device: sparse soft objects, each view's periodic blur, Poisson counts."""
    dev = torch.device("cuda")
    g = torch.Generator(device=dev)
    g.manual_seed(int(seed) * 7919 + 17)
    shape = (c["Z"], c["Y"], c["X"])
    u = torch.rand(shape, generator=g, device=dev)
    density = 3000.0 / (256 * 256 * 128) * (8 if u.numel() < 1 << 18 else 1)
    obj = torch.where(u < density, 0.5 + 0.5 * u / density, torch.zeros_like(u))
    del u
    k = min(17, *[(n - 1) | 1 if n % 2 else n - 1 for n in shape])
    r = np.arange(k) - k // 2
    ball = np.exp(-0.5 * (r[:, None, None] ** 2 + r[None, :, None] ** 2 + r[None, None, :] ** 2) / 2.2 ** 2)
    f = torch.fft.rfftn(obj) * _spectrum(ball.astype(np.float32), shape, torch.float32, dev)
    del obj
    views = [torch.fft.irfftn(f * _spectrum(p, shape, torch.float32, dev), s=shape).clamp_(min=0) for p in psfs]
    del f
    scale = c["peak"] / max(float(v.max()) for v in views)
    for i in range(len(views)):
        lam = views[i] * scale + c["background"]
        views[i] = None
        views[i] = torch.poisson(lam, generator=g).contiguous()
        del lam
    return views


def _weights(c):
    """Blending images: view v covers 70% of the volume along x, with cosine borders."""
    out = []
    for v in range(c["views"]):
        n = c["X"]
        lo = int(0.3 * n * v / max(1, c["views"] - 1))
        i = np.arange(n)
        d = np.minimum(i - lo, lo + int(0.7 * n) - 1 - i).astype(np.float64)
        w = np.where(d < 0, 0.0, np.where(d < 8, 0.5 * (1 - np.cos(np.pi * (d + 1) / 9)), 1.0)).astype(np.float32)
        out.append(torch.from_numpy(w).cuda().expand(c["Z"], c["Y"], n).contiguous())
    return out


def _parts(c):
    """The cases of a batch's volumes: sizes from 0.6 to 1.4 of the batch's, each smooth."""
    out = []
    for i in range(c["volumes"]):
        f = [0.6 + 0.8 * ((i * s + o) % c["volumes"]) / max(1, c["volumes"] - 1) for s, o in ((1, 0), (5, 1), (7, 2))]
        out.append(dict(c, kind="iterate", X=_smooth(int(c["X"] * f[0])), Y=_smooth(int(c["Y"] * f[1])),
                        Z=_smooth(int(c["Z"] * f[2])), views=2 + (c["views"] + i) % 3))
    return out


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

class _Borrowed:
    """The library's device buffer of the estimate, for torch.as_tensor; the tensor keeps this object, and
    with it the buffer's owner, alive."""

    def __init__(self, ptr, shape, owner):
        self.owner = owner
        self.__cuda_array_interface__ = {"shape": tuple(shape), "typestr": "<f4", "data": (ptr, False), "version": 2,
                                         "strides": None}


def _estimate(d, owner=None):
    t = torch.as_tensor(_Borrowed(mvd.mvd_result_device(d.ctx), d.shape, owner or d), device="cuda")
    t.owner = owner or d
    return t


class _Batch:
    def __init__(self, volumes, iters):
        self.volumes = volumes
        self.handle = mvd.mvd_batch_create([d.ctx for d in volumes], iters)

    def __del__(self):
        mvd.mvd_batch_destroy(self.handle)
        for d in self.volumes:
            d.close()


def _deconvolver(c, seed, stream):
    psfs = _psfs(c)
    views = _volumes(c, psfs, seed)
    torch.cuda.current_stream().synchronize()  # the library works on its own stream
    d = mvd.Deconvolver(views, psfs, "efficient", stream=stream, precision=c["precision"], boundary=c["boundary"])
    if c["lam"]:
        d.set_regularization(c["lam"])
    if c["weights"]:
        w = _weights(c)
        torch.cuda.current_stream().synchronize()
        d.set_weights(w, "min_overlap")
    d.synchronize()
    return d


def prepare(case, seed):
    c = dict(case)
    s = {"c": c, "stream": torch.cuda.Stream()}
    if c["kind"] in ("iterate", "kernels"):
        s["d"] = _deconvolver(_measured(c, seed), seed, s["stream"])
    elif c["kind"] == "batch":
        parts = [_deconvolver(p, seed * 31 + i, s["stream"]) for i, p in enumerate(_parts(c))]
        s["batch"] = _Batch(parts, c["iters"])
    elif c["kind"] == "series":
        psfs = _psfs(c)
        views = _volumes(c, psfs, seed)
        torch.cuda.current_stream().synchronize()
        s["d"] = mvd.Deconvolver(views, psfs, "efficient", stream=s["stream"], precision=c["precision"])
        s["pinned"] = [v.cpu().pin_memory() for v in views]
        s["views"] = [v.numpy() for v in s["pinned"]]
        s["out_t"] = torch.empty((c["Z"], c["Y"], c["X"]), dtype=torch.float32).pin_memory()
        s["out"] = s["out_t"].numpy()
    elif c["kind"] == "noalloc":
        psfs = _psfs(c)
        s["views"] = _volumes(c, psfs, seed)
        s["flat"] = float(np.float32(np.mean([float(v.double().mean()) for v in s["views"]])))
        comp = [k.to(torch.float32).cuda().contiguous() for k in _compound([torch.from_numpy(p).double() for p in psfs])]
        s["psfs"] = [torch.from_numpy(p).cuda() for p in psfs]
        s["comp"], s["psi"] = comp, torch.empty_like(s["views"][0])
    else:  # grad
        psfs = _psfs(c)
        v = torch.stack(_volumes(c, psfs, seed))
        s["target"] = v.mean(0)
        s["views"] = v.requires_grad_()
        s["psfs"] = [torch.from_numpy(p).requires_grad_() for p in psfs]
    return s


def run(state):
    c = state["c"]
    kind = c["kind"]
    if kind == "iterate":
        d = state["d"]
        d.set_estimate(None)
        if c["combined"]:
            d.iterate_combined(c["iters"])
        else:
            d.iterate(c["iters"])
        return _estimate(d)
    if kind == "noalloc":
        psi = state["psi"]
        psi.fill_(state["flat"])
        for phi, p, k in zip(state["views"], state["psfs"], state["comp"]):
            mvd.mvd_update_direct_noalloc(psi, phi, p, k, 1e-4 * state["flat"])
        return psi
    if kind == "batch":
        b = state["batch"]
        for d in b.volumes:
            d.set_estimate(None)
        mvd.mvd_batch_run(b.handle)
        mvd.mvd_batch_wait(b.handle)
        return [_estimate(d, b) for d in b.volumes]
    if kind == "series":
        d = state["d"]
        d.set_views(state["views"])
        d.iterate(c["iters"])
        return d.result(state["out"])
    if kind == "kernels":
        d = state["d"]
        mvd.mvd_precompute_kernels(d.ctx, c["variant"])
        return [d.compound_kernel(v) for v in range(d.n_views)]
    psi = autograd.unrolled_deconvolve(state["views"], state["psfs"], c["iters"])
    loss = ((psi - state["target"]) ** 2).mean()
    return [psi.detach(), *torch.autograd.grad(loss, [state["views"], *state["psfs"]])]


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def work(case):
    """Bytes: every view update reads the estimate and one view and writes the estimate. Operations: two
    convolutions per update, by real FFTs or directly, whichever is less."""
    c = dict(case)
    if c["kind"] == "batch":
        each = [work(p) for p in _parts(c)]
        return {k: sum(w[k] for w in each) for k in ("bytes", "flops")}
    M, n = c["X"] * c["Y"] * c["Z"], c["views"]
    taps = [p.size for p in _psfs(c)]
    if c["kind"] == "kernels":  # two linear convolutions per pair of kernels
        t = max(taps)
        return {"bytes": 4.0 * 2 * sum(taps), "flops": n * (n - 1) * 2 * 3 * 2.5 * 8 * t * math.log2(8 * t)}
    updates = n * c["iters"]
    conv = min(2.0 * max(taps) * M, 2 * 2.5 * M * math.log2(M) + 3 * M)
    w = {"bytes": 12.0 * M * updates, "flops": 2 * conv * updates}
    if c["kind"] == "grad":  # the reverse pass: four more convolutions and two correlations per update
        w = {"bytes": 3 * w["bytes"], "flops": 4 * w["flops"]}
    if c["kind"] == "series":
        w["bytes"] += 4.0 * M * (n + 1)
    return w


# ---------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------

def _flip(p):
    return torch.flip(p, (0, 1, 2))


def _linear(a, b):
    """Full linear convolution of two centred kernels (centred on the sum of the boxes)."""
    n = [x + y - 1 for x, y in zip(a.shape, b.shape)]
    return torch.fft.irfftn(torch.fft.rfftn(a, s=n) * torch.fft.rfftn(b, s=n), s=n)


def _on_box(q, shape):
    """The part of centred ``q`` on a centred box (zero outside q)."""
    for a, k in enumerate(shape):
        d = (q.shape[a] - k) // 2
        if d >= 0:
            q = q.narrow(a, d, k)
        else:
            pad = [0, 0, 0, 0, 0, 0]
            pad[2 * (2 - a)] = pad[2 * (2 - a) + 1] = -d
            q = torch.nn.functional.pad(q, pad)
    return q


def _compound(psfs, variant="efficient"):
    out = []
    for v, p in enumerate(psfs):
        m = _flip(p)
        k = m
        for w, q in enumerate(psfs):
            if w != v:
                a = _linear(m, q)
                if variant == "efficient":
                    a = _linear(a, _flip(q))
                k = k * _on_box(a, p.shape)
        out.append(k / k.sum())
    return out


class _Model:
    """Forward blur and back-projection of one view, for each boundary."""

    def __init__(self, shape, boundary, halo, P, K):
        self.n, self.boundary, self.h = shape, boundary, halo
        self.grid = tuple(shape) if boundary == "periodic" else tuple(n + 4 * h for n, h in zip(shape, halo))
        self.P, self.K = (_spectrum(k, self.grid, torch.float64, "cuda") for k in (P, K))
        self.s = None
        if boundary != "periodic":
            self.s = self.back(torch.ones(shape, dtype=torch.float64, device="cuda"))

    def conv(self, f, spec):
        return torch.fft.irfftn(torch.fft.rfftn(f, s=self.grid) * spec, s=self.grid)

    def crop(self, f):
        return f[tuple(slice(0, n) for n in self.n)]

    def blur(self, f):
        if self.boundary == "periodic":
            return self.conv(f, self.P)
        if self.boundary == "zero":
            return self.crop(self.conv(f, self.P))
        for a, (n, h) in enumerate(zip(self.n, self.h)):  # half-sample reflection on both sides
            f = torch.cat([f.narrow(a, 0, h).flip(a), f, f.narrow(a, n - h, h).flip(a)], a)
        f = self.conv(f, self.P)
        return f[tuple(slice(h, h + n) for n, h in zip(self.n, self.h))]

    def back(self, r):
        if self.boundary == "periodic":
            return self.conv(r, self.K)
        c = self.conv(r, self.K)
        if self.boundary == "zero":
            return self.crop(c)
        for a, (n, h) in enumerate(zip(self.n, self.h)):  # fold what lands past a face back
            core = c.narrow(a, 0, n).clone()
            core.narrow(a, 0, h).add_(c.narrow(a, c.shape[a] - h, h).flip(a))
            core.narrow(a, n - h, h).add_(c.narrow(a, n, h).flip(a))
            c = core
        return c


def _deconvolve64(c, psfs, views):
    f32 = np.float32
    P = [torch.from_numpy(p).cuda().double() for p in psfs]
    P = [p / p.sum() for p in P]
    K = _compound(P)
    shape = tuple(views[0].shape)
    mean = float(sum(v.sum(dtype=torch.float64) for v in views)) / (len(views) * views[0].numel())
    psi = torch.full(shape, float(f32(mean)), dtype=torch.float64, device="cuda")
    eps = float(f32(1e-4 * mean))
    halo = [max(p.shape[a] // 2 for p in P) for a in range(3)]
    wts = None
    if c["weights"]:
        wts = [w.double() for w in _weights(c)]
        total, count = sum(wts), sum((w > 0).double() for w in wts)
        T = float(count[count > 0].min())
        wts = [w * torch.clamp(T / total.clamp(min=1e-30), max=1.0) for w in wts]
    keep = len(views) * np.prod(shape) < 1 << 28
    models = [_Model(shape, c["boundary"], halo, p, k) for p, k in zip(P, K)] if keep else None
    for _ in range(c["iters"]):
        prod = None
        for v, phi in enumerate(views):
            m = models[v] if keep else _Model(shape, c["boundary"], halo, P[v], K[v])
            r = phi.double() / m.blur(psi).clamp_(min=eps)
            f = m.back(r)
            del r
            if m.s is not None:
                f = f / m.s
            if c["combined"]:
                prod = f if prod is None else prod * f
                continue
            if c["lam"]:
                f = f / (1 + c["lam"] * psi)
            if wts is not None:
                f = 1 + wts[v] * (f - 1)
            psi = (psi * f).clamp_(min=eps)
            del f, m
        if c["combined"]:
            psi = (psi * prod.clamp(min=0) ** (1.0 / len(views))).clamp_(min=eps)
    return psi


def exact(case, seed):
    c = dict(case)
    if c["kind"] == "batch":
        return [exact(p, seed * 31 + i) for i, p in enumerate(_parts(c))]
    psfs = _psfs(_measured(c, seed))
    if c["kind"] == "kernels":
        P = [torch.from_numpy(p).cuda().double() for p in psfs]
        return _compound([p / p.sum() for p in P], c["variant"])
    views = _volumes(c, psfs, seed)
    if c["kind"] in ("iterate", "series"):
        return _deconvolve64(c, psfs, views)
    if c["kind"] == "noalloc":
        shape = tuple(views[0].shape)
        flat = float(np.float32(np.mean([float(v.double().mean()) for v in views])))
        eps = float(np.float32(1e-4 * flat))
        psi = torch.full(shape, flat, dtype=torch.float64, device="cuda")
        for phi, p, k in zip(views, psfs, _compound([torch.from_numpy(p).double() for p in psfs])):
            m = _Model(shape, "periodic", None, p, k.float().cuda())
            psi = (psi * m.back(phi.double() / m.blur(psi).clamp(min=eps))).clamp(min=eps)
        return psi
    raw = [torch.from_numpy(p).cuda().double().requires_grad_() for p in psfs]
    vs = torch.stack(views)
    target = vs.mean(0).double()
    vs = vs.double().requires_grad_()
    P = [p / p.sum() for p in raw]
    shape = tuple(vs.shape[1:])
    models = [_Model(shape, "periodic", None, p, k) for p, k in zip(P, _compound(P))]
    psi = vs.mean().expand(shape)
    eps = torch.tensor(float(np.float32(1e-4 * float(vs.mean()))), dtype=torch.float64, device="cuda")
    for _ in range(c["iters"]):
        for v, m in enumerate(models):
            psi = (psi * m.back(vs[v] / m.blur(psi).clamp(min=eps))).clamp(min=eps)
    loss = ((psi - target) ** 2).mean()
    grads = torch.autograd.grad(loss, [vs, *raw])
    return [psi.detach(), *[g.detach() for g in grads]]
