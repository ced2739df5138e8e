"""Timed cases of the library: the calls of an angular differential imaging reduction, over the frame sides
(64 to 1024 pixels) and sequence lengths (one frame to 2000) that it takes.

Every case is one call (or the short run of calls of one step) of the Python binding on the default context, the
way a reduction script makes it: device cubes and their output buffers are allocated once and used again, per-frame
parameters are numpy arrays.  Inputs follow the recipes of ``synth.py``, generated on the GPU from the seed: a star
with a quasi-static speckle halo that decorrelates slowly and follows the detector, dithered by less than a pixel
(or by tens of pixels for registration), sky and read noise, alt-az or linear parallactic angles.

``exact`` restates each step in 64 bits with plain torch operations.
"""
import math

import numpy as np
import torch

from paper_1510_04331_gb300 import graphic

FWHM, N_FWHM = 4.0, 1.5
DEV = "cuda"
SURVEY_PIXELS = 2000 * 512 * 512   # the largest cube: the survey sequence


# ---- the cases ----------------------------------------------------------------------------------------------------

def listed():
    return [
        # one frame recentred, as an interactive quick look does: the smallest call, latency and launches
        {"name": "shift 1x512", "kind": "shift", "frames": 1, "n": 512},
        # a long sequence of small subarray frames (fast readout windows), recentred
        {"name": "shift 777x128", "kind": "shift", "frames": 777, "n": 128},
        # full-detector frames derotated: 2048-point lines, the longest the library has
        {"name": "rotate 60x1024", "kind": "rotate", "frames": 60, "n": 1024},
        # cubes of all sides of several targets recentred and derotated in one call (the scheduler's mode)
        {"name": "batch 14 cubes", "kind": "batch", "cubes": 14, "tmin": 3, "tmax": 48, "layout": 3},
        # PSF subtraction of one night's binned sequence, angles falling (a southern target), an odd frame count
        {"name": "adi 301x256", "kind": "adi", "frames": 301, "n": 256, "down": True, "t_max": 0.0},
        # the same step with the maximum time separation of the reference frames (hours)
        {"name": "adi time gate 600x256", "kind": "adi", "frames": 600, "n": 256, "down": False, "t_max": 0.5},
        # the whole reduction: the quick-look size, whose call is mostly launches and host work
        {"name": "reduce 32x128", "kind": "reduce", "frames": 32, "n": 128, "linear": True},
        # the whole reduction of the survey sequence, the headline workload
        {"name": "reduce 2000x512", "kind": "reduce", "frames": 2000, "n": 512, "linear": False},
        # the whole reduction from pinned host memory, as a pipeline that reads frames from disk calls it
        {"name": "reduce host 250x512", "kind": "reduce_host", "frames": 250, "n": 512, "linear": False},
        # pre-processing of raw frames: master skies, sky subtraction, bad pixel map, bad pixel correction
        {"name": "prep 200x512", "kind": "prep", "frames": 200, "n": 512, "skies": 4, "sky_frames": 50},
        # registration of raw frames: brightest patch, centroid, Moffat fit; a tenth of the frames lost
        {"name": "register 400x256", "kind": "register", "frames": 400, "n": 256},
        # median binning of a long sequence by 10, the last bin ragged
        {"name": "bin 1003x512 by 10", "kind": "bin", "frames": 1003, "n": 512, "bin": 10},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["shift", "rotate", "batch", "adi", "adi", "reduce", "reduce", "reduce_host", "prep", "register",
                       "bin"])
    n = rng.choice([64, 128, 256, 512, 1024])
    cap = SURVEY_PIXELS // (n * n)
    if kind in ("shift", "rotate"):
        return {"kind": kind, "frames": _log(rng, 1, min(2000, cap)), "n": n}
    if kind == "batch":
        return {"kind": kind, "cubes": rng.randint(2, 24), "tmin": rng.randint(1, 16), "tmax": rng.randint(17, 64),
                "layout": rng.randint(0, 10 ** 6)}
    if kind == "adi":
        gated = rng.random() < 0.35
        return {"kind": kind, "frames": _log(rng, 16, min(1000 if gated else 2048, cap // 4)), "n": n,
                "down": rng.random() < 0.5, "t_max": round(rng.uniform(0.2, 1.5), 3) if gated else 0.0}
    if kind in ("reduce", "reduce_host"):
        return {"kind": kind, "frames": _log(rng, 16, min(2000, cap // (4 if kind == "reduce_host" else 1))), "n": n,
                "linear": rng.random() < 0.5}
    if kind == "prep":
        return {"kind": kind, "frames": _log(rng, 8, min(1000, cap // 4)), "n": n, "skies": rng.randint(1, 6),
                "sky_frames": rng.randint(5, 60)}
    if kind == "register":
        return {"kind": kind, "frames": _log(rng, 1, min(2000, cap // 2)), "n": rng.choice([100, 128, 256, 512])}
    return {"kind": "bin", "frames": _log(rng, 20, min(2000, cap)), "n": n,
            "bin": rng.choice([2, 3, 5, 10, 16, 20, 32, 50, 64, 100])}


# ---- inputs -------------------------------------------------------------------------------------------------------

def _gen(seed, salt=0):
    return torch.Generator(device=DEV).manual_seed(1000003 * int(seed) + salt)


def _altaz(T):
    """Parallactic angles of a target at dec -30 seen from latitude -24.6, 1.5 h either side of the transit."""
    h = np.radians(np.linspace(-1.5, 1.5, T) * 15.0)
    d, p = math.radians(-30.0), math.radians(-24.6)
    return np.degrees(np.arctan2(math.cos(p) * np.sin(h),
                                 math.cos(d) * math.sin(p) - math.sin(d) * math.cos(p) * np.cos(h)))


def _edges(n):
    """Annulus edges 4, 8, ... n/2 pixels and one past the corner."""
    e = [4.0]
    while e[-1] * 2 <= n / 2:
        e.append(e[-1] * 2)
    return np.array(e + [float(math.ceil(n * math.sqrt(2.0) / 2.0) + 1)])


def _star_frames(x0, y0, n, sigma, amp):
    """Gaussian stars at (x0[t], y0[t]), amp[t] high: (T, n, n) float32."""
    g = torch.arange(n, device=DEV, dtype=torch.float64)
    gx = torch.exp(-(g[None, :] - x0[:, None]) ** 2 / (2 * sigma * sigma)).float()
    gy = (amp[:, None] * torch.exp(-(g[None, :] - y0[:, None]) ** 2 / (2 * sigma * sigma))).float()
    return gy[:, :, None] * gx[:, None, :]


def _halos(count, n, peak, rho, gen):
    """Speckle halos of AR(1) phase screens over a pupil of n/2 pixels: (count, n, n), mean maximum = peak."""
    G = 2 * n
    ax = torch.arange(G, device=DEV, dtype=torch.float32) - G / 2 + 0.5
    pupil = (ax[None, :] ** 2 + ax[:, None] ** 2) < (n / 4) ** 2
    f = torch.fft.fftfreq(G, device=DEV)
    r = torch.hypot(f[None, :], f[:, None])
    r[0, 0] = 1.0
    amp = r ** (-11.0 / 6.0)
    amp[0, 0] = 0.0

    def screen():
        w = torch.complex(torch.randn((G, G), generator=gen, device=DEV), torch.randn((G, G), generator=gen, device=DEV))
        s = torch.fft.ifft2(w * amp).real
        s = s - s[pupil].mean()
        return s * (0.3 / s[pupil].std())

    out = torch.empty((count, n, n), device=DEV)
    phi = screen()
    for a in range(count):
        if a:
            phi = rho * phi + math.sqrt(max(0.0, 1 - rho * rho)) * screen()
        e = torch.where(pupil, torch.polar(torch.ones_like(phi), phi), torch.zeros((), device=DEV, dtype=torch.complex64))
        e = torch.where(pupil, e - e[pupil].mean(), e)
        h = torch.fft.fftshift(torch.fft.fft2(e)).abs() ** 2
        out[a] = h[n // 2:n // 2 + n, n // 2:n // 2 + n]
    return out * (peak / out.amax(dim=(1, 2)).mean())


def _adi_cube(T, n, seed, parang, peak):
    """A dithered star with its speckle halo, two companions, sky and read noise; and the recentring shifts."""
    gen = _gen(seed)
    rng = np.random.default_rng(seed)
    anchors = max(2, T // 50 + 1)
    rho = 0.99 ** (T / (anchors - 1))
    halos = _halos(anchors, n, 1e-2 * peak, rho, gen)
    delta = rng.uniform(-0.5, 0.5, (T, 2))
    sigma = FWHM / (2 * math.sqrt(2 * math.log(2)))
    cube = torch.empty((T, n, n), device=DEV)
    comps = [(0.12 * n, rng.uniform(0, 360), 1e-3), (0.3 * n, rng.uniform(0, 360), 1e-4)]
    step = max(1, (1 << 26) // (n * n))
    for t0 in range(0, T, step):
        t = np.arange(t0, min(T, t0 + step))
        u = t / max(1, T - 1) * (anchors - 1)
        a = np.minimum(u.astype(int), anchors - 2)
        w = torch.as_tensor(u - a, device=DEV, dtype=torch.float32)[:, None, None]
        ai = torch.as_tensor(a, device=DEV)
        fr = torch.lerp(halos[ai], halos[ai + 1], w)
        x = torch.as_tensor(n / 2 + delta[t, 0], device=DEV)
        y = torch.as_tensor(n / 2 + delta[t, 1], device=DEV)
        one = torch.ones(len(t), device=DEV, dtype=torch.float64)
        fr += _star_frames(x, y, n, sigma, peak * one)
        for (rad, pa, con) in comps:
            ang = torch.as_tensor(np.radians(pa + parang[t]), device=DEV)
            fr += _star_frames(x + rad * torch.cos(ang), y + rad * torch.sin(ang), n, sigma, con * peak * one)
        fr += torch.sqrt(fr.clamp_min(0) + 75.0) * torch.randn(fr.shape, generator=gen, device=DEV)
        cube[t0:t0 + len(t)] = fr
    return cube, -delta[:, 0].copy(), -delta[:, 1].copy()


def _batch_layout(case):
    rng = np.random.default_rng(case["layout"])
    return [(int(rng.choice([64, 128, 256, 512, 1024])), int(rng.integers(case["tmin"], case["tmax"] + 1)))
            for _ in range(case["cubes"])]


def _plain_frames(T, n, seed, salt):
    """Noise frames with a star at the centre."""
    gen = _gen(seed, salt)
    cube = torch.randn((T, n, n), generator=gen, device=DEV)
    c = torch.full((1,), n / 2, device=DEV, dtype=torch.float64)
    cube += _star_frames(c, c, n, 1.7, 100.0 * torch.ones_like(c))
    return cube


def _angles(case):
    T = case["frames"]
    if case.get("linear"):
        return np.linspace(0.0, 40.0, T)
    a = _altaz(T)
    return a[::-1].copy() if case.get("down") else a


def _prep_inputs(case, seed):
    T, n, ns, nf = case["frames"], case["n"], case["skies"], case["sky_frames"]
    gen = _gen(seed)
    rng = np.random.default_rng(seed)
    det = np.random.default_rng(77)   # the detector's defects are the same in every night
    science = torch.randn((T, n, n), generator=gen, device=DEV) * 10.0 + 100.0
    skyf = torch.randn((ns * nf, n, n), generator=gen, device=DEV) * 3.0 + 100.0
    dark = torch.randn((n, n), generator=gen, device=DEV)
    dark.view(-1)[torch.as_tensor(det.choice(n * n, n * n // 1000, replace=False), device=DEV)] = 100.0
    for (r0, c0) in det.integers(4, n - 8, (5, 2)):
        dark[r0:r0 + 3, c0:c0 + 3] = 100.0
    cosmic = torch.as_tensor(rng.integers(0, T * n * n, max(1, T * n * n // 100000)), device=DEV)
    science.view(-1)[cosmic] = float("nan")
    x0, y0 = rng.uniform(0.2 * n, 0.8 * n, ns * nf), rng.uniform(0.2 * n, 0.8 * n, ns * nf)
    return dict(science=science, skyf=skyf, dark=dark, x0=x0, y0=y0, mask_r=0.06 * n,
                frame_t=np.linspace(0.0, 1.0, T), sky_t=np.linspace(0.0, 1.0, ns))


def _raw_stars(case, seed):
    T, n = case["frames"], case["n"]
    rng = np.random.default_rng(seed)
    x = torch.as_tensor(n / 2 + rng.uniform(-0.2 * n, 0.2 * n, T), device=DEV)
    y = torch.as_tensor(n / 2 + rng.uniform(-0.2 * n, 0.2 * n, T), device=DEV)
    amp = torch.as_tensor(np.where(rng.random(T) < 0.1, 100.0, 1e4), device=DEV)
    sigma = FWHM / (2 * math.sqrt(2 * math.log(2)))
    gen = _gen(seed)
    cube = torch.empty((T, n, n), device=DEV)
    step = max(1, (1 << 26) // (n * n))
    for a in range(0, T, step):
        s = slice(a, min(T, a + step))
        fr = _star_frames(x[s], y[s], n, sigma, amp[s])
        fr += _star_frames(x[s], y[s], n, 2.0 * sigma, 0.08 * amp[s])
        fr += _star_frames(x[s], y[s], n, 4.5 * sigma, 0.012 * amp[s])
        fr += torch.sqrt(fr.clamp_min(0) + 75.0) * torch.randn(fr.shape, generator=gen, device=DEV)
        cube[s] = fr
    return cube


REG = dict(thresh=1e3, R=16, min_size=4, max_size=400, w=10)


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case, "kind": kind}
    if kind == "batch":
        rng = np.random.default_rng(seed)
        lay = _batch_layout(case)
        s["cubes"] = [_plain_frames(T, n, seed, i) for i, (n, T) in enumerate(lay)]
        s["outs"] = [torch.empty_like(c) for c in s["cubes"]]
        s["dx"] = [rng.uniform(-2, 2, T) for (_, T) in lay]
        s["dy"] = [rng.uniform(-2, 2, T) for (_, T) in lay]
        s["theta"] = [rng.uniform(0, 360, T) for (_, T) in lay]
        return s
    T, n = case["frames"], case["n"]
    if kind in ("shift", "rotate"):
        rng = np.random.default_rng(seed)
        s["cube"] = _plain_frames(T, n, seed, 0)
        s["out"] = torch.empty_like(s["cube"])
        s["dx"], s["dy"] = rng.uniform(-2, 2, T), rng.uniform(-2, 2, T)
        s["theta"] = rng.uniform(0, 360, T)
    elif kind == "adi":
        s["parang"], s["edges"] = _angles(case), _edges(n)
        s["times"] = np.linspace(0.0, 3.0, T) if case["t_max"] > 0 else None
        s["cube"] = _adi_cube(T, n, seed, s["parang"], 1e5)[0]
        s["out"] = torch.empty_like(s["cube"])
    elif kind in ("reduce", "reduce_host"):
        s["parang"], s["edges"] = _angles(case), _edges(n)
        s["cube"], s["dx"], s["dy"] = _adi_cube(T, n, seed, s["parang"], 1e4 if case["linear"] else 1e5)
        if kind == "reduce_host":
            host = torch.empty((T, n, n), pin_memory=True)
            host.copy_(s["cube"])
            s["cube"] = host
            s["out"] = torch.empty((n, n), pin_memory=True)
        else:
            s["work"] = torch.empty_like(s["cube"])
            s["out"] = torch.empty((n, n), device=DEV)
    elif kind == "prep":
        s.update(_prep_inputs(case, seed))
        s["work"] = torch.empty_like(s["science"])
        s["sky"] = torch.empty((case["skies"], n, n), device=DEV)
    elif kind == "register":
        s["cube"] = _raw_stars(case, seed)
        s["out"] = torch.empty((T, 8), dtype=torch.float64, device=DEV)
    else:
        s["cube"] = _plain_frames(T, n, seed, 0)
        s["out"] = torch.empty((-(-T // case["bin"]), n, n), device=DEV)
    return s


def run(s):
    kind, case = s["kind"], s["case"]
    if kind == "shift":
        return graphic.graphic_shift(s["cube"], s["dx"], s["dy"], out=s["out"])
    if kind == "rotate":
        return graphic.graphic_rotate(s["cube"], s["theta"], out=s["out"])
    if kind == "batch":
        return graphic.context().graphic_batch_geom(s["cubes"], s["dx"], s["dy"], s["theta"], outs=s["outs"])
    if kind == "adi":
        return graphic.graphic_adi_subtract(s["cube"], s["parang"], FWHM, N_FWHM, s["edges"], out=s["out"],
                                            times=s["times"], t_max=case["t_max"] if s["times"] is not None else None)
    if kind == "reduce":
        return graphic.graphic_reduce(s["cube"], s["dx"], s["dy"], s["parang"], FWHM, N_FWHM, s["edges"],
                                      work=s["work"], out=s["out"])
    if kind == "reduce_host":
        return graphic.graphic_reduce_host(s["cube"], s["dx"], s["dy"], s["parang"], FWHM, N_FWHM, s["edges"],
                                           out_host=s["out"])
    if kind == "prep":
        ctx, nf = graphic.context(), case["sky_frames"]
        for j in range(case["skies"]):
            k = slice(j * nf, (j + 1) * nf)
            ctx.graphic_sky_median(s["skyf"][k], s["x0"][k], s["y0"][k], s["mask_r"], out=s["sky"][j])
        ctx.graphic_sky_subtract(s["science"], s["sky"], s["frame_t"], s["sky_t"], out=s["work"])
        bad = ctx.graphic_bad_pixel_map(s["dark"], 5.0)
        ctx.graphic_bad_pixel_fix(s["work"], bad)
        return {"sky": s["sky"], "bad": bad, "frames": s["work"]}
    if kind == "register":
        return graphic.graphic_register(s["cube"], out=s["out"], **REG)
    return graphic.graphic_bin_median(s["cube"], case["bin"], out=s["out"])


# ---- what a pass cannot do without --------------------------------------------------------------------------------

def _fft_flops(n, lines):
    """Forward and inverse complex transforms of 2n points, two real lines each."""
    m = 2 * n
    return (lines / 2) * 2 * 5 * m * math.log2(m)


def _shift_flops(T, n):
    return T * 2 * _fft_flops(n, n)


def _rotate_flops(T, n):
    return T * (2 * _fft_flops(n, n) + _fft_flops(n, 2 * n))


def work(case):
    kind = case["kind"]
    if kind == "batch":
        lay = _batch_layout(case)
        return {"bytes": sum(8 * T * n * n for n, T in lay),
                "flops": sum(_shift_flops(T, n) + _rotate_flops(T, n) for n, T in lay)}
    T, n = case["frames"], case["n"]
    cube, img = 4 * T * n * n, 4 * n * n
    if kind == "shift":
        return {"bytes": 2 * cube, "flops": _shift_flops(T, n)}
    if kind == "rotate":
        return {"bytes": 2 * cube, "flops": _rotate_flops(T, n)}
    if kind == "adi":
        return {"bytes": 2 * cube, "flops": 0}
    if kind in ("reduce", "reduce_host"):
        return {"bytes": cube + img, "flops": _shift_flops(T, n) + _rotate_flops(T, n)}
    if kind == "prep":
        return {"bytes": 2 * cube + (case["skies"] * (case["sky_frames"] + 1) + 1) * img + n * n, "flops": 0}
    if kind == "register":
        return {"bytes": cube + 64 * T, "flops": 0}
    return {"bytes": cube + 4 * n * n * -(-T // case["bin"]), "flops": 0}


# ---- the steps in 64 bits -----------------------------------------------------------------------------------------

def _phase(m, d):
    """Half-spectrum factors of periodic shifts d (any shape) of m-point lines: exp(-i 2 pi k d / m), the Nyquist
    bin cos(pi d)."""
    k = torch.arange(m // 2 + 1, device=DEV, dtype=torch.float64)
    h = torch.polar(torch.ones((), device=DEV, dtype=torch.float64).expand(d.shape + k.shape).contiguous(),
                    -2 * math.pi / m * d[..., None] * k)
    h[..., m // 2] = torch.cos(math.pi * d).to(h.dtype)
    return h


def _lines(x, d):
    """Each line of the last axis of x moved by d (periodic)."""
    return torch.fft.irfft(torch.fft.rfft(x) * _phase(x.shape[-1], d), n=x.shape[-1])


def _pad(x, n):
    """n samples of the last axis at offset n/2 of 2n."""
    return torch.nn.functional.pad(x, (n // 2, n - n // 2))


def _crop(x, n):
    return x[..., n // 2:n // 2 + n]


def _shift64(cube, dx, dy):
    n = cube.shape[-1]
    out = torch.empty(cube.shape, device=DEV, dtype=torch.float64)
    step = max(1, (1 << 24) // (n * n))
    for a in range(0, cube.shape[0], step):
        s = slice(a, a + step)
        x = cube[s].to(DEV).double()
        mx, my = (torch.as_tensor(v[s], device=DEV)[:, None] for v in (dx, dy))
        x = _crop(_lines(_pad(x, n), mx), n)
        x = _crop(_lines(_pad(x.mT, n), my), n).mT
        out[s] = x
    return out


def _quarter(x, q):
    """The exact quarter turns: output (x, y) takes the input at the point turned back, zero outside the frame."""
    n = x.shape[-1]
    r = torch.arange(n, device=DEV)
    row, col = torch.meshgrid(r, r, indexing="ij")
    X, Y = col - n // 2, row - n // 2
    sx, sy = [(X, Y), (Y, -X), (-X, -Y), (-Y, X)][q]
    sc, sr = sx + n // 2, sy + n // 2
    ok = (sc >= 0) & (sc < n) & (sr >= 0) & (sr < n)
    return torch.where(ok, x[..., sr.clamp(0, n - 1), sc.clamp(0, n - 1)], torch.zeros((), device=DEV, dtype=x.dtype))


def _rotate64(cube, theta):
    T, n = cube.shape[0], cube.shape[-1]
    q = np.floor(np.asarray(theta) / 90.0 + 0.5)
    r = np.radians(np.asarray(theta) - 90.0 * q)
    out = torch.empty(cube.shape, device=DEV, dtype=torch.float64)
    step = max(1, (1 << 23) // (n * n))
    for a in range(0, T, step):
        s = slice(a, min(T, a + step))
        x = torch.stack([_quarter(cube[t].to(DEV).double(), int(q[t]) % 4) for t in range(s.start, s.stop)])
        ta = torch.as_tensor(np.tan(r[s] / 2), device=DEV)[:, None]
        sn = torch.as_tensor(np.sin(r[s]), device=DEV)[:, None]
        y = torch.arange(n, device=DEV, dtype=torch.float64)[None, :] - n // 2
        xc = torch.arange(2 * n, device=DEV, dtype=torch.float64)[None, :] - n
        x = _lines(_pad(x, n), -ta * y)
        x = _crop(_lines(_pad(x.mT, n), sn * xc), n).mT
        out[s] = _crop(_lines(x, -ta * y), n)
    return out


def _median64(x):
    """Median over the first axis, the two middle values averaged."""
    v = torch.sort(x, dim=0).values
    T = x.shape[0]
    return (v[(T - 1) // 2] + v[T // 2]) / 2


def _adi64(cube, parang, edges, times=None, t_max=0.0):
    T, n = cube.shape[0], cube.shape[-1]
    flat = cube.reshape(T, -1)
    out = torch.zeros((T, n * n), device=DEV, dtype=torch.float64)
    g = torch.arange(n, device=DEV, dtype=torch.float64) - n // 2
    rho2 = (g[:, None] ** 2 + g[None, :] ** 2).reshape(-1)
    ang = torch.as_tensor(np.asarray(parang), device=DEV)
    tt = None if times is None else torch.as_tensor(np.asarray(times), device=DEV)
    for e0, e1 in zip(edges[:-1], edges[1:]):
        pix = torch.nonzero((rho2 >= e0 * e0) & (rho2 < e1 * e1))[:, 0]
        amin = 2 * math.degrees(math.asin(min(1.0, N_FWHM * FWHM / (2 * e0))))
        sep = (ang[:, None] - ang[None, :]).abs()
        near = torch.ones_like(sep, dtype=torch.bool) if tt is None else (tt[:, None] - tt[None, :]).abs() < t_max
        ref = (sep > amin) & near
        for t in torch.nonzero(~ref.any(1))[:, 0].tolist():
            ref[t] = near[t] & (sep[t] == sep[t][near[t]].max())
        for part in torch.split(pix, max(1, (1 << 24) // T)):
            x = flat[:, part].double()
            v, order = torch.sort(x, dim=0)
            cnt = ref.sum(1).tolist()
            for t in range(T):
                c = torch.cumsum(ref[t][order].to(torch.int16), 0, dtype=torch.int16)
                lo = (c <= (cnt[t] - 1) // 2).sum(0, keepdim=True)
                hi = (c <= cnt[t] // 2).sum(0, keepdim=True)
                out[t, part] = x[t] - (v.gather(0, lo)[0] + v.gather(0, hi)[0]) / 2
    return out.reshape(T, n, n)


def _fix64(x, bad):
    """NaN and flagged pixels filled by the median of their finite neighbours, pass by pass."""
    x = torch.where(bad[None] | ~torch.isfinite(x), torch.full((), float("nan"), device=DEV, dtype=x.dtype), x)
    for _ in range(2 * x.shape[-1]):
        hole = torch.isnan(x)
        at = torch.nonzero(hole)
        if not len(at):
            break
        p = torch.nn.functional.pad(x, (1, 1, 1, 1), value=float("nan"))
        t, r, c = at.unbind(1)
        nb = torch.stack([p[t, r + i, c + j] for i in range(3) for j in range(3) if (i, j) != (1, 1)])
        m = torch.isfinite(nb).sum(0)
        v = torch.sort(torch.where(torch.isnan(nb), torch.full_like(nb, float("inf")), nb), dim=0).values
        k = m.clamp_min(1)[None]
        med = (v.gather(0, (k - 1) // 2)[0] + v.gather(0, k // 2)[0]) / 2
        x = x.clone()
        x[t, r, c] = torch.where(m > 0, med, torch.full_like(med, float("nan")))
    return x


def _prep64(case, seed):
    d, nf = _prep_inputs(case, seed), case["sky_frames"]
    T, n = case["frames"], case["n"]
    g = torch.arange(n, device=DEV, dtype=torch.float64)
    skies = []
    for j in range(case["skies"]):
        k = slice(j * nf, (j + 1) * nf)
        x = d["skyf"][k].double()
        cx, cy = (torch.as_tensor(d[a][k], device=DEV) for a in ("x0", "y0"))
        out = ((g[None, None, :] - cx[:, None, None]) ** 2 + (g[None, :, None] - cy[:, None, None]) ** 2
               < d["mask_r"] ** 2) | ~torch.isfinite(x)
        v = torch.sort(torch.where(out, torch.full_like(x, float("inf")), x), dim=0).values
        m = (~out).sum(0, keepdim=True)
        k = m.clamp_min(1)
        med = (v.gather(0, (k - 1) // 2) + v.gather(0, k // 2)) / 2
        skies.append(torch.where(m > 0, med, torch.full_like(med, float("nan")))[0])
    sky = torch.stack(skies)
    near = np.abs(d["frame_t"][:, None] - d["sky_t"][None, :]).argmin(1)
    dark = d["dark"].double()
    v = torch.sort(dark.reshape(-1)).values
    med = (v[(n * n - 1) // 2] + v[n * n // 2]) / 2
    bad = (dark - med).abs() > 5.0 * dark.std(correction=0)
    frames = torch.cat([_fix64(d["science"][a:a + 64].double() - sky[torch.as_tensor(near[a:a + 64], device=DEV)], bad)
                        for a in range(0, T, 64)])
    return {"sky": sky, "bad": None, "frames": frames}


def _register64(case, seed):
    """The patch centroid of each frame's star, then the least-squares Moffat profile of the window around it."""
    cube = _raw_stars(case, seed)
    T, n = cube.shape[0], cube.shape[-1]
    R, w = REG["R"], REG["w"]
    out = torch.zeros((T, 8), device=DEV, dtype=torch.float64)
    keep, X, Y, V, P = [], [], [], [], []
    for t in range(T):
        fr = cube[t]
        at = int(torch.argmax(fr))
        r, c = at // n, at % n
        if float(fr[r, c]) <= REG["thresh"]:
            continue
        r0, c0 = max(0, r - R), max(0, c - R)
        box = fr[r0:r + R + 1, c0:c + R + 1].double()
        # a single smooth star: every pixel of the box above the threshold belongs to its patch
        i, j = torch.nonzero(box > REG["thresh"]).unbind(1)
        v = box[i, j]
        cx, cy = float((v * (j + c0)).sum() / v.sum()), float((v * (i + r0)).sum() / v.sum())
        rc, cc = math.floor(cy + 0.5), math.floor(cx + 0.5)
        if min(rc, cc) < w or max(rc, cc) + w >= n:
            return None   # a clipped window: the windows of a batched fit have one size
        keep.append(t)
        g = torch.arange(-w, w + 1, device=DEV, dtype=torch.float64)
        Y.append((g + rc)[:, None].expand(2 * w + 1, 2 * w + 1).reshape(-1))
        X.append((g + cc)[None, :].expand(2 * w + 1, 2 * w + 1).reshape(-1))
        z = fr[rc - w:rc + w + 1, cc - w:cc + w + 1].double().reshape(-1)
        V.append(z)
        bg = float(z.min())
        P.append([float((z - bg).sum()), cx, cy, max(1.0, math.sqrt(len(i) / math.pi)), 2.5, bg])
    if not keep:
        return out
    X, Y, V, p = torch.stack(X), torch.stack(Y), torch.stack(V), torch.tensor(P, device=DEV, dtype=torch.float64)

    def model(p):
        I0, x0, y0, al, be, bg = (p[:, k:k + 1] for k in range(6))
        dx, dy = X - x0, Y - y0
        rr = dx * dx + dy * dy
        u = 1 + rr / al ** 2
        pw = u ** -be
        c = (be - 1) / (math.pi * al ** 2)
        A = I0 * c
        J = torch.stack([c * pw, 2 * A * be / al ** 2 * pw / u * dx, 2 * A * be / al ** 2 * pw / u * dy,
                         -2 * A / al * pw + 2 * A * be / al ** 3 * rr * pw / u,
                         I0 / (math.pi * al ** 2) * pw - A * torch.log(u) * pw, torch.ones_like(pw)], 2)
        e = A * pw + bg - V
        return e, J, (e * e).sum(1)

    lam = torch.full((len(keep),), 1e-3, device=DEV, dtype=torch.float64)
    e, J, cost = model(p)
    for _ in range(80):
        H = J.mT @ J
        A = H + torch.diag_embed(lam[:, None] * torch.diagonal(H, dim1=1, dim2=2))
        q = p - torch.linalg.solve(A, (J.mT @ e[..., None]))[..., 0]
        q = torch.where(((q[:, 3:4] > 0) & (q[:, 4:5] > 1)), q, p)
        e2, J2, cost2 = model(q)
        good = cost2 <= cost
        p = torch.where(good[:, None], q, p)
        e, J = torch.where(good[:, None], e2, e), torch.where(good[:, None, None], J2, J)
        cost = torch.where(good, cost2, cost)
        lam = torch.where(good, lam / 10, lam * 10).clamp(1e-12, 1e6)
    k = torch.as_tensor(keep, device=DEV)
    fw = 2 * p[:, 3] * torch.sqrt(2 ** (1 / p[:, 4]) - 1)
    out[k] = torch.stack([torch.ones_like(fw), p[:, 1], p[:, 2], fw, p[:, 0], p[:, 3], p[:, 4], p[:, 5]], 1)
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        s = prepare(case, seed)
        return [_rotate64(_shift64(c, dx, dy), th) for c, dx, dy, th in zip(s["cubes"], s["dx"], s["dy"], s["theta"])]
    T, n = case["frames"], case["n"]
    if kind in ("adi", "reduce", "reduce_host") and T * T * n * n > 3e10:
        return None   # the medians of every frame by brute force would take minutes
    if kind == "prep":
        return _prep64(case, seed)
    if kind == "register":
        return _register64(case, seed)
    s = prepare(case, seed)
    if kind == "shift":
        return _shift64(s["cube"], s["dx"], s["dy"])
    if kind == "rotate":
        return _rotate64(s["cube"], s["theta"])
    if kind == "adi":
        return _adi64(s["cube"], s["parang"], s["edges"], s["times"], case["t_max"])
    if kind in ("reduce", "reduce_host"):
        x = _adi64(_shift64(s["cube"], s["dx"], s["dy"]), s["parang"], s["edges"])
        return _median64(_rotate64(x, -s["parang"]))
    B = case["bin"]
    return torch.stack([_median64(s["cube"][a:a + B].double()) for a in range(0, T, B)])
