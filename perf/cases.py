"""Workloads of the light-pollution convolution library, by what its users run.

Each case is one call (or one batch of requests) through the public entry
points of ``paper_1907_02891_gb300.lp``.  The kinds are the forms of the map:

* ``map``         ``lp_map``: one radiance map against ``n`` PSF spectra, SAME
                  or FULL output, point-symmetric PSFs (real spectra) or not
                  (complex spectra), FP32 or split-BF16 column transforms;
* ``multiclass``  ``lp_map_multiclass``: several source classes summed, one
                  PSF each;
* ``tiled``       ``lp_map_tiled`` at the padding ``lp_tiled_pad`` picks: maps
                  beyond the longest transform, or the SAME crop's padding;
* ``spectrum``    ``lp_kernel_spectrum`` of a PSF that is not cached yet, and
                  its copy: what every new atmosphere costs first;
* ``serve``       a batch of requests of mixed sizes and PSFs through the
                  scheduler (``lp_serve_submit`` / ``lp_serve_poll``).

A program keeps one context and a bank of spectra and maps many radiance
grids with them, so the context and the spectra are made once per process and
the maps come from the seed.
"""

import math

import numpy as np
import torch

from paper_1907_02891_gb300 import lp

# (a, p, lambda km) of the PSF families K(r) = (r^2 + a)^-p exp(-r / lambda)
FAMILY = [(0.1, p, lam) for lam in (80.0, 40.0, 120.0, 200.0) for p in (1.25, 2.0, 1.0, 1.5)]
PX_KM = 0.742

# request mix of a serving batch: every size with few and with many PSFs
SERVE_COUNTS = (3, 8, 5, 1, 6, 2, 7, 4)


def listed():
    return [
        # the smallest map of the test configurations: 12 cities of one region, launch-bound
        {"name": "map_256_psf101", "kind": "map", "h": 256, "w": 256, "hk": 101, "wk": 101, "n": 1,
         "full": False, "sym": True, "split": False, "cities": 12, "lit": 0.0},
        # a ragged regional map in FULL output with two wind-skewed (not point-symmetric) PSFs
        {"name": "full_1000x1333_skew2", "kind": "map", "h": 1000, "w": 1333, "hk": 161, "wk": 241, "n": 2,
         "full": True, "sym": False, "split": False, "cities": 60, "lit": 0.05},
        # a serving-size tile against the whole bank of eight atmospheres
        {"name": "map_2048_psf201x8", "kind": "map", "h": 2048, "w": 2048, "hk": 201, "wk": 201, "n": 8,
         "full": False, "sym": True, "split": False, "cities": 120, "lit": 0.05},
        # the ordinary national map (the benchmark's headline)
        {"name": "map_4096_psf541", "kind": "map", "h": 4096, "w": 4096, "hk": 541, "wk": 541, "n": 1,
         "full": False, "sym": True, "split": False, "cities": 400, "lit": 0.05},
        # the same map with the column transforms on the tensor cores
        {"name": "split_4096_psf541", "kind": "map", "h": 4096, "w": 4096, "hk": 541, "wk": 541, "n": 1,
         "full": False, "sym": True, "split": True, "cities": 400, "lit": 0.05},
        # batching: one map, sixteen atmospheres (4 extinction lengths x 4 exponents)
        {"name": "map_8192_psf601x16", "kind": "map", "h": 8192, "w": 8192, "hk": 601, "wk": 601, "n": 16,
         "full": False, "sym": True, "split": False, "cities": 1600, "lit": 0.05},
        # the paper's own map shape with its two maps (all-sky ratio at 300 km, zenith brightness)
        {"name": "map_11920x11804_psf1485x2", "kind": "map", "h": 11920, "w": 11804, "hk": 1485, "wk": 1485, "n": 2,
         "full": False, "sym": True, "split": False, "cities": 3300, "lit": 0.05},
        # the largest map one transform holds
        {"name": "map_16384_psf801", "kind": "map", "h": 16384, "w": 16384, "hk": 801, "wk": 801, "n": 1,
         "full": False, "sym": True, "split": False, "cities": 6400, "lit": 0.05},
        # three classes of sources (lamp types), one PSF each, summed
        {"name": "multiclass_4096_x3", "kind": "multiclass", "h": 4096, "w": 4096, "hk": 541, "wk": 541, "n": 3,
         "full": False, "sym": True, "split": False, "cities": 400, "lit": 0.05},
        # a map longer than the longest transform, in overlap-save tiles
        {"name": "tiled_17800x21000_psf801", "kind": "tiled", "h": 17800, "w": 21000, "hk": 801, "wk": 801, "n": 1,
         "full": False, "sym": True, "split": False, "cities": 8900, "lit": 0.05},
        # a new PSF for the national map: its spectrum
        {"name": "spectrum_541_4704", "kind": "spectrum", "h": 4096, "w": 4096, "hk": 541, "wk": 541, "n": 1,
         "full": False, "sym": True, "split": False, "cities": 0, "lit": 0.0},
        # a burst of requests of mixed tile sizes and PSF counts through the scheduler
        {"name": "serve_12", "kind": "serve", "h": 256, "w": 4096, "hk": 201, "wk": 201, "n": 12,
         "full": False, "sym": True, "split": False, "cities": 40, "lit": 0.05},
    ]


def _odd(x):
    return max(1, int(x)) | 1


def _between(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    """A case of the listed kinds with sizes over their whole range."""
    kind = rng.choice(("map", "map", "map", "map", "multiclass", "tiled", "spectrum", "serve"))
    c = {"kind": kind, "full": False, "sym": True, "split": False, "lit": 0.05}
    if kind == "serve":
        lo, hi = sorted((int(_between(rng, 200, 4096)), int(_between(rng, 200, 4096))))
        c.update(h=lo, w=hi, hk=_odd(_between(rng, 31, 201)), n=rng.randint(4, 12), cities=40)
        c["wk"] = c["hk"]
        return c
    big = {"map": 16384, "multiclass": 6000, "tiled": 16384, "spectrum": 9000}[kind]
    h = int(_between(rng, 200, big))
    w = min(big, max(200, int(h * _between(rng, 0.6, 1.6))))
    hk = min(_odd(_between(rng, 31, 1485)), _odd(h), _odd(17280 - h))
    wk = hk if rng.random() < 0.5 else min(_odd(hk * _between(rng, 0.7, 1.4)), _odd(w), _odd(17280 - w))
    most = max(1, min(16, int(2.5e8 / (float(h) * w))))
    n = 1
    if kind == "map":
        n = min(most, rng.choice((1, 1, 1, 2, 4, 8, 16)))
    elif kind == "multiclass":
        n = min(most, rng.randint(2, 4))
    c.update(h=h, w=w, hk=hk, wk=wk, n=n, cities=max(4, int(h * w / 42000)))
    c["sym"] = rng.random() < 0.75
    if kind == "map":
        c["full"] = rng.random() < 0.25
        c["split"] = rng.random() < 0.15
    return c


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------

def _radiance(h, w, cities, lit, gen):
    """Mostly dark FP32 map: Gaussian city blobs (sigma 1-5 px, log-normal
    peak; where blobs overlap the brighter one) and isolated lit pixels."""
    dev = "cuda"
    flat = torch.zeros(h * w, device=dev)
    if cities:
        d = torch.arange(-25, 26, device=dev)
        for part in range(0, cities, 2048):
            k = min(2048, cities - part)
            u = torch.rand(3, k, generator=gen, device=dev)
            peak = torch.exp(1.5 * torch.randn(k, generator=gen, device=dev))
            y, x, s = u[0] * h, u[1] * w, 1.0 + 4.0 * u[2]
            yi, xi = y.long()[:, None] + d, x.long()[:, None] + d
            gy = torch.exp(-(yi - y[:, None]) ** 2 / (2 * s[:, None] ** 2))
            gx = torch.exp(-(xi - x[:, None]) ** 2 / (2 * s[:, None] ** 2))
            v = peak[:, None, None] * gy[:, :, None] * gx[:, None, :]
            ok = ((yi >= 0) & (yi < h))[:, :, None] & ((xi >= 0) & (xi < w))[:, None, :]
            at = (yi.clamp(0, h - 1)[:, :, None] * w + xi.clamp(0, w - 1)[:, None, :])
            flat.scatter_reduce_(0, at[ok], v[ok], "amax")
    L = flat.view(h, w)
    if lit > 0.0:
        rows = max(1, (1 << 26) // w)
        for r in range(0, h, rows):
            b = L[r:r + rows]
            m = torch.rand(b.shape, generator=gen, device=dev) < lit
            b += m * torch.exp(1.5 * torch.randn(b.shape, generator=gen, device=dev))
    return L


def _psf(hk, wk, i, sym, scale=1.0):
    """PSF i of the family, FP64; not point-symmetric ones are skewed along
    a wind direction."""
    a, p, lam = FAMILY[i % len(FAMILY)]
    y = PX_KM * (torch.arange(hk, dtype=torch.float64, device="cuda") - hk // 2)[:, None]
    x = PX_KM * (torch.arange(wk, dtype=torch.float64, device="cuda") - wk // 2)[None, :]
    r = torch.hypot(y, x)
    K = (r * r + a) ** (-p) * torch.exp(-r / (lam * scale))
    if not sym:
        K = K * (1.0 + 0.4 * (math.cos(1.0 + i) * y + math.sin(1.0 + i) * x) / (r + 1.0))
    return K.contiguous()


_CTX = None
_SERVING = False
_SPECTRA = {}


def _context():
    global _CTX
    if _CTX is None:
        _CTX = lp.lp_create(0)
    return _CTX


def _spectrum(hk, wk, i, sym, ny, nx, split):
    key = (hk, wk, i % len(FAMILY), sym, ny, nx, split)
    if key not in _SPECTRA:
        K = _psf(hk, wk, i, sym)
        _SPECTRA[key] = lp.lp_kernel_spectrum(_context(), K, pad_ny=ny, pad_nx=nx,
                                              prec=lp.LP_PREC_SPLIT_BF16 if split else lp.LP_PREC_FP32)
        lp.lp_sync_status(_context())
    return _SPECTRA[key]


def _pads(case):
    h, w, hk, wk = case["h"], case["w"], case["hk"], case["wk"]
    if case["kind"] == "tiled":
        return lp.lp_tiled_pad(h, w, hk, wk)
    ny = lp.lp_supported_size(h + hk - 1)
    if case["split"]:
        ny = next(n for n in sorted(lp.supported_sizes()) if n >= h + hk - 1 and lp.lp_split_supported(n))
    return ny, lp.lp_supported_size(w + wk - 1)


def _out_shape(case):
    h, w = case["h"], case["w"]
    return (h + case["hk"] - 1, w + case["wk"] - 1) if case["full"] else (h, w)


def _requests(case):
    """(side, PSF numbers) of each request of a serving batch: sides between
    h and w, in powers of two where they are such, PSF counts of 1 to 8."""
    n, lo, hi = case["n"], case["h"], case["w"]
    out = []
    for r in range(n):
        f = ((5 * r) % n) / max(1, n - 1)
        side = int(round(lo * (hi / lo) ** f))
        if lo & (lo - 1) == 0 and hi & (hi - 1) == 0:
            side = 1 << int(round(math.log2(side)))
        k = SERVE_COUNTS[r % len(SERVE_COUNTS)]
        out.append((side, [(3 * r + q) % 8 for q in range(k)]))
    return out


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def prepare(case, seed):
    global _SERVING
    gen = _generator(seed)
    ctx = _context()
    kind = case["kind"]
    s = {"case": case, "ctx": ctx}
    if kind == "serve":
        if not _SERVING:
            lp.lp_serve_start(ctx, 4)
            _SERVING = True
        s["requests"] = []
        for side, ks in _requests(case):
            pad = lp.lp_supported_size(side + case["hk"] - 1)
            L = _radiance(side, side, case["cities"], case["lit"], gen)
            spectra = [_spectrum(case["hk"], case["wk"], k, True, pad, pad, False) for k in ks]
            s["requests"].append((L, spectra, [torch.empty_like(L) for _ in ks]))
        return s
    ny, nx = _pads(case)
    if kind == "spectrum":
        # a PSF of its own for every seed: attenuation length +-20 %
        f = 0.8 + 0.4 * torch.rand(1, generator=gen, device="cuda").item()
        s["K"] = _psf(case["hk"], case["wk"], 0, case["sym"], f)
        s["pad"] = (ny, nx)
        s["out"] = torch.empty(nx // 2 + 1, ny, 1 if case["sym"] else 2, device="cuda")
        return s
    s["spectra"] = [_spectrum(case["hk"], case["wk"], i, case["sym"], ny, nx, case["split"])
                    for i in range(case["n"])]
    maps = case["n"] if kind == "multiclass" else 1
    s["L"] = [_radiance(case["h"], case["w"], case["cities"], case["lit"], gen) for _ in range(maps)]
    outs = 1 if kind == "multiclass" else case["n"]
    s["out"] = [torch.empty(_out_shape(case), device="cuda") for _ in range(outs)]
    return s


def run(state):
    case, ctx = state["case"], state["ctx"]
    kind = case["kind"]
    mode = lp.LP_OUT_FULL if case["full"] else lp.LP_OUT_SAME
    prec = lp.LP_PREC_SPLIT_BF16 if case["split"] else lp.LP_PREC_FP32
    if kind == "map":
        lp.lp_map(ctx, state["L"][0], state["spectra"], state["out"], mode=mode, prec=prec)
    elif kind == "multiclass":
        lp.lp_map_multiclass(ctx, state["L"], state["spectra"], state["out"][0], mode=mode)
    elif kind == "tiled":
        lp.lp_map_tiled(ctx, state["L"][0], state["spectra"], state["out"])
    elif kind == "spectrum":
        ny, nx = state["pad"]
        spec = lp.lp_kernel_spectrum(ctx, state["K"], pad_ny=ny, pad_nx=nx)
        lp.lp_spectrum_copy(spec, state["out"])
        lp.lp_spectrum_release(ctx, spec)
    else:
        tickets = [lp.lp_serve_submit(ctx, L, spectra, outs) for L, spectra, outs in state["requests"]]
        for t in tickets:
            lp.lp_serve_poll(ctx, t)
        return [outs for _, _, outs in state["requests"]]
    return state["out"]


# --------------------------------------------------------------------------
# what a pass needs, and its exact values
# --------------------------------------------------------------------------

def _map_work(h, w, ny, nx, ho, wo, maps, spectra, outs, sym):
    pts = float(ny) * nx
    fft = 2.5 * pts * math.log2(pts)   # one real transform
    k = (nx // 2 + 1) * float(ny) * (4 if sym else 8)
    return (4.0 * h * w * maps + k * spectra + 4.0 * ho * wo * outs,
            fft * (maps + outs) + pts * (1 if sym else 3) * spectra)


def work(case):
    kind, hk, wk = case["kind"], case["hk"], case["wk"]
    if kind == "serve":
        b = f = 0.0
        for side, ks in _requests(case):
            pad = lp.lp_supported_size(side + hk - 1)
            x, y = _map_work(side, side, pad, pad, side, side, 1, len(ks), len(ks), True)
            b, f = b + x, f + y
        return {"bytes": b, "flops": f}
    ny, nx = _pads(case)
    if kind == "spectrum":
        per = 4.0 if case["sym"] else 8.0
        out = (nx // 2 + 1) * float(ny) * per
        # copy to the caller's buffer included: the spectrum written, read and written again
        pts = float(ny) * nx
        return {"bytes": 8.0 * hk * wk + 3 * out, "flops": 2.5 * pts * math.log2(pts)}
    if kind == "tiled":
        # the whole map as one linear convolution
        ny, nx = max(ny, case["h"] + hk - 1), max(nx, case["w"] + wk - 1)
    n = case["n"]
    multi = kind == "multiclass"
    ho, wo = _out_shape(case)
    b, f = _map_work(case["h"], case["w"], ny, nx, ho, wo, n if multi else 1, n, 1 if multi else n, case["sym"])
    return {"bytes": b, "flops": f}


def _smooth(n):
    while True:
        m = n
        for p in (2, 3, 5, 7):
            while m % p == 0:
                m //= p
        if m == 1:
            return n
        n += 1


def _wrapped(K, ny, nx):
    hk, wk = K.shape
    P = torch.zeros(ny, nx, dtype=torch.float64, device="cuda")
    P[:hk, :wk] = K
    return torch.roll(P, (-(hk // 2), -(wk // 2)), (0, 1))


def _convolved(Lhat, K, ny, nx, h, w, full):
    """Crop of the linear convolution whose map has the spectrum Lhat."""
    hk, wk = K.shape
    B = torch.fft.irfft2(torch.fft.rfft2(_wrapped(K, ny, nx)).mul_(Lhat), s=(ny, nx))
    if not full:
        return B[:h, :w].clone()
    B = torch.roll(B, (hk // 2, wk // 2), (0, 1))
    return B[:h + hk - 1, :w + wk - 1].clone()


def exact(case, seed):
    s = prepare(case, seed)
    kind, hk, wk = case["kind"], case["hk"], case["wk"]
    if kind == "serve":
        res = []
        for (L, _, _), (side, ks) in zip(s["requests"], _requests(case)):
            m = _smooth(side + hk - 1)
            Lh = torch.fft.rfft2(L.double(), s=(m, m))
            res.append([_convolved(Lh, _psf(hk, wk, k, True), m, m, side, side, False) for k in ks])
        return res
    if kind == "spectrum":
        ny, nx = s["pad"]
        S = torch.fft.rfft2(_wrapped(s["K"], ny, nx)).mul_(1.0 / (2.0 * ny * nx)).t()
        return (S.real.unsqueeze(-1) if case["sym"] else torch.view_as_real(S.contiguous())).contiguous()
    h, w = case["h"], case["w"]
    ny, nx = _smooth(h + hk - 1), _smooth(w + wk - 1)
    if kind == "multiclass":
        total = None
        for i, L in enumerate(s["L"]):
            B = _convolved(torch.fft.rfft2(L.double(), s=(ny, nx)), _psf(hk, wk, i, case["sym"]), ny, nx, h, w,
                           case["full"])
            total = B if total is None else total + B
        return [total]
    Lh = torch.fft.rfft2(s["L"][0].double(), s=(ny, nx))
    return [_convolved(Lh, _psf(hk, wk, i, case["sym"]), ny, nx, h, w, case["full"]) for i in range(case["n"])]
