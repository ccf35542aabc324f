"""The work that a user of fastmap has it do, as cases to be timed and compared.

Every case is one pass through a public entry point of
`paper_1204_4293_gb300.fastmap`, on inputs a user's program would have on the
GPU: shear of a Gaussian random field (P(k) ~ k^-2, rms 0.02) with 0.1 shape
noise a pixel and component, a 15 % star mask where there is one.
"""
import math

import numpy as np
import torch

from paper_1204_4293_gb300 import fastmap as fm

DEV = "cuda"
DTYPES = {"f32": torch.float32, "f64": torch.float64}
FILTERS = {"starlet": (fm.FM_FILTER_STARLET, 2.0), "s98": (fm.FM_FILTER_S98, 1.0), "jbj04": (fm.FM_FILTER_JBJ04, 5.0)}


# ---- the cases -------------------------------------------------------------------
def listed():
    return [
        # one small map at a time, as a server gets them: launches and latency
        {"name": "map 256 single", "kind": "map", "n": 256, "J": 6, "batch": 1, "dtype": "f32", "periodic": False, "keep": False},
        # the paper's workload: one 1024 x 1024 map, radii 2 .. 64 px
        {"name": "map 1024 single", "kind": "map", "n": 1024, "J": 7, "batch": 1, "dtype": "f32", "periodic": False, "keep": False},
        # a survey's tiles: batches of maps into one kept pyramid buffer (the benchmark's step)
        {"name": "map 1024 batch 32", "kind": "map", "n": 1024, "J": 7, "batch": 32, "dtype": "f32", "periodic": False, "keep": True},
        # the largest field
        {"name": "map 8192 single", "kind": "map", "n": 8192, "J": 9, "batch": 1, "dtype": "f32", "periodic": False, "keep": False},
        # the paper's workload in double precision
        {"name": "map 1024 f64", "kind": "map", "n": 1024, "J": 7, "batch": 1, "dtype": "f64", "periodic": False, "keep": False},
        # convergence maps with the B mode as the null test
        {"name": "ks 2048 E and B", "kind": "ks", "n": 2048, "batch": 8, "dtype": "f32", "with_b": True},
        # the transform alone on convergence maps whose side is no power of two
        {"name": "starlet 1500", "kind": "starlet", "n": 1500, "J": 7, "batch": 3, "dtype": "f32", "periodic": True},
        # a noise and a S/N map from 100 rotated realisations
        {"name": "noise 1024 R 100", "kind": "noise", "n": 1024, "J": 7, "R": 100, "dtype": "f32", "periodic": False},
        # the same variance's exact expectation
        {"name": "noise expected 1024", "kind": "expected", "n": 1024, "J": 7, "dtype": "f32"},
        # the direct sum with the starlet-shaped filter (the comparison path)
        {"name": "direct 1024", "kind": "direct", "n": 1024, "batch": 1, "filter": "starlet", "theta": 16.0, "dtype": "f32"},
        # fields with masked stars: only the direct estimator takes weights
        {"name": "masked 1000", "kind": "masked", "n": 1000, "batch": 2, "filter": "s98", "theta": 16.0, "dtype": "f32"},
        # <M_ap^2>, skewness and kurtosis of every band of a batch
        {"name": "moments 1024", "kind": "moments", "n": 1024, "J": 7, "batch": 8, "dtype": "f32"},
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, round(math.exp(rng.uniform(math.log(lo), math.log(hi))))))


def draw(rng):
    while True:
        c = _draw(rng)
        w = work(c)
        flops = 3e9 if c["dtype"] == "f64" else 5.5e10 if c["kind"] == "direct" else 2e10
        if w["bytes"] <= 2.9e9 and (c["kind"] not in ("direct", "masked") or w["flops"] <= flops):
            return c


def _draw(rng):
    kind = rng.choices(["map", "ks", "starlet", "noise", "expected", "direct", "masked", "moments"],
                       [8, 2, 3, 2, 1, 2, 2, 1])[0]
    dtype = "f64" if rng.random() < 0.2 else "f32"
    periodic = rng.random() < 0.3
    n = 1 << rng.randint(6, 13)  # the FFT's sizes in use: 64 .. 8192
    room = max(1, (1 << (25 if dtype == "f32" else 24)) // n**2)
    batch = rng.choice([1, _log_int(rng, 1, min(256, room))])
    J = rng.randint(max(3, int(math.log2(n)) - 4), min(10, int(math.log2(n)) - 1))
    if kind == "map":
        return {"kind": kind, "n": n, "J": J, "batch": batch, "dtype": dtype, "periodic": periodic, "keep": rng.random() < 0.5}
    if kind == "ks":
        return {"kind": kind, "n": n, "batch": batch, "dtype": dtype, "with_b": rng.random() < 0.5}
    if kind == "starlet":
        n = _log_int(rng, 50, 5000)
        batch = rng.choice([1, _log_int(rng, 1, max(1, min(64, (1 << 24) // n**2)))])
        J = rng.randint(3, min(10, int(math.log2(n)) - 1))
        return {"kind": kind, "n": n, "J": J, "batch": batch, "dtype": dtype, "periodic": periodic}
    if kind == "noise":
        n = 1 << rng.randint(6, 11)
        J = min(J, int(math.log2(n)) - 1)
        R = _log_int(rng, 10, 300 if n < 1024 else 100 if n == 1024 else 25)
        return {"kind": kind, "n": n, "J": J, "R": R if dtype == "f32" else max(5, R // 8), "dtype": dtype, "periodic": periodic}
    if kind == "expected":
        n = 1 << rng.randint(6, 11)
        return {"kind": kind, "n": n, "J": min(J, int(math.log2(n)) - 1), "dtype": dtype}
    if kind == "moments":
        n = _log_int(rng, 60, 4096)
        return {"kind": kind, "n": n, "J": rng.randint(3, 9), "batch": _log_int(rng, 1, max(1, min(16, (1 << 24) // n**2))), "dtype": dtype}
    n = _log_int(rng, 60, 2048)
    return {"kind": kind, "n": n, "batch": _log_int(rng, 1, max(1, min(8, (1 << 21) // n**2))), "filter": rng.choice(sorted(FILTERS)),
            "theta": round(math.exp(rng.uniform(math.log(2), math.log(64))), 1), "dtype": dtype}


# ---- inputs ----------------------------------------------------------------------
def _shear(n, batch, dtype, seed):
    """Shear maps [batch, n, n] (batch 0: one [n, n] map) on the GPU."""
    g = torch.Generator(device=DEV).manual_seed(int(seed))
    ky = torch.fft.fftfreq(n, 1.0 / n, device=DEV, dtype=dtype)[:, None]
    kx = torch.fft.rfftfreq(n, 1.0 / n, device=DEV, dtype=dtype)[None, :]
    k2 = (kx * kx + ky * ky).clamp_(min=1.0)
    out = torch.empty((2, max(1, batch), n, n), device=DEV, dtype=dtype)
    for b in range(max(1, batch)):
        f = torch.fft.rfft2(torch.randn((n, n), device=DEV, dtype=dtype, generator=g)) / k2.sqrt()
        f[0, 0] = 0
        f *= 0.02 / torch.fft.irfft2(f, s=(n, n)).std()
        out[0, b] = torch.fft.irfft2(f * ((kx * kx - ky * ky) / k2), s=(n, n))
        out[1, b] = torch.fft.irfft2(f * (2 * kx * ky / k2), s=(n, n))
    out += 0.1 * torch.randn(out.shape, device=DEV, dtype=dtype, generator=g)
    g1, g2 = out[0], out[1]
    return (g1[0], g2[0]) if batch == 0 else (g1, g2)


def _kappa(n, batch, dtype, seed):
    g = torch.Generator(device=DEV).manual_seed(int(seed))
    k = torch.fft.fftfreq(n, 1.0 / n, device=DEV, dtype=dtype)
    k2 = (k[: n // 2 + 1][None, :] ** 2 + k[:, None] ** 2).clamp_(min=1.0)
    out = torch.empty((batch, n, n), device=DEV, dtype=dtype)
    for b in range(batch):
        f = torch.fft.rfft2(torch.randn((n, n), device=DEV, dtype=dtype, generator=g)) / k2.sqrt()
        f[0, 0] = 0
        m = torch.fft.irfft2(f, s=(n, n))
        out[b] = m * (0.02 / m.std())
    return out.add_(torch.randn(out.shape, device=DEV, dtype=dtype, generator=g), alpha=0.07)


def _mask(n, dtype, seed):
    """0/1 weights: about 15 % of the field in masked discs and one bad column pair."""
    g = torch.Generator().manual_seed(int(seed) + 7)
    y = torch.arange(n, device=DEV, dtype=torch.float32)
    w = torch.ones((n, n), device=DEV, dtype=dtype)
    r_max, area = max(2.0, n / 32), 0.0
    while area < 0.16 * n * n:
        cy, cx, u = torch.rand(3, generator=g).tolist()
        r = math.exp(math.log(2.0) + u * math.log(r_max / 2.0))
        y0, y1 = max(0, int(cy * n - r)), min(n, int(cy * n + r) + 2)
        x0, x1 = max(0, int(cx * n - r)), min(n, int(cx * n + r) + 2)
        w[y0:y1, x0:x1][(y[y0:y1, None] - cy * n) ** 2 + (y[None, x0:x1] - cx * n) ** 2 <= r * r] = 0
        area += math.pi * r * r
    c = int(torch.randint(0, n - 2, (1,), generator=g))
    w[:, c:c + 2] = 0
    return w


def _pyramid(n, J, batch, dtype, seed):
    """Bands as they come from noisy maps: rms falling with scale, mildly skewed."""
    g = torch.Generator(device=DEV).manual_seed(int(seed))
    x = torch.randn((batch, J, n, n), device=DEV, dtype=dtype, generator=g)
    x += 0.05 * x * x
    x *= (0.06 * 0.45 ** torch.arange(J, device=DEV, dtype=dtype))[None, :, None, None]
    return x


def prepare(case, seed):
    c, dt = case, DTYPES[case["dtype"]]
    s = {"case": c, "boundary": fm.FM_PERIODIC if c.get("periodic") else fm.FM_MIRROR}
    if c["kind"] == "starlet":
        s["kappa"] = _kappa(c["n"], c["batch"], dt, seed)
    elif c["kind"] == "moments":
        s["pyramid"] = _pyramid(c["n"], c["J"], c["batch"], dt, seed)
    else:
        s["g1"], s["g2"] = _shear(c["n"], c.get("batch", 0), dt, seed)
    if c["kind"] == "masked":
        s["weight"] = _mask(c["n"], dt, seed)
    if c["kind"] == "noise":
        s["seed"] = 1000 + int(seed)
    if c.get("keep"):
        s["out"] = torch.empty((c["batch"], c["J"], c["n"], c["n"]), device=DEV, dtype=dt)
    return s


# ---- one pass --------------------------------------------------------------------
def run(state):
    s, c = state, state["case"]
    kind = c["kind"]
    if kind == "map":
        return fm.fm_map_starlet(s["g1"], s["g2"], c["J"], boundary=s["boundary"], out=s.get("out"))
    if kind == "ks":
        return fm.fm_ks_invert(s["g1"], s["g2"], with_b=c["with_b"])
    if kind == "starlet":
        return fm.fm_starlet_forward(s["kappa"], c["J"], boundary=s["boundary"])
    if kind == "noise":
        var, snr = fm.fm_map_noise(s["g1"], s["g2"], c["J"], c["R"], s["seed"], boundary=s["boundary"])
        # kept beside the maps it belongs to, in their type
        return {"variance": var.to(s["g1"].dtype), "snr": snr}
    if kind == "expected":
        return fm.fm_map_noise_expected(s["g1"], s["g2"], c["J"])
    if kind == "direct":
        return fm.fm_map_direct(s["g1"], s["g2"], FILTERS[c["filter"]][0], c["theta"])
    if kind == "masked":
        return fm.fm_map_direct_masked(s["g1"], s["g2"], s["weight"], FILTERS[c["filter"]][0], c["theta"], coverage=True)
    return fm.fm_band_moments(s["pyramid"])


# ---- what a pass cannot do without -------------------------------------------------
def _fft_flops(n, maps):
    return maps * 2 * 5.0 * n * n * 2 * math.log2(n)  # there and back, complex


def work(case):
    c = case
    es = 8 if c["dtype"] == "f64" else 4
    n, J, batch = c["n"], c.get("J", 0), c.get("batch", 1)
    px = float(n) * n * batch
    lift = 22.0 * px * max(0, J - 1)  # two 5-tap filters and a difference a scale
    if c["kind"] == "map":
        return {"bytes": px * es * (2 + J), "flops": _fft_flops(n, batch) + lift}
    if c["kind"] == "ks":
        return {"bytes": px * es * (4 if c["with_b"] else 3), "flops": _fft_flops(n, batch)}
    if c["kind"] == "starlet":
        return {"bytes": px * es * (1 + J), "flops": lift}
    if c["kind"] == "noise":
        return {"bytes": px * (2 * es + (J - 1) * (8 + es)), "flops": c["R"] * (_fft_flops(n, 1) + lift + 3 * px * (J - 1))}
    if c["kind"] == "expected":
        return {"bytes": px * es * (1 + J), "flops": _fft_flops(n, J + 1) + 2 * lift}
    if c["kind"] == "moments":
        return {"bytes": px * es * J, "flops": 7 * px * J}
    taps = math.pi * (FILTERS[c["filter"]][1] * c["theta"]) ** 2
    if c["kind"] == "masked":
        return {"bytes": px * es * 4 + n * n * es, "flops": px * taps * 5}
    return {"bytes": px * es * 3, "flops": px * taps * 4}


# ---- the same in 64 bits, in plain torch --------------------------------------------
def _freq(n):
    k = torch.fft.fftfreq(n, 1.0 / n, device=DEV, dtype=torch.float64)
    return k[None, :], k[:, None]


def _ks64(g1, g2):
    k1, k2 = _freq(g1.shape[-1])
    den = k1 * k1 + k2 * k2
    den[0, 0] = 1.0
    d = torch.complex((k1 * k1 - k2 * k2) / den, -2 * k1 * k2 / den)  # conj(D); 0 at k = 0
    return torch.fft.ifft2(torch.fft.fft2(torch.complex(g1.double(), g2.double())) * d)


def _smooth(c, step, periodic, axis):
    n = c.shape[axis]
    i = torch.arange(n, device=DEV)
    out = 0.375 * c
    for h, off in ((0.25, step), (0.25, -step), (0.0625, 2 * step), (0.0625, -2 * step)):
        j = i + off
        if periodic:
            j = j % n
        else:
            j = j.abs() % (2 * (n - 1))
            j = torch.where(j >= n, 2 * (n - 1) - j, j)
        out += h * c.index_select(axis, j)
    return out


def _starlet64(kappa, J, periodic):
    c, out = kappa.double(), torch.empty((J,) + tuple(kappa.shape), device=DEV, dtype=torch.float64)
    for j in range(1, J):
        nxt = _smooth(_smooth(c, 1 << (j - 1), periodic, 1), 1 << (j - 1), periodic, 0)
        out[j - 1] = c - nxt
        c = nxt
    out[J - 1] = c
    return out


def _rotated(g1, g2, seed, r):
    """Realisation r: every pixel's shear turned by 2 pi u, u from SplitMix64 at the pixel's counter."""
    n = g1.shape[-1]

    def i64(v):
        v &= (1 << 64) - 1
        return v - (1 << 64) if v >> 63 else v

    def shr(z, k):
        return (z >> k) & ((1 << (64 - k)) - 1)

    z = (torch.arange(n * n, device=DEV, dtype=torch.int64) + (r * n * n + 1)) * i64(0x9E3779B97F4A7C15) + i64(seed)
    z = (z ^ shr(z, 30)) * i64(0xBF58476D1CE4E5B9)
    z = (z ^ shr(z, 27)) * i64(0x94D049BB133111EB)
    u = shr(z ^ shr(z, 31), 40).double().reshape(n, n) * 2.0**-24
    w = torch.complex(g1.double(), g2.double()) * torch.polar(torch.ones_like(u), 2 * math.pi * u)
    return w.real, w.imag


def _q(name, theta, r):
    """Q(|d|) of the filters of the paper's Sec. 4.1 and 4.2."""
    if name == "s98":
        x2 = np.minimum((r / theta) ** 2, 1.0)
        return 4.0 * 5.0 / (math.pi * theta**2) * x2 * (1.0 - x2) ** 3
    if name == "jbj04":
        x = 0.5 * (r / theta) ** 2
        return x * np.exp(-x) / theta**2
    e = r / theta
    a = lambda v: np.abs(v) ** 3  # noqa: E731
    s = -279.0 * e * e * a(e)
    for sg in (1.0, -1.0):
        s = s + 8.0 * (1 + sg * 6 * e + 24 * e * e) * a(0.5 - sg * e)
        s = s - 9.0 * (1 + sg * 3 * e + 6 * e * e) * a(1.0 - sg * e)
        s = s + (1 + sg * 1.5 * e + 1.5 * e * e) * a(2.0 - sg * e)
    return s / (45.0 * e * e) / theta**2


def _correlate(taps, maps, R):
    """sum over d of taps[d] maps[x + d], zero outside the field, through FFTs of the padded field."""
    n = maps.shape[-1]
    m = n + R
    k = torch.zeros((max(m, 2 * R + 1),) * 2, dtype=torch.float64, device=DEV)
    i = torch.arange(-R, R + 1, device=DEV) % k.shape[0]
    k[i[:, None], i[None, :]] = torch.from_numpy(taps).to(DEV)
    f = torch.fft.rfft2(k).conj() * torch.fft.rfft2(maps.double(), s=tuple(k.shape))
    return torch.fft.irfft2(f, s=tuple(k.shape))[..., :n, :n]


def _direct64(c, s):
    theta = c["theta"]
    cut = FILTERS[c["filter"]][1] * theta
    R = int(math.floor(cut))
    d = np.arange(-R, R + 1, dtype=np.float64)
    dx, dy = d[None, :], d[:, None]
    r2 = dx * dx + dy * dy
    disc = (r2 > 0) & (r2 <= cut * cut)
    r2s = np.where(r2 > 0, r2, 1.0)
    q = np.where(disc, _q(c["filter"], theta, np.sqrt(r2s)), 0.0)
    a, b = -q * (dx * dx - dy * dy) / r2s, -q * 2 * dx * dy / r2s
    w = s["weight"].double() if "weight" in s else 1.0
    m = _correlate(a, s["g1"].double() * w, R) + _correlate(b, s["g2"].double() * w, R)
    if "weight" not in s:
        return m
    n_r = float(disc.sum())
    data = _correlate(disc.astype(np.float64), s["weight"], R).round()
    m = torch.where(data > 0, n_r * m / data.clamp(min=1.0), torch.zeros_like(m))
    return m, (data / n_r).expand(m.shape)


def exact(case, seed):
    c = case
    s = prepare(c, seed)
    J, periodic = c.get("J", 0), bool(c.get("periodic"))
    if c["kind"] == "map":
        s.pop("out", None)
        out = torch.empty((c["batch"], J, c["n"], c["n"]), device=DEV, dtype=torch.float64)
        for b in range(c["batch"]):
            out[b] = _starlet64(_ks64(s["g1"][b], s["g2"][b]).real, J, periodic)
        return out
    if c["kind"] == "ks":
        k = torch.stack([_ks64(s["g1"][b], s["g2"][b]) for b in range(c["batch"])])
        return k.real, k.imag if c["with_b"] else None
    if c["kind"] == "starlet":
        return torch.stack([_starlet64(m, J, periodic) for m in s["kappa"]])
    if c["kind"] == "noise":
        bands = lambda a, b: _starlet64(_ks64(a, b).real, J, periodic)[:-1]  # noqa: E731
        data = bands(s["g1"], s["g2"])
        s1, s2 = torch.zeros_like(data), torch.zeros_like(data)
        for r in range(c["R"]):
            w = bands(*_rotated(s["g1"], s["g2"], s["seed"], r))
            s1 += w
            s2 += w * w
        var = (s2 - s1 * s1 / c["R"]) / (c["R"] - 1)
        return {"variance": var, "snr": data / var.sqrt()}
    if c["kind"] == "expected":
        one = torch.zeros((c["n"], c["n"]), device=DEV, dtype=torch.float64)
        zero = torch.zeros_like(one)
        one[0, 0] = 1.0
        k2 = sum(_starlet64(_ks64(*p).real, J, True)[:-1] ** 2 for p in ((one, zero), (zero, one)))
        p = s["g1"].double() ** 2 + s["g2"].double() ** 2
        return 0.5 * torch.fft.irfft2(torch.fft.rfft2(k2) * torch.fft.rfft2(p), s=(c["n"], c["n"]))
    if c["kind"] == "moments":
        x = s["pyramid"].double()
        mean = x.mean(dim=(-1, -2))
        d = x - mean[..., None, None]
        m2, m3, m4 = ((d**p).mean(dim=(-1, -2)) for p in (2, 3, 4))
        return torch.stack([mean, m2, m3 / m2**1.5, m4 / m2**2 - 3.0], dim=-1)
    return _direct64(c, s)
