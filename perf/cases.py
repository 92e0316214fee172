"""What the speed of this framework is judged by: solves through its public
entry points, over the plane sizes, point counts, precisions and point
distributions that its users have.

A case is a dict of plain values.  `call` says which entry point it takes:

  plane  one NU-ASM / NU-FRE solve of type 1 or 2 on a plan kept by the caller
  type3  one solve between two non-uniform point sets (two plans)
  batch  several planes of mixed sizes, recorded once and replayed
  rs     the Rayleigh-Sommerfeld direct sum that the solves are compared with

Inputs are drawn on the GPU from the seed.  `exact` evaluates the definitions
in 64-bit torch / numpy: plane FFTs, the transfer function on the modes, and
a gridded non-uniform transform with 16 taps (error about 1e-14).
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1308_6644_gb300 as lib

DEV = "cuda"


def listed():
    asm = dict(call="plane", kind="asm", kernel="es", tol=0.0, weights=False, ox=0.0)
    fre = dict(asm, kind="fresnel")
    return [
        # the smallest plane that is solved: 64 x 64, its core sampled twice as densely, double precision
        dict(asm, name="asm1_small_f64", type=1, prec="f64", n=64, m=4864, points="core", lam=633e-9, z=0.05,
             pitch=10e-6),
        # the paper's own experiment: 256 x 256 samples with a pitch per quadrant and area weights
        dict(asm, name="asm1_quadrant_f32", type=1, prec="f32", n=256, m=65536, points="quadrant", lam=500e-9, z=8e-3,
             pitch=5e-6, weights=True),
        # a hologram plane to points whose pitch grades towards the edge, off axis
        dict(asm, name="asm2_graded_f32", type=2, prec="f32", n=1024, m=1048576, points="graded", lam=532e-9, z=0.2,
             pitch=8e-6, ox=1e-3),
        # a large plane and clustered points, paraxial, each direction in each precision
        dict(fre, name="fre1_clustered_f32", type=1, prec="f32", n=2048, m=4194304, points="clustered", lam=633e-9,
             z=1.0, pitch=4e-6),
        dict(fre, name="fre2_clustered_f32", type=2, prec="f32", n=2048, m=4194304, points="clustered", lam=633e-9,
             z=1.0, pitch=4e-6),
        dict(fre, name="fre1_clustered_f64", type=1, prec="f64", n=2048, m=4194304, points="clustered", lam=633e-9,
             z=1.0, pitch=4e-6),
        dict(fre, name="fre2_clustered_f64", type=2, prec="f64", n=2048, m=4194304, points="clustered", lam=633e-9,
             z=1.0, pitch=4e-6),
        # the largest plane that is served, an odd number of points on a jittered lattice
        dict(asm, name="asm1_largest_f32", type=1, prec="f32", n=4096, m=9999999, points="jitter", lam=532e-9, z=0.3,
             pitch=8e-6),
        # two non-uniform planes: a clustered source and a graded destination, ragged counts
        dict(asm, call="type3", name="asm3_mixed_f32", type=3, prec="f32", n=512, m=200003, m2=150001,
             points="clustered", points2="graded", lam=532e-9, z=0.05, pitch=8e-6),
        # depth layers / colour channels of mixed sizes replayed as one batch
        dict(call="batch", name="batch_mixed_f32", prec="f32", planes=12, n=256, n_max=1024),
        # the accuracy reference: the paper's 256 x 256 samples, and its double-precision form at 128 x 128
        dict(call="rs", name="rs_quadrant_f32", prec="f32", m=65536, m2=65536, side=1.28e-3, lam=500e-9, z=8e-3,
             ox=0.0),
        dict(call="rs", name="rs_quadrant_f64", prec="f64", m=16384, m2=16384, side=0.64e-3, lam=500e-9, z=8e-3,
             ox=0.0),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    """One more case: planes of 32 to 4096 (double precision to 2048) samples a side with a quarter to
    four times as many points, rarely a batch or a type-3 pair, and direct sums of 10^3 to 65536 points."""
    call = rng.choices(["plane", "type3", "batch", "rs"], [9, 2, 1, 2])[0]
    prec = rng.choice(["f32", "f32", "f64"])
    lam = rng.choice([450e-9, 500e-9, 532e-9, 633e-9])
    if call == "rs":
        top = 65536 if prec == "f32" else 16384
        m, m2 = int(_log(rng, 1000, top)), int(_log(rng, 1000, top))
        return dict(call="rs", prec=prec, m=m, m2=m2, side=rng.uniform(0.2e-3, 1.2e-3), lam=lam,
                    z=_log(rng, 8e-3, 0.128), ox=rng.choice([0.0, 20e-6]))
    if call == "batch":
        return dict(call="batch", prec="f32", planes=rng.randint(3, 16), n=rng.choice([64, 128, 256]),
                    n_max=rng.choice([512, 1024]))
    n = 1 << (rng.randint(5, 12) if prec == "f32" else rng.randint(5, 11))
    kind = rng.choice(["asm", "asm", "fresnel"])
    pitch = rng.choice([4e-6, 5e-6, 8e-6, 10e-6])
    gauss = rng.random() < 0.1
    top = 10 ** 7 if prec == "f32" else 5 * 10 ** 6
    if gauss or call == "type3":
        top //= 5
    points = rng.choice(["jitter", "graded", "clustered", "lattice"])
    m = max(1, min(top, int(_log(rng, 0.25, 4.0) * n * n)))
    # a distance at which the plane's own sampling resolves the propagation
    z = n * pitch * pitch / lam * _log(rng, 0.3, 3.0)
    case = dict(call=call, type=rng.choice([1, 2]), kind=kind, prec=prec, n=n, m=m, points=points, lam=lam, z=z,
                pitch=pitch, kernel="gaussian" if gauss else "es",
                tol=rng.choice([0.0, 0.0, 1e-10 if prec == "f64" else 1e-5]) if not gauss else 0.0,
                weights=rng.random() < 0.3 and points != "lattice", ox=rng.choice([0.0, 0.1 * n * pitch]))
    if call == "type3":
        case |= dict(type=3, points2=rng.choice(["jitter", "graded", "clustered"]),
                     m2=max(1, min(top, int(_log(rng, 0.25, 4.0) * n * n))))
    return case


# ------------------------------------------------------------------ inputs
def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(seed)


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device=DEV, dtype=torch.float64)


def _lattice_t(m):
    """m points of a near-square lattice over (-1, 1)^2, row by row."""
    side = max(1, math.isqrt(m - 1) + 1) if m > 1 else 1
    i = torch.arange(m, device=DEV)
    rows = -(-m // side)
    return ((i % side).double() + 0.5) * (2.0 / side) - 1, ((i // side).double() + 0.5) * (2.0 / rows) - 1, 2.0 / side


def _lattice_shape(m):
    side = max(1, math.isqrt(m))   # a square plane of at most m samples
    return side, side


def _points(g, how, n, pitch, m):
    """(x, y, relative areas) of m points inside the window of an n x n plane."""
    half = 0.5 * n * pitch
    area = None
    if how == "quadrant":   # pitch 0.9 / 0.8 / 0.7 / 1.0 in the four quadrants, outwards from the centre
        h = n // 2
        i = (torch.arange(h, device=DEV, dtype=torch.float64) + 0.5) * pitch
        xs, ys, ar = [], [], []
        for sx, sy, s in ((1, 1, 0.9), (-1, 1, 0.8), (-1, -1, 0.7), (1, -1, 1.0)):
            yy, xx = torch.meshgrid(i * s * sy, i * s * sx, indexing="ij")
            xs.append(xx.reshape(-1))
            ys.append(yy.reshape(-1))
            ar.append(torch.full_like(xs[-1], s * s))
        x, y, area = torch.cat(xs), torch.cat(ys), torch.cat(ar)
    elif how == "core":     # a jittered lattice whose central n/4 x n/4 samples are twice as dense per axis
        c = n // 4
        k = torch.arange(n, device=DEV) - n // 2
        yy, xx = torch.meshgrid(k, k, indexing="ij")
        keep = ~(((xx + 0.5).abs() < c / 2) & ((yy + 0.5).abs() < c / 2))
        k2 = (torch.arange(2 * c, device=DEV) - c) * 0.5
        y2, x2 = torch.meshgrid(k2, k2, indexing="ij")
        x = torch.cat([xx[keep].double(), x2.reshape(-1).double()])
        y = torch.cat([yy[keep].double(), y2.reshape(-1).double()])
        j = torch.full_like(x, 0.4)
        j[-4 * c * c:] = 0.2
        x = (x + j * (2 * _rand(g, len(x)) - 1)) * pitch
        y = (y + j * (2 * _rand(g, len(y)) - 1)) * pitch
    elif how == "graded":   # the pitch doubles from half at the centre to twice at the edge
        tx, ty, base = _lattice_t(m)
        rho = torch.maximum(tx.abs(), ty.abs())
        local = 0.5 * (1 + 3 * rho * rho) * base * 0.3
        x = (tx * 0.5 * (1 + rho * rho) + local * (2 * _rand(g, m) - 1)) * half
        y = (ty * 0.5 * (1 + rho * rho) + local * (2 * _rand(g, m) - 1)) * half
    elif how == "clustered":   # three quarters in four Gaussian patches, the rest all over the window
        mc = (3 * m) // 4
        centres = (2 * _rand(g, 4, 2) - 1) * 0.6 * half
        which = torch.randint(0, 4, (mc,), generator=g, device=DEV)
        xy = centres[which] + 0.2 * half * torch.randn(mc, 2, generator=g, device=DEV, dtype=torch.float64)
        xy = torch.cat([xy, (2 * _rand(g, m - mc, 2) - 1) * half])
        xy = xy[torch.randperm(m, generator=g, device=DEV)]
        x, y = xy[:, 0].contiguous(), xy[:, 1].contiguous()
    elif how == "lattice":   # a plane of another pitch (scaled diffraction)
        nx, ny = _lattice_shape(m)
        p2 = 2 * half / max(nx, ny)
        j, i = torch.meshgrid(torch.arange(ny, device=DEV).double(), torch.arange(nx, device=DEV).double(),
                              indexing="ij")
        x, y = (-half + i * p2).reshape(-1), (-half + j * p2).reshape(-1)
    else:                    # jitter
        tx, ty, base = _lattice_t(m)
        x = (tx + 0.4 * base * (2 * _rand(g, m) - 1)) * half
        y = (ty + 0.4 * base * (2 * _rand(g, m) - 1)) * half
    top = half * (1 - 1e-12)
    return x.clamp(-half, top), y.clamp(-half, top), area


def _phasor(g, count, prec):
    v = torch.polar(_rand(g, count), 2 * math.pi * _rand(g, count))
    return v.to(torch.complex128 if prec == "f64" else torch.complex64)


def _beam(x, y, w0, prec):
    return torch.exp(-(x * x + y * y) / (w0 * w0)).to(torch.complex128 if prec == "f64" else torch.complex64)


def _plane_inputs(c, seed):
    """Points, weights and source values of one plane (a Gaussian beam where the solve is paraxial)."""
    g = _gen(seed)
    n, pitch = c["n"], c["pitch"]
    x, y, area = _points(g, c["points"], n, pitch, c["m"])
    w = None
    if c["weights"]:
        w = area if area is not None else 0.5 + _rand(g, len(x))
    if c["kind"] == "fresnel":
        w0 = n * pitch / 16
        if c["type"] != 2:
            src = _beam(x, y, w0, c["prec"])
        else:
            k = (torch.arange(n, device=DEV) - n // 2) * pitch
            gy, gx = torch.meshgrid(k, k, indexing="ij")
            src = _beam(gx, gy, w0, c["prec"]).reshape(-1)
    else:
        src = _phasor(g, len(x) if c["type"] != 2 else n * n, c["prec"])
    return x, y, w, src


def _params(c):
    return lib.make_params(c["n"], c["pitch"], c["lam"], c["z"], ox=c["ox"], kind=c["kind"], prec=c["prec"],
                           tol=c["tol"], kernel=c["kernel"])


def _plan(c, x, y, w):
    if c["points"] == "lattice":
        nx, ny = _lattice_shape(c["m"])
        half = 0.5 * c["n"] * c["pitch"]
        return lib.nuasm_plan_lattice(_params(c), nx, ny, 2 * half / max(nx, ny), -half, -half)
    return lib.nuasm_plan(_params(c), x, y, w)


def _planes(c):
    """The planes of a batch: sizes n, 2n, ... n_max in turn, both directions, 1/4 to 2 points a sample."""
    sizes = [c["n"] << k for k in range(8) if c["n"] << k <= c["n_max"]]
    out = []
    for i in range(c["planes"]):
        n = sizes[i % len(sizes)]
        out.append(dict(call="plane", type=1 + (i // len(sizes) + i) % 2, kind="asm", prec=c["prec"], n=n,
                        m=max(1, int(n * n * 2.0 ** (i % 4 - 2)) - i), points=("jitter", "clustered")[i % 2],
                        lam=(450e-9, 532e-9, 633e-9)[i % 3], z=0.02 + 0.03 * i, pitch=8e-6, kernel="es", tol=0.0,
                        weights=False, ox=0.0))
    return out


def _out_count(c):
    return c["n"] ** 2 if c["type"] == 1 else c["m2"] if c["type"] == 3 else _count(c)


def _count(c):
    if c["points"] == "lattice":
        nx, ny = _lattice_shape(c["m"])
        return nx * ny
    return c["m"]


def _rs_inputs(c, seed):
    g = _gen(seed)
    x1, y1, _ = _points(g, "jitter", 1, c["side"], c["m"])
    x2, y2, _ = _points(g, "jitter", 1, c["side"], c["m2"])
    area = (0.5 + _rand(g, c["m"])) * (c["side"] ** 2 / c["m"])
    return x1, y1, _phasor(g, c["m"], c["prec"]), area, x2, y2


def prepare(case, seed):
    c = case
    cdt = torch.complex128 if c["prec"] == "f64" else torch.complex64
    if c["call"] == "rs":
        a = _rs_inputs(c, seed)
        p = lib.make_params(16, 1e-6, c["lam"], c["z"], ox=c["ox"], prec=c["prec"])
        return dict(case=c, params=p, args=a, out=torch.empty(c["m2"], dtype=cdt, device=DEV))
    if c["call"] == "batch":
        items = []
        for i, p in enumerate(_planes(c)):
            x, y, w, src = _plane_inputs(p, 1000 * seed + i)
            items.append((_plan(p, x, y, w), p["type"], src, torch.empty(_out_count(p), dtype=cdt, device=DEV)))
        return dict(case=c, items=items, batch=lib.nuasm_batch_create(items))
    x, y, w, src = _plane_inputs(c, seed)
    s = dict(case=c, src=src, plan=_plan(c, x, y, w), out=torch.empty(_out_count(c), dtype=cdt, device=DEV))
    if c["call"] == "type3":
        x2, y2, _ = _points(_gen(seed + 77), c["points2"], c["n"], c["pitch"], c["m2"])
        s["dst"] = lib.nuasm_plan(_params(c), x2, y2)
    return s


def run(state):
    c = state["case"]
    if c["call"] == "rs":
        return lib.nuasm_rs_direct(state["params"], *state["args"], state["out"])
    if c["call"] == "batch":
        lib.nuasm_batch_execute(state["batch"])
        return [it[3] for it in state["items"]]
    if c["call"] == "type3":
        f = lib.nuasm3_execute if c["kind"] == "asm" else lib.nufresnel3_execute
        return f(state["plan"], state["dst"], state["src"], state["out"])
    if c["kind"] == "fresnel":
        return lib.nufresnel_execute(state["plan"], c["type"], state["src"], state["out"])
    f = lib.nuasm1_execute if c["type"] == 1 else lib.nuasm2_execute
    return f(state["plan"], state["src"], state["out"])


# ------------------------------------------------------------------ work
def work(case):
    """Values in and out once, 4 bytes of cell and two fractions a point; transforms at 5 L log2 L a line
    (of the padded plane, twice for the oversampled side), a complex multiply-add a kernel tap, and 40
    operations a pair of the direct sum."""
    c = case
    cb = 16 if c["prec"] == "f64" else 8
    if c["call"] == "rs":
        return {"bytes": (c["m"] + c["m2"]) * (16 + cb) + 8 * c["m"], "flops": 40.0 * c["m"] * c["m2"]}
    if c["call"] == "batch":
        parts = [work(p) for p in _planes(c)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    n, np_ = c["n"], 2 * c["n"]
    w = lib.nuasm_kernel_shape(c["tol"], 1 if c["prec"] == "f64" else 0, 1 if c["kernel"] == "gaussian" else 0)[0]
    pts = _count(c) + c.get("m2", 0)
    line = 5.0 * np_ * math.log2(np_)
    if c["type"] == 3:
        lines, values = 4 * 2 * n + 4 * np_, pts
    else:
        lines, values = 2 * 2 * n + 3 * np_ + n, pts + n * n
    return {"bytes": values * cb + pts * (4 + cb) + (8 * pts if c["weights"] else 0),
            "flops": line * lines + 6.0 * np_ * np_ + 4.0 * w * w * pts}


# ------------------------------------------------------------------ 64-bit values
_W = 16
_BETA = 2.30 * _W


def _es(t):
    return torch.exp(_BETA * (torch.sqrt((1 - (2 * t / _W) ** 2).clamp(min=0)) - 1))


def _es_hat(nu):
    t, wt = np.polynomial.legendre.leggauss(200)
    t, wt = (t + 1) * _W / 4, wt * _W / 4
    f = np.exp(_BETA * (np.sqrt(1 - (2 * t / _W) ** 2) - 1)) * wt
    return torch.tensor(2 * (np.cos(2 * np.pi * np.outer(nu, t)) @ f), device=DEV)


def _taps(x, pitch, G):
    """Grid cells and kernel values of the 16 taps around each coordinate."""
    gx = 2 * (x / pitch)
    l0 = torch.ceil(gx - _W / 2)
    i = torch.arange(_W, device=DEV, dtype=torch.float64)
    return torch.remainder((l0[:, None] + i).long(), G), _es(l0[:, None] + i - gx[:, None])


def _modes(np_):
    return np.fft.fftfreq(np_, 1.0 / np_)   # k in FFT order


def _nufft1(x, y, v, pitch, np_):
    G = 2 * np_
    grid = torch.zeros(G * G, 2, dtype=torch.float64, device=DEV)
    for a in range(0, len(x), 1 << 18):
        s = slice(a, a + (1 << 18))
        (ix, wx), (iy, wy) = _taps(x[s], pitch, G), _taps(y[s], pitch, G)
        for q in range(_W):
            val = torch.view_as_real(v[s])[:, None, :] * (wy[:, q, None] * wx)[:, :, None]
            grid.index_add_(0, (iy[:, q, None] * G + ix).reshape(-1), val.reshape(-1, 2))
    k = torch.tensor(_modes(np_), device=DEV).long()
    F = torch.fft.fft2(torch.view_as_complex(grid).view(G, G))
    F = F[torch.remainder(k, G)][:, torch.remainder(k, G)]
    h = _es_hat(_modes(np_) / G)
    return F / (h[:, None] * h[None, :])


def _nufft2(S, x, y, pitch, np_):
    G = 2 * np_
    k = torch.tensor(_modes(np_), device=DEV).long()
    h = _es_hat(_modes(np_) / G)
    grid = torch.zeros(G, G, dtype=torch.complex128, device=DEV)
    idx = torch.remainder(k, G)
    grid[idx[:, None], idx[None, :]] = S / (h[:, None] * h[None, :])
    grid = torch.fft.ifft2(grid, norm="forward").reshape(-1)
    out = []
    for a in range(0, len(x), 1 << 18):
        s = slice(a, a + (1 << 18))
        (ix, wx), (iy, wy) = _taps(x[s], pitch, G), _taps(y[s], pitch, G)
        acc = torch.zeros(ix.shape[0], dtype=torch.complex128, device=DEV)
        for q in range(_W):
            acc += wy[:, q] * (grid[iy[:, q, None] * G + ix] * wx).sum(1)
        out.append(acc)
    return torch.cat(out)


def _cis(c):
    """exp(2 pi i c) of an extended-precision phase in cycles."""
    c = (c - np.rint(c)).astype(np.float64)
    return np.exp(2j * np.pi * c)


def _transfer(c, np_):
    """H on the modes in FFT order, 64 bits."""
    L = np.longdouble
    lam, z, pitch = L(c["lam"]), L(c["z"]), L(c["pitch"])
    k = _modes(np_).astype(L)
    f = k / (np_ * pitch)
    axes = []
    for o in (L(0), L(c["ox"])):   # y, x
        if c["kind"] == "fresnel":
            a = np.fft.fft(_cis((k * pitch + o) ** 2 / (2 * lam * z))) * float(pitch)
        else:
            s = float(c["n"] * pitch)
            fd = f.astype(np.float64)
            root = np.sqrt(np.maximum(1 / c["lam"] ** 2 - fd * fd, 0))
            ok = (fd * c["lam"] < 1) & (np.abs(float(o) * root - c["z"] * fd) <= s * root)
            a = _cis(o * f - z * lam * f * f / 2) * ok
        axes.append(torch.tensor(a, device=DEV))
    const = _cis(np.array([z / lam]))[0]
    H = axes[0][:, None] * axes[1][None, :]
    if c["kind"] == "fresnel":
        return H * complex(const / (1j * c["lam"] * c["z"]))
    sv = torch.tensor((lam * f).astype(np.float64) ** 2, device=DEV)
    sv = sv[:, None] + sv[None, :]
    q = sv / (1 + torch.sqrt((1 - sv).clamp(min=0)))
    rest = -c["z"] / (2 * c["lam"]) * q * q
    rest = rest - torch.round(rest)
    return H * torch.polar((sv < 1).double(), 2 * math.pi * rest) * complex(const)


def _exact_plane(c, seed):
    n, np_ = c["n"], 2 * c["n"]
    x, y, w, src = _plane_inputs(c, seed)
    src = src.to(torch.complex128)
    idx = torch.remainder(torch.arange(n, device=DEV) - n // 2, np_)
    H = _transfer(c, np_)
    if c["type"] == 2:
        pad = torch.zeros(np_, np_, dtype=torch.complex128, device=DEV)
        pad[idx[:, None], idx[None, :]] = src.view(n, n)
        return _nufft2(torch.fft.fft2(pad) * H / float(np_) ** 2, x, y, c["pitch"], np_)
    F = _nufft1(x, y, src if w is None else src * w, c["pitch"], np_) * H
    if c["type"] == 3:
        x2, y2, _ = _points(_gen(seed + 77), c["points2"], n, c["pitch"], c["m2"])
        return _nufft2(F / float(np_) ** 2, x2, y2, c["pitch"], np_)
    return torch.fft.ifft2(F)[idx][:, idx].reshape(-1)


def _two_sum(a, b):
    s = a + b
    t = s - a
    return s, (a - (s - t)) + (b - t)


def _sq(a):
    """a^2 as a sum of two doubles."""
    p = a * a
    t = a * 134217729.0
    h = t - (t - a)
    l = a - h
    return p, ((h * h - p) + 2 * h * l) + l * l


def _exact_rs(c, seed):
    """Eq. 10 with r and the phase as sums of two doubles (the phase reaches 10^4 cycles)."""
    x1, y1, v, area, x2, y2 = _rs_inputs(c, seed)
    v = v.to(torch.complex128) * area
    x2 = x2 + c["ox"]
    z, lam = c["z"], c["lam"]
    L = np.longdouble
    zc = L(z) / L(lam)
    zfrac = float(zc - np.rint(zc))
    zz = L(z) * L(z)
    zh, zl = float(zz), float(zz - L(float(zz)))
    il = L(1) / L(lam)
    ih, ilo = float(il), float(il - L(float(il)))
    out = torch.zeros(c["m2"], dtype=torch.complex128, device=DEV)
    step = max(1, (1 << 24) // c["m2"])
    for a in range(0, c["m"], step):
        s = slice(a, a + step)
        dx, dy = x2[:, None] - x1[None, s], y2[:, None] - y1[None, s]
        (p, e), (q, f) = _sq(dx), _sq(dy)
        rho, t = _two_sum(p, q)
        rlo = t + (e + f)
        h, t = _two_sum(rho, torch.full_like(rho, zh))
        lo = t + (rlo + zl)
        r = torch.sqrt(h + lo)
        sh, sl = _sq(r)
        rl = (((h - sh) - sl) + lo) / (2 * r)
        # (r - z) / lambda = rho^2 / ((r + z) lambda)
        dh, dl = _two_sum(r, torch.full_like(r, z))
        dl = dl + rl
        qh = rho / dh
        # remainder of the division, its product split exactly
        t1 = qh * 134217729.0
        qa = t1 - (t1 - qh)
        qb = qh - qa
        t2 = dh * 134217729.0
        da = t2 - (t2 - dh)
        db = dh - da
        prod = qh * dh
        perr = ((qa * da - prod) + qa * db + qb * da) + qb * db
        ql = (((rho - prod) - perr) + rlo - qh * dl) / dh
        ch = qh * ih
        t1 = ih * 134217729.0
        ia = t1 - (t1 - ih)
        ib = ih - ia
        cerr = ((qa * ia - ch) + qa * ib + qb * ia) + qb * ib
        ph = (ch - torch.round(ch)) + (cerr + qh * ilo + ql * ih) + zfrac
        ph = ph - torch.round(ph)
        e = torch.polar(z / (r * r * r), 2 * math.pi * ph)
        k = torch.complex(torch.ones_like(r), -(2 * math.pi / lam) * r) * e
        out += k @ v[s]
    return out / (2 * math.pi)


def exact(case, seed):
    c = case
    if c["call"] == "rs":
        return _exact_rs(c, seed)
    if c["call"] == "batch":
        return [_exact_plane(p, 1000 * seed + i) for i, p in enumerate(_planes(c))]
    return _exact_plane(c, seed)
