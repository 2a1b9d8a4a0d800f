"""The work a user of the framework has it do, as cases that can be timed.

Every case is one interpolation step through the public Python entry points:
new points are set and the fields evaluated there, as each time step of a
semi-Lagrangian model does (the departure points move every step, so both
belong to the step).  ``prepare`` makes what such a program holds before the
step, ``run`` does one step, ``exact`` gives its result in FP64 by plain torch.

Kinds of case
  spectral : points and spectral coefficients on the device (Plan.set_points,
             Plan.execute);
  grid     : samples on the arrival grid instead of coefficients
             (Plan.interpolate_grid);
  gauss    : the same with Gauss-Legendre latitudes;
  semilag  : the whole step of a model on Grid [0]: departure points of the
             wind, the fields carried there, the wind rotated to the arrival
             frame;
  host     : points and coefficients from pinned host memory, values back to it
             (Plan.execute_points_host);
  ensemble : many members on uneven grids in one call (Ensemble.run).
Points are departure points of a smooth wind of at most 80 m/s, one
per arrival-grid point (which crowds them at the poles), or scattered evenly on
the sphere (stations, tracers) in any number and order.  Fields are random with
|k|^-3 spectra and the double Fourier sphere's parities: a scalar, then wind
components.
"""
import functools
import math

import numpy as np
import torch

from paper_2605_01313_gb300 import nufft

WIND = 80.0                                # m/s, the fastest wind
RADIUS = 6.371e6                           # m, the Earth's
TOL = {"f64": 1e-12, "f32": 1e-6}
REAL = {"f64": torch.float64, "f32": torch.float32}
CPLX = {"f64": torch.complex128, "f32": torch.complex64}


def _case(name, kind, dtype, n_lon, n_lat, fields=3, points="departure", count=0, real=True,
          members=1, minutes=30.0):
    """count: scattered points (departure points are one per grid point);
    real: plan option for real fields; members: per grid of an ensemble, whose
    grids halve from n_lon x n_lat three times; minutes: the time step."""
    return {"name": name, "kind": kind, "dtype": dtype, "n_lon": n_lon, "n_lat": n_lat,
            "fields": fields, "points": points, "count": count, "real": real,
            "members": members, "minutes": minutes}


def listed():
    return [
        # the smallest grid of the golden tests: one field, launch latency throughout
        _case("spectral_64x32_f64", "spectral", "f64", 64, 32, fields=1),
        # a one-degree grid (no power of two) with a plan of default options
        _case("spectral_360x180_f32_general", "spectral", "f32", 360, 180, real=False),
        # scattered points in an odd number on a medium grid
        _case("spectral_512x256_f32_scattered", "spectral", "f32", 512, 256, points="scattered",
              count=200003),
        # the paper's shallow-water fields at medium resolution in double precision
        _case("spectral_512x256_f64", "spectral", "f64", 512, 256),
        # the benchmark's workload, single and double precision
        _case("spectral_2048x1024_f32", "spectral", "f32", 2048, 1024),
        _case("spectral_2048x1024_f64", "spectral", "f64", 2048, 1024),
        # the largest grid a plan takes
        _case("spectral_4096x2048_f32", "spectral", "f32", 4096, 2048),
        # a grid-point model in double precision
        _case("grid_1024x512_f64", "grid", "f64", 1024, 512),
        # a model on the Gauss-Legendre grid of spherical harmonics
        _case("gauss_1024x512_f32", "gauss", "f32", 1024, 512),
        # the whole semi-Lagrangian step
        _case("semilag_2048x1024_f32", "semilag", "f32", 2048, 1024),
        # a host model that hands its arrays over
        _case("host_2048x1024_f32", "host", "f32", 2048, 1024),
        # an ensemble of 64 members on four grids, 128 x 64 to 1024 x 512
        _case("ensemble_64_f32", "ensemble", "f32", 1024, 512, members=16),
    ]


def draw(rng):
    kind = rng.choice(["spectral"] * 5 + ["grid", "gauss", "semilag", "host", "ensemble"])
    dtype = rng.choice(["f32", "f32", "f64"])
    if kind in ("gauss", "ensemble"):
        dtype = "f32"
    fields = rng.choice([1, 2, 3, 3, 4])
    if kind in ("grid", "gauss", "semilag"):       # grids whose transforms are powers of two
        n_lat = 2 ** rng.randint(5, {"gauss": 9}.get(kind, 10 if dtype == "f32" else 9))
        n_lon = 2 * n_lat
        if kind == "semilag":
            fields = 3
    elif kind == "ensemble":
        n_lat = 2 ** rng.randint(7, 9)
        n_lon, fields = 2 * n_lat, 3
    else:
        top = 2048 if dtype == "f32" and kind == "spectral" else 1024
        n_lat = int(round(math.exp(rng.uniform(math.log(24), math.log(top)))))
        n_lon = 2 * n_lat if rng.random() < 0.7 else 2 * rng.randint(n_lat // 2, n_lat)
    if n_lat > 1024:
        fields = min(fields, 3)
    real = kind != "spectral" or rng.random() < 0.6
    if not real and n_lat > 512:
        real = dtype == "f64"
    points, count = "departure", 0
    if kind not in ("semilag", "ensemble") and rng.random() < 0.4:
        most = n_lon * n_lat
        points = "scattered"
        count = int(round(math.exp(rng.uniform(math.log(max(1, most // 16)), math.log(most)))))
    return {"kind": kind, "dtype": dtype, "n_lon": n_lon, "n_lat": n_lat, "fields": fields,
            "points": points, "count": count, "real": real,
            "members": rng.randint(2, 16) if kind == "ensemble" else 1,
            "minutes": round(rng.uniform(5.0, 60.0), 2)}


# ------------------------------------------------------------------ inputs

def _gen(seed, salt):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed * 1000003 + salt)
    return g


def _parity(fields):
    return [1 if f == 0 else -1 for f in range(fields)]


def _spectrum(gen, members, parity, n_lon, n_lat):
    """(members, fields, 2 n_lat, n_lon) FP64 coefficients of real fields with
    amplitudes |k|^-3, scaled to 100 (scalar) or 20 (wind component) r.m.s."""
    n2, n1 = 2 * n_lat, n_lon
    n = (torch.arange(n2, device="cuda") - n_lat).double()[:, None]
    m = (torch.arange(n1, device="cuda") - n_lon // 2).double()[None, :]
    amp = (n * n + m * m).clamp(min=1.0) ** -1.5
    amp[0, :] = 0.0                                   # Nyquist row and column
    amp[:, 0] = 0.0
    par = torch.tensor(parity, device="cuda", dtype=torch.float64)[:, None, None]
    sgn = par * torch.where(m % 2 == 0, 1.0, -1.0)
    c = torch.randn((members, len(parity), n2, n1), generator=gen, device="cuda",
                    dtype=torch.complex128) * amp

    def mirror(x, dims):
        return torch.roll(torch.flip(x, dims), [1] * len(dims), dims)

    # f(phi + pi, -theta) = parity f(phi, theta), then real values
    c = 0.5 * (c + sgn * mirror(c, (-2,)))
    c = 0.5 * (c + torch.conj(mirror(c, (-2, -1))).resolve_conj())
    rms = torch.sqrt((c.real ** 2 + c.imag ** 2).sum(dim=(-2, -1), keepdim=True))
    return c * (torch.where(par > 0, 100.0, 20.0) / rms)


def _xyz(lon, colat):
    s = torch.sin(colat)
    return torch.stack([s * torch.cos(lon), s * torch.sin(lon), torch.cos(colat)], -1)


def _lonlat(r):
    lon = torch.remainder(torch.atan2(r[..., 1], r[..., 0]), 2 * math.pi)
    lon = torch.where(lon >= 2 * math.pi, torch.zeros_like(lon), lon)
    return lon, torch.atan2(torch.hypot(r[..., 0], r[..., 1]), r[..., 2])


def _arrival(n_lon, n_lat):
    colat = (torch.arange(n_lat, device="cuda", dtype=torch.float64) + 0.5) * (math.pi / n_lat)
    lon = torch.arange(n_lon, device="cuda", dtype=torch.float64) * (2 * math.pi / n_lon)
    cc, ll = torch.meshgrid(colat, lon, indexing="ij")
    return ll.reshape(-1), cc.reshape(-1)


def _wind(gen, r):
    """A smooth tangential wind at unit vectors r, largest speed 1: a rotation
    about a tilted axis plus a divergent quadratic part."""
    axis = torch.randn(3, generator=gen, device="cuda", dtype=torch.float64)
    a = torch.randn((3, 3), generator=gen, device="cuda", dtype=torch.float64)
    axis = axis / axis.norm()
    g = r @ (0.15 * (a + a.T))
    v = torch.linalg.cross(axis.expand_as(r), r) + g - (g * r).sum(-1, keepdim=True) * r
    return v / v.norm(dim=-1).max()


def _points(gen, case, n_lon, n_lat):
    if case["points"] == "scattered":
        u = torch.rand((2, case["count"]), generator=gen, device="cuda", dtype=torch.float64)
        return (2 * math.pi * u[0]).contiguous(), torch.acos(2 * u[1] - 1).contiguous()
    r = _xyz(*_arrival(n_lon, n_lat))
    v = _wind(gen, r) * (WIND * 60.0 * case["minutes"] / RADIUS)
    d = v.norm(dim=-1, keepdim=True)
    lon, colat = _lonlat(torch.cos(d) * r - torch.sin(d) * v / d.clamp(min=1e-300))
    return lon.contiguous(), colat.contiguous()


@functools.lru_cache(maxsize=8)
def _gauss_colat(n_lat):
    return np.arccos(np.polynomial.legendre.leggauss(n_lat)[0][::-1])


def _row_colat(case):
    if case["kind"] == "gauss":
        return torch.from_numpy(_gauss_colat(case["n_lat"]).copy()).cuda()
    return (torch.arange(case["n_lat"], device="cuda", dtype=torch.float64) + 0.5) * (
        math.pi / case["n_lat"])


def _modes(n):
    return (torch.arange(n, device="cuda") - n // 2).double()


def _samples(case, c):
    """Real (fields, n_lat, n_lon) samples on the arrival grid of coefficients c."""
    e = torch.polar(torch.ones((), device="cuda", dtype=torch.float64),
                    _row_colat(case)[:, None] * _modes(2 * case["n_lat"])[None, :])
    col = torch.stack([e @ f for f in c])
    return (torch.fft.ifft(torch.fft.ifftshift(col, dim=-1), dim=-1) * case["n_lon"]).real


def _frame(n_lon, n_lat):
    lon, colat = _arrival(n_lon, n_lat)
    zero = torch.zeros_like(lon)
    east = torch.stack([-torch.sin(lon), torch.cos(lon), zero], -1)
    north = torch.stack([-torch.cos(colat) * torch.cos(lon), -torch.cos(colat) * torch.sin(lon),
                         torch.sin(colat)], -1)
    return _xyz(lon, colat), east, north


def _inputs(case, seed):
    """Everything a pass reads, on the device, in the case's precision."""
    n_lon, n_lat, rd, cd = case["n_lon"], case["n_lat"], REAL[case["dtype"]], CPLX[case["dtype"]]
    if case["kind"] == "ensemble":
        groups = []
        for k in range(4):
            nl, nt = n_lon >> k, n_lat >> k
            c = _spectrum(_gen(seed, 2 * k), case["members"], _parity(3), nl, nt).to(cd)
            pts = [_points(_gen(seed, 100 + 64 * k + j), case, nl, nt)
                   for j in range(case["members"])]
            groups.append({"n_lon": nl, "n_lat": nt, "coeffs": c.contiguous(),
                           "lon": torch.cat([p[0] for p in pts]),
                           "colat": torch.cat([p[1] for p in pts]),
                           "counts": [nl * nt] * case["members"]})
        return {"groups": groups}
    par = _parity(case["fields"])
    c = _spectrum(_gen(seed, 1), 1, par, n_lon, n_lat)[0]
    s = {"parity": par}
    if case["kind"] in ("spectral", "host"):
        s["coeffs"] = c.to(cd).contiguous()
    else:
        s["samples"] = _samples(case, c).to(rd).contiguous()
    if case["kind"] == "semilag":
        r, east, north = _frame(n_lon, n_lat)
        gen = _gen(seed, 2)
        v, va = _wind(gen, r) * WIND, _wind(gen, r) * (0.05 * WIND)
        for key, x in (("w", v), ("w_arrival", va)):
            s[key] = torch.stack([(x * east).sum(-1), (x * north).sum(-1)]).reshape(
                2, n_lat, n_lon).to(rd).contiguous()
        s["dt_over_a"] = 60.0 * case["minutes"] / RADIUS
        s["iterations"] = 3
    else:
        s["lon"], s["colat"] = _points(_gen(seed, 3), case, n_lon, n_lat)
    return s


def prepare(case, seed):
    s = _inputs(case, seed)
    s["kind"] = case["kind"]
    rd, n_lon, n_lat = REAL[case["dtype"]], case["n_lon"], case["n_lat"]
    opts = nufft.Options.make(real_fields=case["real"], gauss=case["kind"] == "gauss")
    if case["kind"] == "ensemble":
        gs = s["groups"]
        s["ensemble"] = nufft.Ensemble([(case["members"], g["n_lon"], g["n_lat"]) for g in gs],
                                       tol=TOL[case["dtype"]], dtype=case["dtype"], n_fields=3,
                                       options=[opts] * len(gs))
        s["points"] = [(g["lon"], g["colat"], g["counts"]) for g in gs]
        s["coeffs"] = [g["coeffs"] for g in gs]
        s["out"] = [torch.empty(3 * g["lon"].numel(), dtype=rd, device="cuda") for g in gs]
        return s
    default = not case["real"] and case["kind"] == "spectral"
    s["plan"] = nufft.Plan(n_lon, n_lat, TOL[case["dtype"]], case["dtype"], case["fields"],
                           options=None if default else opts)
    n_points = n_lon * n_lat if case["kind"] == "semilag" else s["lon"].numel()
    if case["kind"] == "host":
        for key in ("lon", "colat", "coeffs"):
            s[key] = s[key].cpu().pin_memory().numpy()
        s["out"] = torch.empty((case["fields"], n_points), dtype=rd).pin_memory().numpy()
        return s
    s["out"] = torch.empty((case["fields"], n_points), dtype=rd, device="cuda")
    if case["kind"] == "semilag":
        s["lon"] = torch.empty(n_points, dtype=torch.float64, device="cuda")
        s["colat"] = torch.empty(n_points, dtype=torch.float64, device="cuda")
        s["pq"] = torch.empty((2, n_points), dtype=rd, device="cuda")
    return s


def run(s):
    if s["kind"] == "ensemble":
        s["ensemble"].run(s["points"], s["coeffs"], s["out"])
        return s["out"]
    plan, out = s["plan"], s["out"]
    if s["kind"] == "host":
        return plan.execute_points_host(s["lon"], s["colat"], s["coeffs"], out)
    if s["kind"] == "semilag":
        nufft.departure_points(s["w"], s["dt_over_a"], s["iterations"], s["w_arrival"],
                               lon_out=s["lon"], colat_out=s["colat"], pq_out=s["pq"])
    plan.set_points(s["lon"], s["colat"])
    if s["kind"] == "spectral":
        return plan.execute(s["coeffs"], out)
    plan.interpolate_grid(s["samples"], s["parity"], out)
    if s["kind"] == "semilag":
        nufft.rotate_to_arrival(plan.n_lon, plan.n_lat, None, None, out[1], out[2],
                                u_a=out[1], v_a=out[2], pq=s["pq"])
        return {"values": out, "lon": s["lon"], "colat": s["colat"]}
    return out


# ------------------------------------------------------------------ what a pass needs

def _work(n_lon, n_lat, fields, points, dtype, real, spectral):
    """Points and coefficients (or samples) read once, values written once; a
    2-D transform of twice the modes in each direction (half of it for real
    values on half of the torus) and 2 w^2 operations a point and field."""
    rb = 8 if dtype == "f64" else 4
    n2, n1 = 2 * n_lat, n_lon
    if spectral:
        given = 2 * rb * n2 * (n1 // 2 + 1 if real else n1)
    else:
        given = rb * n_lat * n_lon
    fine = 4 * n1 * n2
    w = 14 if dtype == "f64" else 7
    return {"bytes": fields * (given + rb * points) + 16 * points,
            "flops": fields * (0.25 * 5 * fine * math.log2(fine) + 2 * w * w * points)}


def work(case):
    if case["kind"] == "ensemble":
        parts = [_work(case["n_lon"] >> k, case["n_lat"] >> k, 3,
                       (case["n_lon"] >> k) * (case["n_lat"] >> k), case["dtype"], case["real"],
                       True) for k in range(4)]
        return {k: case["members"] * sum(p[k] for p in parts) for k in ("bytes", "flops")}
    grid = case["n_lon"] * case["n_lat"]
    points = case["count"] if case["points"] == "scattered" else grid
    w = _work(case["n_lon"], case["n_lat"], case["fields"], points, case["dtype"], case["real"],
              case["kind"] in ("spectral", "host"))
    if case["kind"] == "semilag":
        # the winds read; the points are written here instead of read; three
        # iterations of two 6 x 6 stencils
        w["bytes"] += 4 * (8 if case["dtype"] == "f64" else 4) * grid
        w["flops"] += 3 * 2 * 2 * 36 * grid
    return w


# ------------------------------------------------------------------ results in 64 bits

KB_W = 17                                   # taps of the reference evaluation


def _kb(z):
    beta = 0.75 * math.pi * KB_W
    u = torch.clamp(1.0 - (2.0 * z / KB_W) ** 2, min=0.0)
    b = beta * torch.sqrt(u)
    return torch.special.i0e(b) * torch.exp(b - beta)


def _kb_hat(n):
    """Fourier transform of _kb at the modes -n/2..n/2-1 of a grid of 2n cells."""
    beta = 0.75 * math.pi * KB_W
    x = torch.sqrt(beta ** 2 - (_modes(n) * (math.pi / (2 * n)) * KB_W) ** 2)
    return KB_W * (torch.exp(x - beta) - torch.exp(-x - beta)) / (2.0 * x)


def _series(c, lon, colat):
    """Re sum c e^{i (m lon + n colat)} for each field: a Kaiser-Bessel window of
    17 taps on twice the modes, whose error is that of FP64 rounding."""
    fields, n2, n1 = c.shape
    f1, f2 = 2 * n1, 2 * n2
    scale = 1.0 / (_kb_hat(n2)[:, None] * _kb_hat(n1)[None, :])
    x, y = lon * (f1 / (2 * math.pi)), colat * (f2 / (2 * math.pi))
    i0, j0 = (torch.floor(v - KB_W / 2).long() + 1 for v in (x, y))
    wx = [_kb(i0 + a - x) for a in range(KB_W)]
    out = torch.zeros((fields, lon.numel()), device=lon.device, dtype=torch.float64)
    for f in range(fields):
        pad = torch.zeros((f2, f1), device=lon.device, dtype=torch.complex128)
        m = c[f].to(torch.complex128) * scale
        # centred modes to FFT order: the four corners of the fine array
        pad[:n2 // 2, :n1 // 2] = m[n2 // 2:, n1 // 2:]
        pad[:n2 // 2, f1 - n1 // 2:] = m[n2 // 2:, :n1 // 2]
        pad[f2 - n2 // 2:, :n1 // 2] = m[:n2 // 2, n1 // 2:]
        pad[f2 - n2 // 2:, f1 - n1 // 2:] = m[:n2 // 2, :n1 // 2]
        g = (torch.fft.ifft2(pad) * (f1 * f2)).real.contiguous().reshape(-1)
        for b in range(KB_W):
            row = torch.remainder(j0 + b, f2) * f1
            s = torch.zeros_like(x)
            for a in range(KB_W):
                s += wx[a] * g[row + torch.remainder(i0 + a, f1)]
            out[f] += _kb(j0 + b - y) * s
    return out


def _coeffs_of(case, samples, parity):
    """Centred coefficients of the trigonometric interpolant on the doubled
    sphere of samples on the arrival grid, rows at any colatitudes."""
    n_lat, n_lon = case["n_lat"], case["n_lon"]
    th, n = _row_colat(case), _modes(2 * n_lat)
    sgn = torch.where(_modes(n_lon) % 2 == 0, 1.0, -1.0)
    nodes = torch.cat([th, -th])
    one = torch.ones((), device="cuda", dtype=torch.float64)
    g = torch.fft.fftshift(torch.fft.fft(samples.double(), dim=-1), dim=-1) / n_lon
    par = torch.tensor(parity, device="cuda", dtype=torch.float64)[:, None, None]
    g = torch.cat([g, par * sgn * g], dim=-2)
    if case["kind"] == "gauss":
        v = torch.polar(one, nodes[:, None] * n[None, :])
        return torch.stack([torch.linalg.solve(v, f) for f in g])
    # evenly spaced colatitudes: the interpolant is the discrete transform
    v = torch.polar(one / (2 * n_lat), -n[:, None] * nodes[None, :])
    return torch.stack([v @ f for f in g])


def _quintic(field, x, y):
    """Quintic Lagrange interpolation of a wind component at index coordinates."""
    n_lat, n_lon = field.shape
    i, j = torch.floor(x), torch.floor(y)

    def weights(t):
        w = []
        for a in range(-2, 4):
            p = torch.ones_like(t)
            for b in range(-2, 4):
                if b != a:
                    p = p * (t - b) / (a - b)
            w.append(p)
        return w

    wx, wy, i, j = weights(x - i), weights(y - j), i.long(), j.long()
    total = torch.zeros_like(x)
    for a in range(6):
        rows = j + a - 2
        over = (rows < 0) | (rows >= n_lat)       # beyond a pole: half a turn away, sign changed
        r = torch.where(rows < 0, -1 - rows, torch.where(rows >= n_lat, 2 * n_lat - 1 - rows, rows))
        s = torch.zeros_like(x)
        for b in range(6):
            cols = torch.remainder(i + b - 2 + torch.where(over, n_lon // 2, 0), n_lon)
            s += wx[b] * field[r, cols]
        total += wy[a] * torch.where(over, -s, s)
    return total


def _departure(case, s):
    """Departure points of the fixed-point iteration and the rotation (p, q)
    from there to the arrival frame."""
    n_lon, n_lat = case["n_lon"], case["n_lat"]
    lon_a, colat_a = _arrival(n_lon, n_lat)
    r, east, north = _frame(n_lon, n_lat)
    w, wa = s["w"].double(), s["w_arrival"].double().reshape(2, -1)

    def rotation(lon, colat):
        den = 1.0 + (r * _xyz(lon, colat)).sum(-1)
        dl = lon_a - lon
        p = (torch.sin(colat_a) * torch.sin(colat)
             + (1.0 + torch.cos(colat_a) * torch.cos(colat)) * torch.cos(dl)) / den
        return p, (torch.cos(colat_a) + torch.cos(colat)) * torch.sin(dl) / den

    lon, colat = lon_a, colat_a
    for _ in range(s["iterations"]):
        x = torch.remainder(lon * (n_lon / (2 * math.pi)), n_lon)
        y = colat * (n_lat / math.pi) - 0.5
        we, wn = _quintic(w[0], x, y), _quintic(w[1], x, y)
        p, q = rotation(lon, colat)
        de = s["dt_over_a"] * (p * we + q * wn - wa[0])
        dn = s["dt_over_a"] * (p * wn - q * we - wa[1])
        d = torch.hypot(de, dn)[:, None]
        back = -(de[:, None] * east + dn[:, None] * north) / d.clamp(min=1e-300)
        lon, colat = _lonlat(torch.cos(d) * r + torch.sin(d) * back)
    return lon, colat, rotation(lon, colat)


def exact(case, seed):
    s = _inputs(case, seed)
    if case["kind"] == "ensemble":
        outs = []
        for g in s["groups"]:
            n = g["n_lon"] * g["n_lat"]
            outs.append(torch.cat([
                _series(c, g["lon"][k * n:(k + 1) * n], g["colat"][k * n:(k + 1) * n]).reshape(-1)
                for k, c in enumerate(g["coeffs"])]))
        return outs
    if case["kind"] in ("spectral", "host"):
        return _series(s["coeffs"], s["lon"], s["colat"])
    c = _coeffs_of(case, s["samples"], s["parity"])
    if case["kind"] != "semilag":
        return _series(c, s["lon"], s["colat"])
    lon, colat, (p, q) = _departure(case, s)
    v = _series(c, lon, colat)
    return {"values": torch.stack([v[0], p * v[1] + q * v[2], p * v[2] - q * v[1]]),
            "lon": lon, "colat": colat}
