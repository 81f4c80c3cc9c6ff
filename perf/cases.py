"""The workloads whose time and accuracy are tracked: what users of this library run, from a small
periodic box to the 768^3 request of a served stream.

Three kinds of call, each through the public Python entry points:
  * ``box``: one script-like evaluation, ``Estimator.paint`` + ``Estimator.multipoles`` (both return
    host values, so each call waits for the GPU);
  * ``survey``: paint and multipoles enqueued back to back with device outputs, as a pipeline that
    keeps the GPU busy does, followed by the wedges where the case asks for them;
  * ``mocks``: data catalogs against cached randoms meshes through ``Estimator.run_batch`` (a served
    request is a batch of one).

Survey-shaped catalogs are a 60 degree cap about (1,1,1) with a 600-1400 Mpc/h shell inside a
2000 Mpc/h box: data follow a lognormal field, randoms are uniform in the cap, FKP P0 = 1e4.
FP32 contexts get max_particles for all their catalogs: the exact tile paint, whose meshes do not
depend on the order of the additions.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1704_02357_gb300 import Estimator, wedges

BOX = 2000.0
P0 = 1e4
NBAR = 3e-4
R_MIN, R_MAX, HALF_ANGLE = 600.0, 1400.0, math.radians(60.0)
MU_EDGES = [0.0, 0.05, 0.2, 0.4, 0.6, 0.8, 1.0]
NGEN = 64  # grid of the lognormal field the data are drawn from


def _case(name, kind, nmesh, ells, n_data, n_randoms, precision="fp32", window="cic", interlaced=True, mocks=1,
          weighted=False, pos="f64", n_bins=0, wedge=False, compensate="sinc"):
    c = dict(kind=kind, nmesh=nmesh, ells=ells, n_data=n_data, n_randoms=n_randoms, precision=precision,
             window=window, interlaced=interlaced, mocks=mocks, weighted=weighted, pos=pos, n_bins=n_bins,
             wedge=wedge, compensate=compensate)
    return dict(name=name, **c) if name else c


def listed():
    return [
        # the smallest call: a notebook-sized box, TSC and interlacing
        _case("box_32_tsc", "box", 32, "0,2,4", 2000, 6000, window="tsc", n_bins=8),
        # the plain FP64 estimator on a periodic box, no interlacing, k bins of 0.01 up to 0.3
        _case("box_64_fp64", "box", 64, "0,2,4", 20000, 100000, precision="fp64", interlaced=False,
              compensate="none", n_bins=30),
        # a small request of a served stream
        _case("request_128", "mocks", 128, "0,2,4", 400_001, 2_000_003),
        # a mock campaign's two mesh sizes; catalogs of 3e5 to 3e6 galaxies
        _case("mocks_256", "mocks", 256, "0,2,4", 1_000_003, 8_000_009, mocks=4),
        _case("mocks_384", "mocks", 384, "0,2,4", 2_500_001, 16_000_007, mocks=2),
        # a survey with completeness weights and a measured n(z) per object, FP32 positions,
        # odd multipoles included
        _case("weighted_256_odd", "box", 256, "0,1,2,3,4", 300_007, 6_000_011, window="tsc", weighted=True, pos="f32"),
        # the survey workload at full size in the library's three precisions
        _case("survey_512", "survey", 512, "0,2,4", 797_000, 15_940_000),
        _case("survey_512_plain", "survey", 512, "0,2,4", 797_000, 15_940_000, precision="fp32_plain"),
        _case("survey_512_fp64", "survey", 512, "0,2,4", 797_000, 15_940_000, precision="fp64"),
        # wedges from every even multipole up to 16
        _case("wedges_384_l16", "survey", 384, "0,2,4,6,8,10,12,14,16", 797_003, 8_000_001, window="tsc", wedge=True),
        # a large request of a served stream
        _case("request_768", "mocks", 768, "0,2,4", 5_000_003, 16_000_003),
    ]


def draw(rng):
    def logint(a, b):
        return int(round(math.exp(rng.uniform(math.log(a), math.log(b))))) | 1

    kind = rng.choice(["box", "survey", "survey", "mocks", "mocks"])
    window = rng.choice(["cic", "tsc"])
    if kind == "box":
        n = rng.choice([32, 48, 64, 96, 128, 192, 256])
        precision = rng.choice(["fp32", "fp32_plain", "fp64"])
        nd = logint(2000, 3e5)
        return _case(None, kind, n, rng.choice(["0,2,4", "0,2", "0,1,2,3,4", "0,2,4,6"]), nd, logint(3 * nd, 20 * nd),
                     precision=precision, window=window, interlaced=rng.random() < 0.7,
                     compensate=rng.choice(["sinc", "sinc", "jing", "none"]), weighted=rng.random() < 0.4,
                     pos=rng.choice(["f64", "f32"]), n_bins=rng.randint(5, n // 2))
    if kind == "survey":
        precision = rng.choice(["fp32", "fp32_plain", "fp64"])
        n = rng.choice([192, 256, 384] if precision == "fp64" else [192, 256, 384, 512])
        nd = logint(1e5, 1e6)
        return _case(None, kind, n, rng.choice(["0,2,4", "0,2,4", "0,2,4,6", "0,2"]), nd, logint(5 * nd, 16 * nd),
                     precision=precision, window=window, weighted=rng.random() < 0.3,
                     pos=rng.choice(["f64", "f64", "f32"]), wedge=rng.random() < 0.3)
    n = rng.choice([128, 192, 256, 384, 512])
    ells = "0,2,4,6,8,10,12,14,16" if n <= 192 and rng.random() < 0.4 else "0,2,4"
    return _case(None, kind, n, ells, logint(1e5, 3e6), logint(2e6, 1.6e7), precision=rng.choice(["fp32", "fp32_plain"]),
                 window=window, mocks=rng.randint(1, 3))


# ---------------------------------------------------------------- geometry and catalogs
def _geometry(case):
    """(box size, corner, observer): a periodic box off the origin, or the survey cap's box."""
    if case["kind"] == "box":
        return 1000.0, [500.0, 500.0, 500.0], [0.0, 0.0, 0.0]
    ang = math.acos(1.0 / math.sqrt(3.0)) + HALF_ANGLE
    centre = 0.5 * (R_MAX * math.cos(ang) + R_MAX)
    return BOX, [centre - 0.5 * BOX] * 3, [0.0, 0.0, 0.0]


def _ells(case):
    return [int(e) for e in case["ells"].split(",")]


def _edges(case):
    L, n = _geometry(case)[0], case["nmesh"]
    kn = math.pi * n / L
    if case["n_bins"]:
        if case["compensate"] == "none" and case["nmesh"] == 64:
            return 0.01 * np.arange(case["n_bins"] + 1)
        return np.linspace(0.0, kn, case["n_bins"] + 1)
    return 0.005 * np.arange(int(kn / 0.005) + 1)


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _gen(seed, salt):
    return torch.Generator(device=_device()).manual_seed(1_000_003 * (seed % 1_000_000_007) + salt)


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device=_device(), dtype=torch.float64)


def _cap_points(n, g):
    """Uniform in the cap and shell."""
    u = _rand(g, n, 3)
    r = (R_MIN ** 3 + u[:, 0] * (R_MAX ** 3 - R_MIN ** 3)) ** (1.0 / 3.0)
    ct = math.cos(HALF_ANGLE) + u[:, 1] * (1.0 - math.cos(HALF_ANGLE))
    st = (1.0 - ct * ct).clamp_min(0.0).sqrt()
    phi = 2.0 * math.pi * u[:, 2]
    s2, s3, s6 = math.sqrt(2.0), math.sqrt(3.0), math.sqrt(6.0)
    e1, e2, e3 = (1 / s2, -1 / s2, 0.0), (1 / s6, 1 / s6, -2 / s6), (1 / s3, 1 / s3, 1 / s3)
    a, b = st * phi.cos(), st * phi.sin()
    return torch.stack([r * (a * e1[d] + b * e2[d] + ct * e3[d]) for d in range(3)], dim=1).contiguous()


def _clustered(n, corner, seed, g):
    """n galaxies in the cap following a lognormal field with P(k) = 2e4 x / (1 + x^2.4), x = k/0.02."""
    rng = np.random.default_rng(seed)
    h = BOX / NGEN
    kf = 2.0 * math.pi / BOX
    kx = np.fft.fftfreq(NGEN, 1.0 / NGEN) * kf
    kz = np.arange(NGEN // 2 + 1) * kf
    x = np.sqrt(kx[:, None, None] ** 2 + kx[None, :, None] ** 2 + kz[None, None, :] ** 2) / 0.02
    amp = np.sqrt(2e4 * x / (1.0 + x ** 2.4) / h ** 3)
    field = np.fft.irfftn(np.fft.rfftn(rng.standard_normal((NGEN,) * 3)) * amp, s=(NGEN,) * 3)
    c = [corner[d] + (np.arange(NGEN) + 0.5) * h for d in range(3)]
    r = np.sqrt(c[0][:, None, None] ** 2 + c[1][None, :, None] ** 2 + c[2][None, None, :] ** 2)
    cosang = (c[0][:, None, None] + c[1][None, :, None] + c[2][None, None, :]) / (math.sqrt(3.0) * r)
    near = (r > R_MIN - h) & (r < R_MAX + h) & (r * np.sin(np.arccos(np.clip(cosang, -1, 1)) - HALF_ANGLE) < h)
    cdf = torch.from_numpy(np.cumsum(np.where(near, np.exp(field), 0.0).ravel())).to(_device())
    got, have = [], 0
    while have < n:
        m = int(1.5 * (n - have)) + 1000
        cell = torch.searchsorted(cdf, _rand(g, m) * cdf[-1]).clamp_max(NGEN ** 3 - 1)
        ijk = torch.stack([cell // (NGEN * NGEN), (cell // NGEN) % NGEN, cell % NGEN], dim=1).double()
        p = torch.tensor(corner, device=_device(), dtype=torch.float64) + (ijk + _rand(g, m, 3)) * h
        rr = p.square().sum(1).sqrt()
        ok = (rr >= R_MIN) & (rr < R_MAX) & (p.sum(1) >= math.cos(HALF_ANGLE) * math.sqrt(3.0) * rr)
        got.append(p[ok])
        have += got[-1].shape[0]
    return torch.cat(got)[:n].contiguous()


def _catalogs(case, seed):
    """data catalogs (one per mock) and randoms as (pos, weight, nbar)."""
    L, corner, _ = _geometry(case)
    data = []
    for m in range(case["mocks"]):
        g = _gen(seed, 17 + m)
        if case["kind"] == "box":
            pos = torch.tensor(corner, device=_device(), dtype=torch.float64) + _rand(g, case["n_data"], 3) * L
        else:
            pos = _clustered(case["n_data"] - 2 * (m * case["n_data"] // 11), corner, seed * 64 + m, g)
        data.append(_extras(case, pos, g))
    g = _gen(seed, 5)
    if case["kind"] == "box":
        pos = torch.tensor(corner, device=_device(), dtype=torch.float64) + _rand(g, case["n_randoms"], 3) * L
    else:
        pos = _cap_points(case["n_randoms"], g)
    return data, _extras(case, pos, g)


def _extras(case, pos, g):
    """Completeness weights around 1 and a smooth n(r), for weighted cases; positions in the case's type."""
    w = nb = None
    if case["weighted"]:
        w = 0.7 + 0.6 * _rand(g, pos.shape[0])
        nb = NBAR * (1.0 + 0.5 * torch.sin(pos.square().sum(1).sqrt() / 150.0))
    if case["pos"] == "f32":
        pos = pos.float()
    return pos, w, nb


def _fkp(case):
    """(P0, nbar) of the context: unit weights in the periodic FP64 box, FKP elsewhere."""
    if case["kind"] == "box":
        n = case["n_data"] / _geometry(case)[0] ** 3
        return (0.0 if case["compensate"] == "none" else P0), n
    return P0, NBAR


# ---------------------------------------------------------------- the measured calls
def prepare(case, seed):
    L, corner, observer = _geometry(case)
    data, randoms = _catalogs(case, seed)
    p0, nbar = _fkp(case)
    ells, edges = _ells(case), _edges(case)
    batch = case["kind"] == "mocks"
    sizes = [d[0].shape[0] for d in data]
    count = max(sizes + [randoms[0].shape[0]]) if batch else sizes[0] + randoms[0].shape[0]
    est = Estimator(nmesh=case["nmesh"], box_size=L, box_corner=corner, observer=observer, window=case["window"],
                    interlaced=case["interlaced"],
                    compensate=False if case["compensate"] == "none" else case["compensate"],
                    precision=case["precision"], ell_max=max(ells), P0=p0, nbar=nbar,
                    max_particles=0 if case["precision"] == "fp64" else count, cache_randoms=batch)
    s = {"case": case, "est": est, "data": data, "randoms": randoms, "ells": ells, "edges": edges}
    if batch:
        est.set_randoms(*randoms)
    elif case["kind"] == "survey":
        nk = len(edges) - 1
        s["P"] = torch.empty((len(ells), nk), dtype=torch.float64, device="cuda")
        s["k"] = torch.empty(nk, dtype=torch.float64, device="cuda")
        s["n"] = torch.empty(nk, dtype=torch.float64, device="cuda")
    return s


def run(s):
    est, kind = s["est"], s["case"]["kind"]
    if kind == "mocks":
        out = est.run_batch(s["data"], s["ells"], s["edges"])
        return {"P": out["P"], "sums": out["sums"], "k_mean": out["k_mean"], "n_modes": out["n_modes"]}
    (dp, dw, dn), (rp, rw, rn) = s["data"][0], s["randoms"]
    if kind == "box":
        st = est.paint(dp, rp, dw, dn, rw, rn)
        out = est.multipoles(s["ells"], s["edges"])
        return {"P": out["P"], "k_mean": out["k_mean"], "n_modes": out["n_modes"],
                "sums": np.array([st["alpha"], st["I"], st["S"], st["W_d"]])}
    est.paint(dp, rp, dw, dn, rw, rn, stats=False)
    est.multipoles_device(s["ells"], s["edges"], s["P"], s["k"], s["n"])
    out = {"P": s["P"], "k_mean": s["k"], "n_modes": s["n"]}
    if s["case"]["wedge"]:
        out["wedges"] = wedges(s["P"], s["ells"], MU_EDGES)
    return out


def work(case):
    """Catalogs read once, results written once; the arithmetic of the transforms and of the
    harmonics' weights and products."""
    n3 = float(case["nmesh"]) ** 3
    ells = _ells(case)
    per = (12 if case["pos"] == "f32" else 24) + (16 if case["weighted"] else 0)
    batch = case["kind"] == "mocks"
    if batch:
        particles = sum(case["n_data"] - 2 * (m * case["n_data"] // 11) for m in range(case["mocks"]))
    else:
        particles = case["n_data"] + case["n_randoms"]
    nk = len(_edges(case)) - 1
    outputs = 8.0 * nk * (case["mocks"] * len(ells) + 2)
    # cached randoms meshes are inputs of a batch: each is read once per batch
    esz = 8 if case["precision"] == "fp64" else 4
    meshes = (2 if case["interlaced"] else 1) * n3 * esz if batch else 0.0
    fft = 2.5 * n3 * math.log2(n3)
    harmonics = sum(2 * l + 1 for l in ells if l)
    base = (2 if case["interlaced"] else 1) + (1 if case["interlaced"] or case["compensate"] in ("sinc", "jing") else 0)
    flops = case["mocks"] * (fft * (base + harmonics) + harmonics * 4.0 * n3)
    return {"bytes": particles * per + outputs + meshes, "flops": flops}


# ---------------------------------------------------------------- the same in 64 bits
def _axis_weights(u, window):
    if window == "cic":
        b = torch.floor(u)
        d = u - b
        return b.long(), [1.0 - d, d]
    c = torch.floor(u + 0.5)
    d = u - c
    return c.long() - 1, [0.5 * (0.5 - d) ** 2, 0.75 - d * d, 0.5 * (0.5 + d) ** 2]


def _paint(mesh, pos, value, case, shift):
    n = case["nmesh"]
    L, corner, _ = _geometry(case)
    for lo in range(0, pos.shape[0], 1 << 22):  # bounded index arrays
        p, v = pos[lo:lo + (1 << 22)].double(), value[lo:lo + (1 << 22)]
        ax = [_axis_weights((p[:, d] - corner[d]) * (n / L) - shift, case["window"]) for d in range(3)]
        for a, wa in enumerate(ax[0][1]):
            for b, wb in enumerate(ax[1][1]):
                for c, wc in enumerate(ax[2][1]):
                    at = (((ax[0][0] + a) % n) * n + (ax[1][0] + b) % n) * n + (ax[2][0] + c) % n
                    mesh.view(-1).index_add_(0, at, v * wa * wb * wc)


def _ylm(l, m, x, y, z):
    """Real spherical harmonic of unit vectors, from the associated Legendre recurrence in l."""
    a = abs(m)
    norm = math.sqrt((2 * l + 1) / (4 * math.pi) * math.factorial(l - a) / math.factorial(l + a))
    norm *= (-1) ** a * (math.sqrt(2.0) if a else 1.0)
    q0 = torch.full_like(z, float(math.prod(range(1, 2 * a, 2))))  # P_a^a / (-sin)^a
    if l > a:
        q1 = (2 * a + 1) * z * q0
        for k in range(a + 2, l + 1):
            q0, q1 = q1, (z * q1).mul_(2 * k - 1).sub_(q0, alpha=k + a - 1).div_(k - a)
        q0 = q1
    if a:
        pr, pi = x, y
        for _ in range(a - 1):
            pr, pi = pr * x - pi * y, pi * x + pr * y
        q0 = q0 * (pr if m > 0 else pi)
    return q0.mul_(norm) if a else q0 * norm


def _unit(vx, vy, vz):
    r2 = vx * vx + vy * vy + vz * vz
    inv = torch.where(r2 > 0, r2, torch.ones_like(r2)).rsqrt_()
    return vx * inv, vy * inv, vz * inv, r2


def _values(cat, p0, nbar):
    n = cat[0].shape[0]
    wc = cat[1] if cat[1] is not None else torch.ones(n, device=_device(), dtype=torch.float64)
    nb = cat[2] if cat[2] is not None else torch.full((n,), nbar, device=_device(), dtype=torch.float64)
    return wc, nb, (1.0 / (1.0 + nb * p0) if p0 > 0 else torch.ones_like(nb))


def _exact_one(case, data, randoms):
    n, dev = case["nmesh"], _device()
    L, corner, observer = _geometry(case)
    p0, nbar = _fkp(case)
    (wd, nd, fd), (wr, nr, fr) = _values(data, p0, nbar), _values(randoms, p0, nbar)
    alpha = float(wd.sum() / wr.sum())
    I = alpha * float((nr * wr * fr * fr).sum())
    S = float((wd * fd).square().sum()) + alpha ** 2 * float((wr * fr).square().sum())
    f = torch.arange(n, device=dev, dtype=torch.float64)
    f = torch.where(f < n // 2, f, f - n)
    fx, fy, fz = f[:, None, None], f[None, :, None], torch.arange(n // 2 + 1, device=dev, dtype=torch.float64)

    def spectrum(shift):
        mesh = torch.zeros((n, n, n), device=dev, dtype=torch.float64)
        _paint(mesh, data[0], wd * fd, case, shift)
        _paint(mesh, randoms[0], -alpha * wr * fr, case, shift)
        return torch.fft.rfftn(mesh), mesh

    X, mesh = spectrum(0.0)
    if case["interlaced"]:
        ph = (-math.pi / n) * (fx + fy + fz)
        X = 0.5 * (X + torch.polar(torch.ones_like(ph), ph) * spectrum(0.5)[0])
        del ph
    nyq = (fx == -(n // 2)) | (fy == -(n // 2)) | (fz == n // 2)
    p = {"cic": 2, "tsc": 3}[case["window"]]
    if case["compensate"] != "none":
        def ax(v):
            if case["compensate"] == "jing":
                s2 = torch.sin(math.pi * v / n) ** 2
                return (1 - 2 / 3 * s2 if p == 2 else 1 - s2 + 2 / 15 * s2 * s2).sqrt()
            return torch.sinc(v / n) ** p
        X = X / (ax(fx) * ax(fy) * ax(fz))
    if case["interlaced"] or case["compensate"] != "none":
        X = torch.where(nyq, torch.zeros_like(X), X)
        real = torch.fft.irfftn(X, s=(n, n, n))
    else:
        real = mesh
    del mesh
    n2 = fx * fx + fy * fy + fz * fz
    t = (torch.from_numpy(np.asarray(_edges(case))).to(dev) * (L / (2.0 * math.pi))) ** 2
    nk = t.shape[0] - 1
    b = torch.bucketize(n2, t, right=True) - 1
    b = torch.where((n2 < t[0]) | (n2 >= t[-1]) | (n2 == 0) | nyq, torch.full_like(b, nk), b).view(-1)
    mult = torch.where(fz == 0, 1.0, 2.0).double().expand(n, n, n // 2 + 1)

    def binned(v):
        return torch.bincount(b, weights=(v * mult).reshape(-1), minlength=nk + 1)[:nk]

    modes = binned(torch.ones_like(n2))
    k_mean = binned((2 * math.pi / L) * n2.sqrt()) / modes
    kx, ky, kz, _ = _unit(fx.expand_as(n2), fy.expand_as(n2), fz.expand_as(n2))
    del n2, nyq
    h = L / n
    g = [corner[d] - observer[d] + h * torch.arange(n, device=dev, dtype=torch.float64) for d in range(3)]
    rx, ry, rz, _ = _unit(g[0][:, None, None].expand(n, n, n), g[1][None, :, None].expand(n, n, n),
                          g[2][None, None, :].expand(n, n, n))
    P = []
    for l in _ells(case):
        if l == 0:
            P.append((binned(X.real.square() + X.imag.square()) / modes - S) / I)
            continue
        acc = torch.zeros(X.shape, device=dev, dtype=torch.float64)
        for m in range(-l, l + 1):
            G = torch.fft.rfftn(real * _ylm(l, m, rx, ry, rz))
            part = G.imag * X.real - G.real * X.imag if l % 2 else G.real * X.real + G.imag * X.imag
            acc.addcmul_(_ylm(l, m, kx, ky, kz), part)
            del G, part
        P.append(4.0 * math.pi * binned(acc) / (I * modes))
    return torch.stack(P), k_mean, modes, [alpha, I, S, float(wd.sum())]


def _lbar(l, a, b):
    if l == 0:
        return 1.0
    q = np.polynomial.legendre.Legendre.basis(l).integ()
    return float(q(b) - q(a)) / (b - a)


def exact(case, seed):
    data, randoms = _catalogs(case, seed)
    got = [_exact_one(case, d, randoms) for d in data]
    P, k_mean, modes, sums = got[0]
    if case["kind"] == "mocks":
        return {"P": torch.stack([o[0] for o in got]), "k_mean": k_mean, "n_modes": modes,
                "sums": torch.tensor([o[3] for o in got], dtype=torch.float64)}
    out = {"P": P, "k_mean": k_mean, "n_modes": modes}
    if case["kind"] == "box":
        out["sums"] = np.array(sums)
    elif case["wedge"]:
        lb = torch.tensor([[_lbar(l, a, b) for l in _ells(case)] for a, b in zip(MU_EDGES[:-1], MU_EDGES[1:])],
                          dtype=torch.float64, device=_device())
        out["wedges"] = lb @ P
    return out
