"""The calls that users of this library make, as cases that can be timed.

Each case is one pass of an estimator through the package's public entry
points (``Plan.power``, ``Plan.power_batch``, ``Plan.power_from_grid``,
``Plan.bispectrum``), on the surveys of this repository's benchmark and tests:
the BOSS-like cap (L = 3500 Mpc/h, observer at the centre, 10,000 deg^2 about
(2, 1, 1.5), 1100 < r < 1700, Gaussian nbar(r)) and the small octant shell
(L = 1000 Mpc/h, 300 < r < 900).  The catalogs are lognormal galaxies with
radial redshift-space distortions and uniform randoms, drawn on the GPU.

The device path computes its spectra in FP32; the binding carries them in
float64 arrays.  ``run`` hands the spectra out as float32, which is what they
are, and the FP64 scalars (alpha, I_22, N_0, ...) as they come.  ``exact`` is
the same estimator in plain torch float64.
"""
import math

import numpy as np
import torch

import paper_1506_02729_gb300 as fkp

P_WANT = {2: fkp.FKP_P0 | fkp.FKP_P2, 4: fkp.FKP_P0 | fkp.FKP_P2 | fkp.FKP_P4 | fkp.FKP_P4B}
B_WANT = {1: fkp.FKP_B0, 2: fkp.FKP_B0 | fkp.FKP_B2, 3: fkp.FKP_B0 | fkp.FKP_B2 | fkp.FKP_B4}
CONTRACT = {"fp32": fkp.FKP_CONTRACT_FP32, "bf16x3": fkp.FKP_CONTRACT_BF16X3, "bf16x6": fkp.FKP_CONTRACT_BF16X6}
SCALARS = ("alpha", "I22", "I33", "N0", "N0_fkp", "S3", "W_g", "W_r")
# even products of 2, 3 and 5 that the two surveys are run on (the cap needs
# three cells inside the 50 Mpc/h between it and the box faces)
OCTANT_GRIDS = (64, 72, 80, 90, 96, 108, 120, 128, 144, 150)
CAP_GRIDS = (216, 240, 250, 256, 270, 288, 300, 320, 360, 384, 400, 432, 450, 480, 486, 500, 512)


def _case(name, call, **kw):
    c = dict(name=name, call=call, survey="cap", N=512, assign=3, lmax=4, n_gal=700000, ratio=50.0, kmin=0.0,
             dk=0.005, nbins=60, host=False, weights=False, interlace=False, mocks=1, shells=0, nl=0,
             contraction="none")
    c.update(kw)
    return c


def _octant(N, **kw):
    kf = 2 * math.pi / 1000.0
    return dict(survey="octant", N=N, n_gal=20000, ratio=10.0, kmin=0.5 * kf, dk=kf, nbins=N // 2, **kw)


def listed():
    return [
        # a quick look at a small survey (the repository's small 64^3 survey): launches and latency
        _case("octant_64", "power", assign=2, **_octant(64)),
        # the benchmark: one BOSS-like mock, P_0, P_2, P_4, P_4b
        _case("cap_512", "power"),
        # one request of the serving mix: catalogs in pinned host memory, 30x randoms
        _case("cap_384_host", "power", N=384, ratio=30.0, host=True),
        # the paper's own gridding: 360^3, fourth-order, interlaced
        _case("cap_360_pcs_interlaced", "power", N=360, assign=4, interlace=True),
        # covariance mocks that share one random catalog: galaxies only per call
        _case("cap_512_cached", "cached"),
        # an ensemble of small uneven mocks in one fused call
        _case("octant_64_batch", "batch", assign=2, mocks=32, **_octant(64)),
        # the estimator on a given periodic field (theory and N-body boxes)
        _case("field_256", "field", survey="box", N=256, n_gal=0, ratio=0.0),
        # weighted catalogs, P_0 and P_2 only, CIC, a grid that is no power of two, bins to the Nyquist k
        _case("cap_300_weighted", "power", N=300, assign=2, lmax=2, ratio=20.0, weights=True, dk=0.01, nbins=26),
        # each object's own line of sight on a small survey
        _case("octant_128_object", "object", **_octant(128)),
        # the bispectrum benchmark: B_0, B_2, B_4 in 37 shells to k = 0.2, accurate tensor-core mode
        _case("cap_360_bispectrum", "bispectrum", N=360, shells=37, nl=3, contraction="bf16x6"),
        # one mock of the batched workload: P_l and B_0 to k = 0.15 on the power spectrum's fine grid
        _case("cap_512_b0", "bispectrum", ratio=30.0, shells=27, nl=1, contraction="bf16x6"),
        # the default (FP32) contraction on the small survey
        _case("octant_64_bispectrum", "bispectrum", shells=6, nl=3, contraction="fp32", **_octant(64)),
    ]


def draw(rng):
    def logint(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    call = rng.choice(("power", "power", "power", "cached", "batch", "field", "object", "bispectrum", "bispectrum"))
    c = _case("", call, assign=rng.choice((2, 3, 3, 4)), lmax=rng.choice((2, 4, 4, 4)))
    del c["name"]
    small = call in ("object",) or rng.random() < 0.35
    if call == "field":
        c.update(survey="box", N=rng.choice(OCTANT_GRIDS + CAP_GRIDS[:11]), n_gal=0, ratio=0.0)
    elif small:
        c.update(_octant(rng.choice(OCTANT_GRIDS)))
        c["n_gal"] = logint(3000, 100000)
        c["ratio"] = float(rng.choice((5, 10, 20)))
    else:
        c["N"] = rng.choice(CAP_GRIDS if call != "batch" else CAP_GRIDS[:5])
        c["n_gal"] = logint(100000, 1200000)
        c["ratio"] = float(rng.choice((10, 20, 30) if c["n_gal"] > 600000 else (20, 30, 50)))
    if c["survey"] != "octant":
        k_nyq = math.pi * c["N"] / 3500.0
        c["dk"] = rng.choice((0.005, 0.01))
        c["nbins"] = max(8, min(int(k_nyq / c["dk"]), int(round(rng.choice((0.2, 0.3, 1.0)) / c["dk"]))))
    if call == "power":
        c["host"] = rng.random() < 0.25
        c["weights"] = rng.random() < 0.3
        c["interlace"] = rng.random() < 0.25
    if call == "batch":
        c["mocks"] = rng.choice((4, 8, 16, 32)) if c["survey"] == "octant" else rng.choice((2, 3, 4))
    if call == "bispectrum":
        c["nl"] = rng.choice((1, 2, 3))
        c["lmax"] = 4
        c["contraction"] = rng.choice(("bf16x3", "bf16x6", "bf16x6"))
        if c["survey"] == "octant":
            c["contraction"] = rng.choice(("fp32", "bf16x3", "bf16x6"))
        elif c["N"] > 400:
            c["nl"] = 1
        most = min(37 if c["nl"] < 3 or c["N"] <= 360 else 27, int((c["N"] / 3.0 - 1.6) / 3.0))
        if c["N"] > 400:
            most = min(most, 27)
        c["shells"] = rng.randint(max(3, most // 2), most)
    return c


# ---------------------------------------------------------------------------
# surveys and catalogs
# ---------------------------------------------------------------------------

def _geometry(c):
    if c["survey"] == "octant":
        L, org, obs = 1000.0, (-3 * 1000.0 / c["N"],) * 3, (0.0, 0.0, 0.0)
    else:
        L, org, obs = 3500.0, (0.0, 0.0, 0.0), (1750.0, 1750.0, 1750.0)
    return dict(L=L, N=c["N"], assign=c["assign"], origin=org, observer=obs, P_fkp=1e4, interlace=c["interlace"],
                periodic=c["survey"] == "box", compensate=c["survey"] != "box")


def _nbar(c, r):
    """nbar(r) with the case's expected galaxy count."""
    if c["survey"] == "octant":
        return torch.full_like(r, c["n_gal"] / (4 * math.pi / 8 * (900.0 ** 3 - 300.0 ** 3) / 3))
    rr = torch.linspace(1100, 1700, 4097, dtype=torch.float64, device="cuda")
    om = 10000.0 * (math.pi / 180) ** 2
    full = om * torch.trapezoid(rr ** 2 * torch.exp(-0.5 * ((rr - 1400) / 117.4) ** 2), rr)
    return c["n_gal"] / full * torch.exp(-0.5 * ((r - 1400) / 117.4) ** 2)


def _pack(c, s, r, g):
    cat = {k: s[:, a].float().contiguous() for a, k in enumerate("xyz")}
    nb = _nbar(c, r)
    cat["nbar"] = nb.float()
    if c["weights"]:  # FKP weights times a completeness weight
        u = torch.rand(r.shape[0], generator=g, device="cuda", dtype=torch.float64)
        cat["w"] = ((0.8 + 0.4 * u) / (1 + 1e4 * nb)).float()
    return cat


def _randoms(c, count, g):
    lo, hi = (300.0, 900.0) if c["survey"] == "octant" else (1100.0, 1700.0)
    rr = torch.linspace(lo, hi, 16385, dtype=torch.float64, device="cuda")
    cdf = torch.cumsum(rr ** 2 * _nbar(c, rr), 0)
    cdf = (cdf - cdf[0]) / (cdf[-1] - cdf[0])
    u = torch.rand((3, count), generator=g, device="cuda", dtype=torch.float64)
    i = torch.searchsorted(cdf, u[0]).clamp(1, rr.numel() - 1)
    r = rr[i - 1] + (rr[i] - rr[i - 1]) * (u[0] - cdf[i - 1]) / (cdf[i] - cdf[i - 1])
    if c["survey"] == "octant":
        ct, ph = u[1], 0.5 * math.pi * u[2]
        e = torch.eye(3, dtype=torch.float64, device="cuda")
    else:
        c0 = 1 - 10000.0 * (math.pi / 180) ** 2 / (2 * math.pi)
        ct, ph = c0 + (1 - c0) * u[1], 2 * math.pi * u[2]
        ax = torch.tensor([2.0, 1.0, 1.5], dtype=torch.float64, device="cuda")
        ax = ax / ax.norm()
        e1 = torch.linalg.cross(ax, torch.tensor([0.0, 1.0, 0.0], dtype=torch.float64, device="cuda"))
        e1 = e1 / e1.norm()
        e = torch.stack([e1, torch.linalg.cross(ax, e1), ax])
    st = torch.sqrt((1 - ct * ct).clamp(min=0))
    d = torch.stack([st * torch.cos(ph), st * torch.sin(ph), ct], 1) @ e
    obs = torch.tensor(_geometry(c)["observer"], dtype=torch.float64, device="cuda")
    return _pack(c, obs + r[:, None] * d, r, g)


def _power_law_modes(n, L, g):
    """Half spectrum of a Gaussian field with P(k) = 2e4 (k/0.02)^-1.5 and the mode components."""
    G = torch.fft.rfftn(torch.randn((n, n, n), generator=g, device="cuda", dtype=torch.float64))
    k1 = torch.fft.fftfreq(n, 1.0 / n, device="cuda", dtype=torch.float64) * 2 * math.pi / L
    kk = (k1[:, None, None], k1[None, :, None], k1[None, None, :n // 2 + 1].abs())
    k2 = kk[0] ** 2 + kk[1] ** 2 + kk[2] ** 2
    k2[0, 0, 0] = 1.0
    k = k2.sqrt()
    pk = 2e4 * (k / 0.02) ** -1.5 * (k <= math.pi * n / L)
    pk[0, 0, 0] = 0.0
    return G * torch.sqrt(pk * (n / L) ** 3), kk, k2


def _galaxies(c, g):
    """Lognormal, Poisson-sampled galaxies with radial redshift-space distortions (f = 0.7)."""
    geom = _geometry(c)
    L, n = geom["L"], 64 if c["survey"] == "octant" else 128
    H = L / n
    G, kk, k2 = _power_law_modes(n, L, g)
    delta = torch.fft.irfftn(G, (n, n, n))
    lo, hi = (300.0, 900.0) if c["survey"] == "octant" else (1100.0, 1700.0)
    env = float(_nbar(c, torch.linspace(lo, hi, 601, dtype=torch.float64, device="cuda")).max())
    lam = (env * H ** 3 * torch.exp(delta - 0.5 * delta.var())).reshape(-1)
    cell = torch.repeat_interleave(torch.arange(n ** 3, device="cuda"), torch.poisson(lam, generator=g).long())
    ijk = torch.stack([cell % n, (cell // n) % n, cell // (n * n)], 1)
    org = torch.tensor(geom["origin"], dtype=torch.float64, device="cuda")
    obs = torch.tensor(geom["observer"], dtype=torch.float64, device="cuda")
    x = org + H * (ijk + torch.rand(ijk.shape, generator=g, device="cuda", dtype=torch.float64))
    d = x - obs
    r = d.norm(dim=1).clamp(min=1e-9)
    d = d / r[:, None]
    psi = torch.stack([torch.fft.irfftn(1j * kk[a] / k2 * G, (n, n, n)).reshape(-1)[cell] for a in (2, 1, 0)], 1)
    r = r + 0.7 * (psi * d).sum(1)
    x = obs + r[:, None] * d
    if c["survey"] == "octant":
        keep = (d > 0).all(1)
    else:
        ax = torch.tensor([2.0, 1.0, 1.5], dtype=torch.float64, device="cuda")
        keep = d @ (ax / ax.norm()) >= 1 - 10000.0 * (math.pi / 180) ** 2 / (2 * math.pi)
    keep &= (r >= lo) & (r < hi)
    keep &= torch.rand(r.shape, generator=g, device="cuda", dtype=torch.float64) < _nbar(c, r) / env
    x, r = x[keep], r[keep]
    p = torch.randperm(r.shape[0], generator=g, device="cuda")  # catalogs are in no spatial order
    return _pack(c, x[p], r[p], g)


def _inputs(c, seed):
    """The catalogs (a list of (galaxies, randoms)), or the field."""
    g = torch.Generator(device="cuda")
    g.manual_seed(1000003 * int(seed) + 17)
    if c["call"] == "field":
        G, _, _ = _power_law_modes(c["N"], 3500.0, g)
        return torch.fft.irfftn(G, (c["N"],) * 3).float().contiguous()
    nr = int(round(c["n_gal"] * c["ratio"]))
    gal, ran = _galaxies(c, g), _randoms(c, nr, g)
    if c["call"] != "batch":
        return [(gal, ran)]
    out = []
    for _ in range(c["mocks"]):  # uneven mocks: 50-100 % subsamples
        pair = []
        for cat in (gal, ran):
            n = cat["x"].numel()
            m = int(n * (0.5 + 0.5 * float(torch.rand((), generator=g, device="cuda"))))
            i = torch.randperm(n, generator=g, device="cuda")[:m]
            pair.append({k: v[i].contiguous() for k, v in cat.items()})
        out.append(tuple(pair))
    return out


def _shells(c):
    return (3, 3, 3, c["shells"]) if c["shells"] else None


def _want(c):
    w = P_WANT[c["lmax"]]
    if c["call"] == "object":
        w |= fkp.FKP_XHAT_OBJECT
    return w | (B_WANT[c["nl"]] if c["shells"] else 0)


def prepare(case, seed):
    c = _case("", "power")
    c.update(case)
    data = _inputs(c, seed)
    plan = fkp.Plan(_geometry(c), (c["kmin"], c["dk"], c["nbins"]), bshells=_shells(c), want=_want(c))
    if c["call"] == "cached":
        plan.cache_randoms(data[0][1])
        data = [(data[0][0], None)]
    if c["host"]:
        data = [tuple({k: v.cpu().pin_memory() for k, v in cat.items()} for cat in pair) for pair in data]
    return dict(case=c, plan=plan, data=data)


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def _spectra(c):
    return ("k_eff", "mono_raw", "P0", "P2", "P4b") + (("P4",) if c["lmax"] >= 4 else ())


def _power_outputs(c, p):
    out = {k: np.asarray(p[k], np.float32) for k in _spectra(c)}
    out["nmodes"] = p["nmodes"]
    if c["call"] != "field":
        out["scalars"] = np.array([p[k] for k in SCALARS])
        out["Lab"] = np.asarray(p["Lab"], np.float32)
    return out


def _bisp_keys(c):
    return tuple(k + str(l) for l in (0, 2, 4)[:c["nl"]] for k in ("B", "N", "T"))


def run(state):
    c, plan, data = state["case"], state["plan"], state["data"]
    if c["call"] == "field":
        return _power_outputs(c, plan.power_from_grid(data))
    if c["call"] == "batch":
        ps = [_power_outputs(c, p) for p in plan.power_batch([g for g, _ in data], [r for _, r in data])]
        return {k: np.stack([p[k] for p in ps]) for k in ps[0]}
    if c["call"] == "bispectrum":
        p, b = plan.bispectrum(*data[0], contraction=CONTRACT[c["contraction"]])
        out = _power_outputs(c, p)
        out.update({k: np.asarray(b[k], np.float32) for k in _bisp_keys(c)})
        out.update(tri=b["tri"], NT=b["NT"], centre_closed=b["centre_closed"])
        return out
    return _power_outputs(c, plan.power(*data[0]))


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def _triangles(S):
    """Shell triples a >= b >= c that close (shells of width 3 about 3 (s + 1))."""
    return [(a, b, c) for a in range(S) for b in range(a + 1) for c in range(b + 1)
            if 3 * a + 1.5 < 3 * b + 4.5 + 3 * c + 4.5]


def work(case):
    c = _case("", "power")
    c.update(case)
    N3 = float(c["N"]) ** 3
    nobj = 0.0
    if c["call"] != "field":
        nobj = c["n_gal"] * (1.0 + (c["ratio"] if c["call"] != "cached" else 0.0))
        nobj *= c["mocks"] * (0.75 if c["call"] == "batch" else 1.0)  # the mean 50-100 % subsample
    passes = c["mocks"] * (2 if c["interlace"] else 1) * (2 if c["shells"] else 1)
    fields = {2: 6, 4: 15}[c["lmax"]]  # 1 + 5 (+ 9) independent moments
    fft = 2.5 * math.log2(N3)
    flops = passes * fields * N3 * (fft + 2) + nobj * (2 if c["interlace"] else 1) * (4 * c["assign"] ** 3 + 40)
    if c["call"] == "object":
        flops += nobj * fields * 2 * c["assign"] ** 3
    byts = nobj * (20 if c["weights"] else 16) + (4 * N3 if c["call"] == "field" else 0)
    byts += c["mocks"] * c["nbins"] * 8 * 7
    if c["shells"]:
        n3 = (3 * (3 * c["shells"] + 1.5)) ** 3  # the coarsest grid that holds the triangle sums
        tri, S = _triangles(c["shells"]), c["shells"]
        flops += c["nl"] * S * n3 * 2.5 * math.log2(n3) + n3 * (2 * len(tri) * c["nl"] + S * (S + 1) / 2)
        byts += len(tri) * (8 + 7 + 24 * c["nl"])
    return {"bytes": byts, "flops": flops}


# ---------------------------------------------------------------------------
# the same in float64
# ---------------------------------------------------------------------------

def _f64(cat):
    pos = torch.stack([cat[k].double() for k in "xyz"], 1)
    nb = cat["nbar"].double()
    return pos, cat["w"].double() if "w" in cat else 1.0 / (1.0 + nb * 1e4), nb


def _taps(u, p):
    """First node and the p weights of the assignment of order p (CIC, TSC, PCS) along one axis."""
    if p == 2:
        i = torch.floor(u)
        d = u - i
        return i, (1 - d, d)
    if p == 3:
        i = torch.floor(u + 0.5)
        d = u - i
        return i - 1, (0.5 * (0.5 - d) ** 2, 0.75 - d * d, 0.5 * (0.5 + d) ** 2)
    i = torch.floor(u)
    d = u - i
    return i - 1, ((1 - d) ** 3 / 6, (4 - 6 * d * d + 3 * d ** 3) / 6, (1 + 3 * d + 3 * d * d - 3 * d ** 3) / 6, d ** 3 / 6)


def _assign(grid, pos, val, geom, org):
    N, p = geom["N"], geom["assign"]
    for s in range(0, val.numel(), 1 << 23):  # in pieces, to bound the memory
        v = val[s:s + (1 << 23)]
        t = [_taps((pos[s:s + (1 << 23), a] - org[a]) * (N / geom["L"]), p) for a in range(3)]
        for iz in range(p):
            for iy in range(p):
                row = (((t[2][0] + iz) % N) * N + (t[1][0] + iy) % N) * N
                wv = v * t[2][1][iz] * t[1][1][iy]
                for ix in range(p):
                    grid.index_add_(0, (row + (t[0][0] + ix) % N).long(), wv * t[0][1][ix])
    return grid


def _modes(N):
    n1 = torch.fft.fftfreq(N, 1.0 / N, device="cuda", dtype=torch.float64)
    return n1[None, None, :N // 2 + 1].abs(), n1[None, :, None], n1[:, None, None]


def _tensor(rank):
    """Exponents (i, j, k) of the distinct rank-2 or rank-4 components and their multiplicities."""
    f = math.factorial
    return [((i, j, rank - i - j), f(rank) // (f(i) * f(j) * f(rank - i - j)))
            for i in range(rank + 1) for j in range(rank + 1 - i)]


def _legendre(field_of, N, lmax):
    """F_0, F_2, F_4 on the half spectrum; field_of(i, j, k) is the moment field F x^i y^j z^k of the unit x^."""
    n = _modes(N)
    inv2 = 1.0 / (n[0] ** 2 + n[1] ** 2 + n[2] ** 2).clamp(min=1.0)
    F = [torch.fft.rfftn(field_of(0, 0, 0))]
    for rank in range(2, lmax + 1, 2):
        S = torch.zeros_like(F[0])
        for e, m in _tensor(rank):
            S += m * (n[0] ** e[0] * n[1] ** e[1] * n[2] ** e[2]) * torch.fft.rfftn(field_of(*e))
        S *= inv2 ** (rank // 2)
        F.append(1.5 * S - 0.5 * F[0] if rank == 2 else 4.375 * S - 2.5 * F[1] - 0.875 * F[0])
    return F


def _unit(d):
    r = d.norm(dim=-1, keepdim=True)
    return torch.where(r > 0, d / r.clamp(min=1e-300), torch.zeros_like(d))


def _node_moments(grid, geom, org):
    """field_of for x^ at the grid nodes."""
    N = geom["N"]
    i = torch.arange(N, device="cuda", dtype=torch.float64) * (geom["L"] / N)
    x, y, z = ((i + org[a] - geom["observer"][a]).reshape([N if b == 2 - a else 1 for b in range(3)]) for a in range(3))
    r = torch.sqrt(x * x + y * y + z * z)
    inv = torch.where(r > 0, 1.0 / r.clamp(min=1e-300), torch.zeros_like(r))

    def field_of(a, b, c):
        return grid * (x ** a * y ** b * z ** c) * inv ** (a + b + c)
    return field_of


def _window(N, p):
    n = _modes(N)
    w = 1.0
    for a in n:
        w = w * torch.sinc(a / N) ** p
    return w


def _survey(c, gal, ran):
    """F_l, the scalars and (with shells) F^w_l, in float64."""
    geom = _geometry(c)
    N, L = geom["N"], geom["L"]
    (pg, wg, _), (pr, wr, nr) = _f64(gal), _f64(ran)
    Wg, Wr = wg.sum(), wr.sum()
    al = Wg / Wr
    obs = torch.tensor(geom["observer"], dtype=torch.float64, device="cuda")
    xg, xr = _unit(pg - obs), _unit(pr - obs)
    sc = dict(alpha=al, I22=al * (nr * wr ** 2).sum(), I33=al * (nr ** 2 * wr ** 3).sum(),
              N0=(wg ** 2).sum() + al ** 2 * (wr ** 2).sum(), N0_fkp=al * (1 + al) * (wr ** 2).sum(),
              S3=(wg ** 3).sum() - al ** 3 * (wr ** 3).sum(), W_g=Wg, W_r=Wr)
    sc = {k: float(v) for k, v in sc.items()}
    sc["Lab"] = [float((xr[:, a] * xr[:, b] * wr).sum() / Wr) for a, b in ((0, 0), (1, 1), (2, 2), (0, 1), (1, 2), (2, 0))]
    n = _modes(N)
    fields = []
    for power in ((1, 2) if c["shells"] else (1,)):
        vg, vr = (wg, -al * wr) if power == 1 else (wg ** 2, al ** 2 * wr ** 2)
        F = None
        for half in ((0, 1) if c["interlace"] else (0,)):
            org = [o + half * 0.5 * L / N for o in geom["origin"]]

            def grid_of(mg, mr):
                g = torch.zeros(N ** 3, device="cuda", dtype=torch.float64)
                return _assign(_assign(g, pg, mg, geom, org), pr, mr, geom, org).view(N, N, N)

            if c["call"] == "object":
                def field_of(i, j, k):
                    f = [x[:, 0] ** i * x[:, 1] ** j * x[:, 2] ** k for x in (xg, xr)]
                    return grid_of(vg * f[0], vr * f[1])
            else:
                field_of = _node_moments(grid_of(vg, vr), geom, org)
            G = _legendre(field_of, N, c["lmax"])
            if half:
                t = -math.pi / N * (n[0] + n[1] + n[2])
                F = [0.5 * (f + torch.polar(torch.ones_like(t), t) * g) for f, g in zip(F, G)]
            else:
                F = G
        w = _window(N, geom["assign"])
        fields.append([f / w for f in F])
    return fields, sc


def _mode_index(N):
    """|n|^2, the full-grid weight and whether the mode is off n = 0 and the Nyquist planes."""
    n = _modes(N)
    n2 = n[0] ** 2 + n[1] ** 2 + n[2] ** 2
    off = (n2 > 0) & (n[0] < N // 2) & (n[1].abs() < N // 2) & (n[2].abs() < N // 2)
    return n2, (1.0 + (n[0] > 0)).expand(n2.shape), off


def _bins(c, F, I22, N0):
    geom = _geometry(c)
    n2, wt, off = _mode_index(c["N"])
    k = 2 * math.pi / geom["L"] * torch.sqrt(n2)
    edges = c["kmin"] + c["dk"] * torch.arange(c["nbins"] + 1, device="cuda", dtype=torch.float64)
    b = torch.searchsorted(edges, k, right=True) - 1
    sel = off & (b >= 0) & (b < c["nbins"])
    b, wt = b[sel], wt[sel]

    def mean(v):
        return torch.bincount(b, weights=wt * v[sel], minlength=c["nbins"]) / nm

    nm = torch.bincount(b, weights=wt, minlength=c["nbins"])  # no modes: 0/0 = nan, as the library says
    s00, s20, s22 = mean(F[0].abs() ** 2), mean((F[1] * F[0].conj()).real), mean(F[1].abs() ** 2)
    out = dict(k_eff=mean(k), mono_raw=s00 / I22, P0=(s00 - N0) / I22, P2=5 * s20 / I22,
               P4b=(17.5 * s22 - 5 * s20 - 3.5 * s00) / I22)
    if c["lmax"] >= 4:
        out["P4"] = 9 * mean((F[2] * F[0].conj()).real) / I22
    return dict({k: v.cpu().numpy() for k, v in out.items()}, nmodes=None)


def _triangle_sums(fa, fc, S, nl):
    """T[l][a][b][c] = sum_x fa[l S + a] fc[b] fc[c] for a >= b >= c."""
    N = fc.shape[-1]
    T = torch.zeros(nl, S, S, S, device="cuda", dtype=torch.float64)
    for b in range(S):
        prod = (fc[:b + 1] * fc[b]).view(b + 1, N, N * N)
        for l in range(nl):
            A = fa[l * S + b:(l + 1) * S].view(S - b, N, N * N)
            T[l, b:, b, :b + 1] = torch.bmm(A.transpose(0, 1), prod.permute(1, 2, 0)).sum(0)
    return T


def _bispectrum(c, F, Fw, sc):
    N, S, nl = c["N"], c["shells"], c["nl"]
    n2, wt, off = _mode_index(N)
    cen = 3.0 * np.arange(1, S + 1)
    edges = torch.arange(S + 1, device="cuda", dtype=torch.float64) * 3.0 + 1.5
    sh = torch.searchsorted(edges ** 2, n2, right=True) - 1
    sh = torch.where(off & (sh >= 0) & (sh < S), sh, torch.full_like(sh, -1))

    def shell_fields(f):
        return torch.stack([torch.fft.irfftn(torch.where(sh == s, f, torch.zeros_like(f)), (N,) * 3) * float(N) ** 3
                            for s in range(S)])
    one = shell_fields(torch.ones_like(F[0]))
    NT = torch.round(_triangle_sums(one, one, S, 1)[0] / float(N) ** 3).cpu().numpy()
    del one
    fa = torch.cat([shell_fields(F[l]) for l in range(nl)])
    T = _triangle_sums(fa, fa[:S], S, nl).cpu().numpy()
    sel = sh >= 0
    nm = torch.bincount(sh[sel], weights=wt[sel], minlength=S)

    def mean(u, v):
        return (torch.bincount(sh[sel], weights=(wt * (u * v.conj()).real)[sel], minlength=S) / nm).cpu().numpy()
    tri = [(a, b, d) for a in range(S) for b in range(a + 1) for d in range(b + 1) if NT[a, b, d] > 0]
    a, b, d = np.array(tri).T
    mu = [np.clip((cen[q] ** 2 - cen[a] ** 2 - cen[p] ** 2) / (2 * cen[a] * cen[p]), -1, 1) for p, q in ((b, d), (d, b))]
    leg = {0: lambda m: 1.0 + 0 * m, 2: lambda m: 1.5 * m * m - 0.5, 4: lambda m: (35 * m ** 4 - 30 * m * m + 3) / 8}
    out = dict(tri=None, NT=None, centre_closed=None)
    for li in range(nl):
        l = 2 * li
        s1, s2 = mean(F[li], Fw[0]), mean(F[0], Fw[li])
        noise = (2 * l + 1) / sc["I33"] * (s1[a] + leg[l](mu[0]) * s2[b] + leg[l](mu[1]) * s2[d])
        if l == 0:
            noise = noise - 2 * sc["S3"] / sc["I33"]
        t = T[li, a, b, d]
        out["T%d" % l], out["N%d" % l] = t, noise
        out["B%d" % l] = (2 * l + 1) * t / (float(N) ** 3 * NT[a, b, d] * sc["I33"]) - noise
    return out


def exact(case, seed):
    c = _case("", "power")
    c.update(case)
    data = _inputs(c, seed)
    if c["call"] == "field":
        F = _legendre(_node_moments(data.double(), _geometry(c), _geometry(c)["origin"]), c["N"], c["lmax"])
        return _bins(c, F, 1.0, 0.0)
    outs = []
    for gal, ran in data:
        fields, sc = _survey(c, gal, ran)
        out = _bins(c, fields[0], sc["I22"], sc["N0"])
        out["scalars"] = np.array([sc[k] for k in SCALARS])
        out["Lab"] = np.array(sc["Lab"])
        if c["shells"]:
            out.update(_bispectrum(c, fields[0], fields[1], sc))
        outs.append(out)
    if c["call"] != "batch":
        return outs[0]
    return {k: None if outs[0][k] is None else np.stack([o[k] for o in outs]) for k in outs[0]}
