"""The workloads that stand for this library's use: each case is one call of a public entry point of
paper_1512_07295_gb300.api on seeded synthetic inputs.

``listed()`` names them, ``draw(rng)`` gives more of the same ranges, ``prepare`` makes what a
program holds before the call, ``run`` makes the call, ``work`` counts the bytes and operations it
cannot do without, and ``exact`` gives its result in 64 bits (plain torch, no code of the library).
"""

import math

import torch

from paper_1512_07295_gb300 import api, catalogs

DEV = "cuda"
TWO_PI = 2.0 * math.pi


def listed():
    return [
        # one small catalogue from device positions: the smallest call, where launches and latency count
        {"name": "pk-small", "kind": "power", "cat": "poisson", "n": 64**3, "ng": 64, "order": 4, "interlace": True,
         "prec": "fp32", "weights": False, "box": 1000.0},
        # the FP64 (oracle-parity) mode on a clustered catalogue
        {"name": "pk-fp64", "kind": "power", "cat": "za", "n": 128**3, "ng": 128, "order": 4, "interlace": True,
         "prec": "fp64", "weights": False, "box": 500.0},
        # mass grids of a 256^3 clustered catalogue, one particle per cell: sort and sparse assignment
        {"name": "assign-sparse", "kind": "assign", "cat": "za", "n": 256**3, "ng": 256, "order": 4, "interlace": True,
         "prec": "fp32", "weights": False, "box": 1500.0},
        # weighted uniform catalogue in random order, CIC, one grid, a grid that the tiles do not divide
        {"name": "assign-cic-weighted", "kind": "assign", "cat": "poisson", "n": 5_000_001, "ng": 180, "order": 2,
         "interlace": False, "prec": "fp32", "weights": True, "box": 1000.0},
        # the bit-reproducible mode, TSC
        {"name": "assign-tsc-fixed64", "kind": "assign", "cat": "za", "n": 192**3, "ng": 128, "order": 3, "interlace": True,
         "prec": "fixed64", "weights": False, "box": 750.0},
        # the large survey-sized measurement: 1024^3 particles resident in the binned layout
        {"name": "pk-large-binned", "kind": "binned", "cat": "za", "n": 1024**3, "ng": 512, "order": 4, "interlace": True,
         "prec": "fp32", "weights": False, "box": 2000.0},
        # many uneven mock catalogues, Poisson and clustered, in one call
        {"name": "batch-mocks", "kind": "batch", "ncat": 96, "lo": 100_000, "hi": 2_000_000, "ng": 128, "order": 4,
         "box": 1000.0},
        # all triangles of 16 shells of a non-Gaussian field
        {"name": "bispectrum", "kind": "bispectrum", "ng": 256, "shell_lo": 0, "shell_w": 4, "nshells": 16, "box": 1500.0},
        # the gradient of a loss over P(k) with respect to the positions (the backward pass)
        {"name": "gradient", "kind": "backward", "cat": "za", "n": 128**3, "ng": 128, "order": 4, "interlace": True,
         "weights": False, "box": 500.0},
        # the alias-free direct sum over all modes of a small grid
        {"name": "direct-sum", "kind": "direct", "cat": "za", "n": 64**3, "ng": 64, "weights": False, "box": 400.0},
        # cross power of two fields (grid estimate against direct sum)
        {"name": "cross-power", "kind": "cross", "ng": 256, "box": 1500.0},
        # four interlaced grids
        {"name": "multigrid-4", "kind": "multigrid", "cat": "za", "n": 256**3, "ng": 256, "order": 4, "ngrids": 4,
         "weights": False, "box": 1500.0},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _even(rng, lo, hi):
    return 2 * _log_int(rng, lo // 2, hi // 2)


def draw(rng):
    kind = rng.choice(["power", "assign", "binned", "batch", "bispectrum", "backward", "direct", "cross", "multigrid"])
    box = round(rng.uniform(300.0, 2500.0), 1)
    c = {"kind": kind, "box": box}

    def catalogue(lo, hi):
        n = _log_int(rng, lo, hi)
        if rng.random() < 0.5:
            c.update(cat="poisson", n=n)
        else:
            c.update(cat="za", n=max(8, 2 * round(n ** (1.0 / 3.0) / 2)) ** 3)

    if kind in ("power", "assign"):
        prec = rng.choice(["fp32", "fp32", "fp64", "fixed64"])
        catalogue(20_000, 3_000_000 if prec == "fp64" else 40_000_000)
        # from about eight particles per cell to one per three cells
        ng = (c["n"] * math.exp(rng.uniform(math.log(0.125), math.log(3.0)))) ** (1.0 / 3.0)
        c.update(ng=min(384, max(24, 2 * round(ng / 2))), prec=prec, weights=rng.random() < 0.3,
                 order=rng.choice([2, 3, 4, 4]), interlace=rng.random() < 0.7)
    elif kind == "binned":
        side = 2 * _log_int(rng, 64, 300)
        dense = rng.random() < 0.5
        c.update(cat="za", n=side**3, ng=2 * round(side * (0.5 if dense else 0.9) / 2), order=rng.choice([2, 3, 4, 4]),
                 interlace=rng.random() < 0.8, prec="fp32", weights=rng.random() < 0.2)
    elif kind == "batch":
        c.update(ncat=_log_int(rng, 4, 64), lo=50_000, hi=_log_int(rng, 200_000, 2_000_000), ng=_even(rng, 48, 140),
                 order=rng.choice([3, 4, 4]))
    elif kind == "bispectrum":
        ns, w = rng.randrange(4, 17), rng.randrange(2, 6)
        c.update(nshells=ns, shell_w=w, shell_lo=rng.randrange(0, 3))
        c["ng"] = 2 * math.ceil((3 * (c["shell_lo"] + ns * w) + rng.randrange(0, 24)) / 2)
    elif kind == "backward":
        catalogue(30_000, 6_000_000)
        c.update(ng=_even(rng, 32, 180), order=rng.choice([2, 3, 4, 4]), interlace=rng.random() < 0.8,
                 weights=rng.random() < 0.3)
    elif kind == "direct":
        catalogue(5_000, 400_000)
        c.update(ng=_even(rng, 16, 90), weights=rng.random() < 0.3)
    elif kind == "cross":
        c.update(ng=_even(rng, 48, 400))
    else:
        catalogue(100_000, 20_000_000)
        c.update(ng=_even(rng, 48, 280), order=rng.choice([2, 3, 4, 4]), ngrids=rng.choice([2, 4, 8]),
                 weights=rng.random() < 0.2)
    return c


# ---- inputs ------------------------------------------------------------------------------------------


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _positions(c, seed):
    """FP64 positions: uniform in random order, or Zel'dovich-displaced in lattice order (rms 4 length units)."""
    if c["cat"] == "poisson":
        return torch.rand((c["n"], 3), generator=_gen(seed), device=DEV, dtype=torch.float64) * c["box"]
    side = round(c["n"] ** (1.0 / 3.0))
    return catalogs.zeldovich_torch(side, c["box"], 4.0, seed, DEV)


def _weights(c, seed):
    if not c.get("weights"):
        return None
    return 0.5 + torch.rand(c["n"], generator=_gen(seed + 7_000_003), device=DEV, dtype=torch.float32)


def _cfg(c):
    return api.Config(ng=c["ng"], box=c["box"], order=c.get("order", 4), interlace=c.get("interlace", True),
                      prec=c.get("prec", "fp32"))


def _field(ng, seed, skew=0.6):
    """Half-complex transform of a non-Gaussian (lognormal) real field with a falling spectrum, complex64."""
    white = torch.randn((ng, ng, ng), generator=_gen(seed), device=DEV, dtype=torch.float32)
    k1 = torch.fft.fftfreq(ng, d=1.0 / ng, device=DEV)
    kz = torch.arange(ng // 2 + 1, device=DEV, dtype=torch.float32)
    k2 = k1[:, None, None] ** 2 + k1[None, :, None] ** 2 + kz[None, None, :] ** 2
    g = torch.fft.irfftn(torch.fft.rfftn(white) * (k2 + 4.0) ** -0.5, s=(ng, ng, ng))
    d = torch.exp(g * (skew / g.std()))
    d = d / d.mean() - 1.0
    out = torch.fft.rfftn(d) / float(ng) ** 3
    out[0, 0, 0] = 0
    return out.contiguous()


def _batch_catalogues(c, seed):
    """Sizes log-uniform in [lo, hi]; even catalogues uniform, odd ones in Gaussian clumps."""
    u = torch.rand(c["ncat"], generator=_gen(seed), device=DEV, dtype=torch.float64).cpu()
    sizes = [int(math.exp(math.log(c["lo"]) + float(v) * math.log(c["hi"] / c["lo"]))) for v in u]
    parts, offs = [], [0]
    for k, n in enumerate(sizes):
        g = _gen(seed * 4099 + k)
        x = torch.rand((n, 3), generator=g, device=DEV, dtype=torch.float64)
        if k % 2:
            nc = max(1, n // 40)
            centre = torch.randint(0, nc, (n,), generator=g, device=DEV)
            x = x[:nc][centre] + 0.01 * torch.randn((n, 3), generator=g, device=DEV, dtype=torch.float64)
            x = x - torch.floor(x)
            x[x >= 1.0] = 0.0
        parts.append(x * c["box"])
        offs.append(offs[-1] + n)
    return torch.cat(parts), offs


def prepare(case, seed):
    c, kind = case, case["kind"]
    s = {"kind": kind}
    if kind == "batch":
        pos, offs = _batch_catalogues(c, seed)
        cfg = _cfg(c)
        batch = c["ncat"]
        s.update(cells=api.prepare(pos, cfg), offs=offs, cfg=cfg, batch=batch)
        s["ws"] = api.batch_workspace(cfg, batch, offs[-1], DEV)
        return s
    if kind == "bispectrum":
        cfg = _cfg(c)
        counts = api.bispectrum_counts(cfg, c["shell_lo"], c["shell_w"], c["nshells"], DEV)
        s.update(cfg=cfg, delta=_field(c["ng"], seed), shells=(c["shell_lo"], c["shell_w"], c["nshells"]), counts=counts)
        return s
    if kind == "cross":
        a = _field(c["ng"], seed)
        s.update(cfg=_cfg(c), a=a, b=(0.8 * a + 0.2 * _field(c["ng"], seed + 1_000_003)).contiguous())
        s["ws"] = api.workspace(s["cfg"], 0, api.ffi.PK_WS_CROSS, DEV)
        return s
    cfg = _cfg(c)
    pos, w = _positions(c, seed), _weights(c, seed)
    s.update(cfg=cfg, w=w)
    if kind == "binned":
        s["binned"] = api.bin_particles(pos, cfg, w)
        s["ws"] = api.workspace(cfg, c["n"], api.ffi.PK_WS_POWER_BINNED, DEV)
        return s
    s["pos"] = pos
    if kind == "power":
        s["ws"] = api.workspace(cfg, c["n"], api.ffi.PK_WS_POWER, DEV)
    elif kind == "backward":
        s["dl"] = torch.randn(cfg.nb, generator=_gen(seed + 11), device=DEV, dtype=torch.float64) / c["box"] ** 3
    elif kind == "direct":
        s["ws"] = api.workspace(cfg, c["n"], api.ffi.PK_WS_DIRECT, DEV)
    elif kind == "multigrid":
        s["ngrids"] = c["ngrids"]
    return s


def run(s):
    kind = s["kind"]
    if kind == "power":
        return api.power(s["pos"], s["cfg"], s["w"], ws=s["ws"])
    if kind == "assign":
        return api.assign(s["pos"], s["cfg"], s["w"])
    if kind == "binned":
        return api.power_binned(s["binned"], s["cfg"], ws=s["ws"])
    if kind == "batch":
        return api.batch_power(s["cells"], s["offs"], s["cfg"], batch=s["batch"], ws=s["ws"])
    if kind == "bispectrum":
        return api.bispectrum(s["delta"], s["cfg"], *s["shells"], counts=s["counts"])
    if kind == "backward":
        return api.power_backward(s["pos"], s["cfg"], s["dl"], s["w"])
    if kind == "direct":
        return api.direct_modes(s["pos"], s["cfg"], s["w"], ws=s["ws"])
    if kind == "cross":
        return api.cross_power(s["a"], s["b"], s["cfg"], ws=s["ws"])
    return api.power_multigrid(s["pos"], s["cfg"], s["ngrids"], s["w"])


def work(case):
    """Inputs once, outputs once; where the method goes through mass grids, each grid written once by the
    assignment and read and written once by its transform. Operations: 2 p^3 per particle and grid for
    the assignment (6 p^3 for the gradient's gather), 5 N^3 log2 N / 2 per real transform and axis set,
    8 per particle and mode for the direct sum, 2 per point and triangle for the bispectrum."""
    c, kind = case, case["kind"]
    real = 4 if c.get("prec", "fp32") == "fp32" else 8
    if kind == "cross":
        modes = c["ng"] ** 2 * (c["ng"] // 2 + 1)
        return {"bytes": 16.0 * modes, "flops": 4.0 * modes}
    if kind == "bispectrum":
        m = 3 * (c["shell_lo"] + c["nshells"] * c["shell_w"] - 1) + 1
        ntri = api.bispectrum_ntri(c["nshells"])
        fft = 2.5 * m**3 * math.log2(m**3) * c["nshells"]
        return {"bytes": 3.0 * 4 * m**3 * c["nshells"] + 8.0 * ntri, "flops": fft + 2.0 * ntri * m**3}
    p3 = c.get("order", 4) ** 3
    ng3 = float(c["ng"]) ** 3
    if kind == "batch":
        n = c["ncat"] * (c["hi"] - c["lo"]) / math.log(c["hi"] / c["lo"])
        grids = 2 * c["ncat"]
        return {"bytes": 16.0 * n + 12.0 * grids * ng3, "flops": grids * (2.5 * ng3 * math.log2(ng3)) + 4.0 * p3 * n}
    n = float(c["n"])
    if kind == "direct":
        modes = c["ng"] ** 2 * (c["ng"] // 2 + 1)
        return {"bytes": 24.0 * n + 8.0 * modes, "flops": 8.0 * n * modes}
    grids = c["ngrids"] if kind == "multigrid" else (2 if c["interlace"] else 1)
    rec = 16.0 if kind == "binned" else 24.0
    b = n * (rec + (4.0 if c["weights"] else 0.0)) + grids * real * ng3
    f = 2.0 * p3 * grids * n
    if kind != "assign":
        b += 2.0 * grids * real * ng3
        f += grids * 2.5 * ng3 * math.log2(ng3)
    if kind == "backward":
        b += 12.0 * n + n * rec + 3.0 * grids * real * ng3
        f += 6.0 * p3 * grids * n + grids * 2.5 * ng3 * math.log2(ng3)
    return {"bytes": b, "flops": f}


# ---- the same results in 64 bits -----------------------------------------------------------------------


def _spline(order, s):
    """Centred B-spline of the order at distance s and its derivative with respect to s."""
    a, sg = s.abs(), torch.sign(s)
    if order == 2:
        return torch.clamp(1 - a, min=0), torch.where(a < 1, -sg, torch.zeros_like(s))
    if order == 3:
        near = a < 0.5
        w = torch.where(near, 0.75 - s * s, 0.5 * torch.clamp(1.5 - a, min=0) ** 2)
        return w, torch.where(near, -2 * s, -sg * torch.clamp(1.5 - a, min=0))
    near = a < 1
    r = torch.clamp(2 - a, min=0)
    w = torch.where(near, (4 - 6 * s * s + 3 * a**3) / 6, r**3 / 6)
    return w, torch.where(near, -2 * s + 1.5 * s * a, -0.5 * sg * r * r)


def _stencils(u, order, ng):
    """Per axis: node indices (order, n) and the weights and their derivatives with respect to u."""
    out = []
    for a in range(3):
        x = u[:, a]
        first = torch.floor(x + 0.5) - 1 if order == 3 else torch.floor(x) - (order // 2 - 1)
        nodes = first[None, :] + torch.arange(order, device=DEV, dtype=torch.float64)[:, None]
        w, dw = _spline(order, nodes - x[None, :])
        out.append((nodes.long() % ng, w, -dw))
    return out


def _mass_grid(u, ng, order, w=None):
    grid = torch.zeros(ng**3, device=DEV, dtype=torch.float64)
    for part in range(0, u.shape[0], 1 << 23):
        (ix, wx, _), (iy, wy, _), (iz, wz, _) = _stencils(u[part:part + (1 << 23)], order, ng)
        if w is not None:
            wx = wx * w[part:part + (1 << 23)].double()[None, :]
        for a in range(order):
            for b in range(order):
                row, v = (ix[a] * ng + iy[b]) * ng, wx[a] * wy[b]
                for d in range(order):
                    grid.index_add_(0, row + iz[d], v * wz[d])
    return grid.view(ng, ng, ng)


def _signed(ng):
    i = torch.arange(ng, device=DEV)
    return torch.where(i < ng // 2, i, i - ng)


def _modes(ng):
    n = _signed(ng)
    return n[:, None, None], n[None, :, None], n[None, None, :]


def _inv_window(ng, order):
    x = math.pi * _signed(ng).double() / ng
    w = torch.where(x == 0, torch.ones_like(x), torch.sin(x) / torch.where(x == 0, torch.ones_like(x), x)) ** -order
    return w[:, None, None] * w[None, :, None] * w[None, None, :]


def _shifted_phase(ng, shift):
    nx, ny, nz = _modes(ng)
    ph = TWO_PI / ng * (shift[0] * nx + shift[1] * ny + shift[2] * nz).double()
    return torch.polar(torch.ones_like(ph), ph)


def _delta(u, ng, order, shifts, w=None):
    """delta(n) on the full grid from mass grids shifted by `shifts` cells."""
    wsum = float(u.shape[0]) if w is None else float(w.double().sum())
    d = torch.zeros((ng, ng, ng), device=DEV, dtype=torch.complex128)
    for sh in shifts:
        g = _mass_grid(u + torch.tensor(sh, device=DEV, dtype=torch.float64), ng, order, w)
        d += torch.fft.fftn(g) * _shifted_phase(ng, sh)
    d *= _inv_window(ng, order) / (len(shifts) * wsum)
    d[0, 0, 0] = 0
    return d


def _bins(ng):
    """Bin of every mode: b (from 0) with (b + 1/2)^2 <= |n|^2 < (b + 3/2)^2, -1 outside 0 .. N/2 - 1."""
    nx, ny, nz = _modes(ng)
    n2 = nx * nx + ny * ny + nz * nz
    b = torch.floor(torch.sqrt(n2.double()) - 0.5).long()
    b = torch.where((2 * b + 1) ** 2 > 4 * n2, b - 1, b)
    b = torch.where((2 * b + 3) ** 2 <= 4 * n2, b + 1, b)
    return torch.where((b < 0) | (b >= ng // 2) | (n2 == 0), torch.full_like(b, -1), b), n2


def _shells(power, ng, box):
    b, n2 = _bins(ng)
    ok = b >= 0
    nb, idx = ng // 2, b[ok]
    cnt = torch.bincount(idx, minlength=nb)
    pk = torch.bincount(idx, weights=power[ok] * box**3, minlength=nb) / cnt
    km = torch.bincount(idx, weights=torch.sqrt(n2[ok].double()), minlength=nb) * (TWO_PI / box) / cnt
    return pk, km, cnt


HALF = (0.5, 0.5, 0.5)


def _shift_set(c):
    j = c.get("ngrids") or (2 if c.get("interlace", True) else 1)
    base = [(0.0, 0.0, 0.0), (0.5, 0.5, 0.0), (0.5, 0.0, 0.5), (0.0, 0.5, 0.5)]
    if j <= 2:
        return [(0.0, 0.0, 0.0), HALF][:j]
    return base if j == 4 else [s for b in base for s in (b, tuple(x + 0.5 for x in b))]


def _exact_backward(c, u, w, dl):
    ng, order, box = c["ng"], c["order"], c["box"]
    shifts = _shift_set(c)
    wsum = float(u.shape[0]) if w is None else float(w.double().sum())
    d = _delta(u, ng, order, shifts, w)
    b, _ = _bins(ng)
    cnt = torch.bincount(b[b >= 0], minlength=ng // 2)
    kappa = torch.where(b >= 0, (dl * box**3 / cnt)[b.clamp(min=0)], torch.zeros((), device=DEV, dtype=torch.float64))
    amp = 2.0 * kappa * torch.conj(d) * _inv_window(ng, order) / (len(shifts) * wsum)
    out = torch.zeros_like(u)
    for sh in shifts:
        g = torch.fft.fftn(amp * _shifted_phase(ng, sh)).real.contiguous().view(-1)
        for part in range(0, u.shape[0], 1 << 22):
            sl = slice(part, part + (1 << 22))
            st = _stencils(u[sl] + torch.tensor(sh, device=DEV, dtype=torch.float64), order, ng)
            (ix, wx, dx), (iy, wy, dy), (iz, wz, dz) = st
            for i in range(order):
                for j in range(order):
                    row = (ix[i] * ng + iy[j]) * ng
                    for k in range(order):
                        v = g[row + iz[k]]
                        out[sl, 0] += v * dx[i] * wy[j] * wz[k]
                        out[sl, 1] += v * wx[i] * dy[j] * wz[k]
                        out[sl, 2] += v * wx[i] * wy[j] * dz[k]
    out *= ng / box
    return out if w is None else out * w.double()[:, None]


def _exact_direct(c, u, w):
    ng = c["ng"]
    n = _signed(ng).double()
    nz = torch.arange(ng // 2 + 1, device=DEV, dtype=torch.float64)
    acc = torch.zeros((ng * (ng // 2 + 1), ng), device=DEV, dtype=torch.complex128)
    t = TWO_PI * u / ng
    for part in range(0, u.shape[0], 8192):
        p = t[part:part + 8192]
        ex, ey, ez = (torch.exp(-1j * (p[:, a, None] * k[None, :])) for a, k in ((0, n), (1, n), (2, nz)))
        if w is not None:
            ex = ex * w[part:part + 8192].double()[:, None]
        acc += (ex[:, :, None] * ez[:, None, :]).reshape(p.shape[0], -1).T @ ey
    # the stored plane i_z = N/2 stands for n_z = -N/2
    last = torch.zeros((ng, ng), device=DEV, dtype=torch.complex128)
    for part in range(0, u.shape[0], 8192):
        p = t[part:part + 8192]
        ex, ey = (torch.exp(-1j * (p[:, a, None] * n[None, :])) for a in (0, 1))
        ez = torch.exp(1j * (p[:, 2] * (ng // 2)))
        if w is not None:
            ez = ez * w[part:part + 8192].double()
        last += (ex * ez[:, None]).T @ ey
    d = acc.view(ng, ng // 2 + 1, ng).permute(0, 2, 1).contiguous()
    d[:, :, ng // 2] = last
    d /= float(u.shape[0]) if w is None else float(w.double().sum())
    d[0, 0, 0] = 0
    return d


def _exact_bispectrum(c, delta):
    ng, lo, w, ns = c["ng"], c["shell_lo"], c["shell_w"], c["nshells"]
    n = _signed(ng)
    nz = torch.arange(ng // 2 + 1, device=DEV)
    n2 = n[:, None, None] ** 2 + n[None, :, None] ** 2 + nz[None, None, :] ** 2
    fields, ones = [], []
    for s in range(ns):
        m = (n2 >= (lo + s * w) ** 2) & (n2 < (lo + (s + 1) * w) ** 2) & (n2 > 0)
        fields.append(torch.fft.irfftn(delta.to(torch.complex128) * m, s=(ng,) * 3, norm="forward"))
        ones.append(torch.fft.irfftn(m.to(torch.complex128), s=(ng,) * 3, norm="forward"))
    out = []
    for a in range(ns):
        for b in range(a + 1):
            cs = [q for q in range(b + 1) if a <= b + q + 1]
            if not cs:
                continue
            f2, o2 = fields[a] * fields[b], ones[a] * ones[b]
            for q in cs:
                tri = torch.round((o2 * ones[q]).sum() / ng**3)
                val = c["box"] ** 6 * (f2 * fields[q]).sum() / ng**3 / tri
                out.append(torch.where(tri > 0, val, torch.full_like(val, math.nan)))
    return torch.stack(out)


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind == "cross":
        s = prepare(case, seed)
        ng, h = c["ng"], c["ng"] // 2
        re = (s["a"].to(torch.complex128) * s["b"].to(torch.complex128).conj()).real
        mult = torch.full((h + 1,), 2.0, device=DEV, dtype=torch.float64)
        mult[0] = mult[h] = 1.0
        b, n2 = (t[:, :, :h + 1] for t in _bins(ng))
        ok = b >= 0
        mm = mult[None, None, :].expand_as(re)[ok]
        nb, idx = ng // 2, b[ok]
        cnt = torch.bincount(idx, weights=mm, minlength=nb)
        pk = torch.bincount(idx, weights=mm * re[ok], minlength=nb) * c["box"] ** 3 / cnt
        km = torch.bincount(idx, weights=mm * torch.sqrt(n2[ok].double()), minlength=nb) * (TWO_PI / c["box"]) / cnt
        return pk, km, cnt.long()
    if kind == "bispectrum":
        return _exact_bispectrum(c, _field(c["ng"], seed)), None
    if kind == "batch":
        pos, offs = _batch_catalogues(c, seed)
        pks, cnts = [], []
        for k in range(c["ncat"]):
            u = pos[offs[k]:offs[k + 1]] * (c["ng"] / c["box"])
            d = _delta(u, c["ng"], c["order"], [(0.0, 0.0, 0.0), HALF])
            pk, _, cnt = _shells(d.real**2 + d.imag**2, c["ng"], c["box"])
            pks.append(pk)
            cnts.append(cnt)
        return torch.stack(pks), torch.stack(cnts)
    if c["n"] > 45_000_000:  # over 20 seconds
        return None
    u, w = _positions(c, seed) * (c["ng"] / c["box"]), _weights(c, seed)
    if kind == "direct":
        return _exact_direct(c, u, w)
    if kind == "backward":
        dl = torch.randn(c["ng"] // 2, generator=_gen(seed + 11), device=DEV, dtype=torch.float64) / c["box"] ** 3
        return _exact_backward(c, u, w, dl)
    shifts = _shift_set(c)
    if kind == "assign":
        grids = [_mass_grid(u + torch.tensor(s, device=DEV, dtype=torch.float64), c["ng"], c["order"], w) for s in shifts]
        return grids[0], grids[1] if len(grids) > 1 else None
    d = _delta(u, c["ng"], c["order"], shifts, w)
    return _shells(d.real**2 + d.imag**2, c["ng"], c["box"])
