"""What a user of this library has it do, as timed cases: single evaluations,
minimisations, MD steps, forces and batches of finite-temperature OF-DFT
hydrogen, from 20^3 to 256^3 grid points, through the public binding
(paper_1406_0835_gb300.ofdft).

Every case is one of six kinds of call:
  static    ofdft_energy_potential_static on device buffers (latency-critical
            callers; the smallest call of the library)
  evaluate  Context.energy_potential with a host density in and the potential
            out (a caller with its own minimiser, or checks)
  minimise  Context.minimize from the uniform density (a single point)
  md        Context.md_step: the first geometry's solve and the steps after it
  forces    Context.energy_potential at the resident density, then
            Context.forces (an outer geometry or MD code)
  batch     ofdft_batch_minimize of several uneven systems (EOS scans)

`exact` evaluates the same equations in binary64 with torch alone (full
complex FFTs, Fermi-Dirac integrals by Gauss-Legendre quadrature).
"""
import math

import numpy as np
import torch

from paper_1406_0835_gb300 import inputs, ofdft

KEYS_E = ("F_tot", "F_s", "minus_TS", "E_H", "E_loc", "F_xc", "E_ion", "E_int", "mu", "E_alphaZ")
KEYS_P = ("P", "P_s", "P_xc", "P_H", "P_loc", "P_ion")


def _case(name, kind, functional, nat, rho, T, grid, **more):
    c = dict(name=name, kind=kind, functional=functional, nat=nat, rho=rho, T=T,
             nx=grid[0], ny=grid[1], nz=grid[2], precision="fp64", tri=False)
    c.update(more)
    return c


def listed():
    return [
        # the allocation-free entry point: one small ftTF system, called in a loop
        _case("static 20^3 ftTF", "static", "fttf", 8, 1.0, 1.0e5, (20, 20, 20)),
        # the same entry point near its limits with the GGA, uneven edges
        _case("static 24x30x40 VT84F", "static", "vt84f", 32, 1.0, 3.125e4, (24, 30, 40)),
        # the single-point workload (8 H, 1 g/cm^3, 100 kK, ftTF): one evaluation
        _case("evaluate 32^3 ftTF", "evaluate", "fttf", 8, 1.0, 1.0e5, (32, 32, 32)),
        # a sheared cell with uneven edges, as a crystal code hands it over
        _case("evaluate 60x54x72 KST2 sheared", "evaluate", "kst2", 32, 1.0, 6.0e4, (60, 54, 72), tri=True),
        # an evaluation at the MD workload's size
        _case("evaluate 96^3 SGA", "evaluate", "sga", 128, 1.0, 3.125e4, (96, 96, 96)),
        # the single-point workload, minimised
        _case("minimise 32^3 ftTF", "minimise", "fttf", 8, 1.0, 1.0e5, (32, 32, 32)),
        # a single point of the GGA on an uneven grid (50 = 2 5 5: no power of two beyond 2)
        _case("minimise 48x50x54 VT84F", "minimise", "vt84f", 24, 1.0, 6.0e4, (48, 50, 54)),
        # the mixed-precision single point: 256 H, 4 g/cm^3, 250 kK, 128^3
        _case("minimise 128^3 VT84F mixed", "minimise", "vt84f", 256, 4.0, 2.5e5, (128, 128, 128),
              precision="mixed"),
        # the MD workload: 128 H, 1 g/cm^3, 31.25 kK, 96^3, ftGGA
        _case("md 96^3 VT84F", "md", "vt84f", 128, 1.0, 3.125e4, (96, 96, 96), steps=1),
        # a small MD system of an EOS sweep, SGA
        _case("md 40^3 SGA", "md", "sga", 16, 1.0, 3.125e4, (40, 40, 40), steps=2),
        # six uneven mixed-precision single points at once (the batched form)
        _case("batch of 6, 32^3-80^3 mixed", "batch", "vt84f", 8, 1.0, 1.0e5, (32, 32, 32),
              precision="mixed", count=6, nat_hi=96),
        # the largest systems of the serving form: 1024 H at 256^3
        _case("forces 256^3 VT84F", "forces", "vt84f", 1024, 1.0, 3.125e4, (256, 256, 256)),
    ]


def _edge(rng, lo, hi):
    """An even {2,3,5}-smooth edge in [lo, hi], uniform in its logarithm before rounding up."""
    m = int(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.999))))
    while not (m % 2 == 0 and inputs.smooth235(m)):
        m += 1
    return min(m, hi)


def draw(rng):
    kind = rng.choice(["static", "evaluate", "evaluate", "minimise", "md", "forces", "batch"])
    fn = rng.choice(["fttf", "sga", "vt84f", "vt84f", "kst2"])
    T = round(math.exp(rng.uniform(math.log(3.0e4), math.log(1.0e6))), 1)
    rho = round(math.exp(rng.uniform(math.log(0.8), math.log(4.0))), 4)
    lo, hi = {"static": (8, 32), "evaluate": (24, 200), "minimise": (24, 96), "md": (24, 72),
              "forces": (40, 240), "batch": (32, 32)}[kind]
    base = _edge(rng, lo, hi)
    grid = tuple(min(hi, _edge(rng, max(lo, int(0.8 * base)), max(lo, base))) for _ in range(3))
    c = _case("", kind, fn, 8, rho, T, grid)
    del c["name"]
    spacing = rng.uniform(0.2, 0.3)                 # bohr per grid point
    vol = (grid[0] * grid[1] * grid[2]) * spacing ** 3
    per = inputs.cell_edge(1, rho) ** 3             # volume of one atom
    most = {"static": 64, "forces": 1024}.get(kind, 512)
    c["nat"] = int(min(most, max(2, round(vol / per))))
    if kind in ("evaluate", "forces"):
        c["tri"] = rng.random() < 0.25
    if kind in ("minimise", "md"):
        c["precision"] = rng.choice(["fp64", "mixed"])
    if kind == "md":
        c["steps"] = rng.choice([1, 2])
    if kind == "batch":
        c.update(nat=8, count=rng.choice([2, 4, 8]), nat_hi=rng.randint(24, 96), precision="mixed")
    return c


# ------------------------------------------------------------------ inputs
def _system(case, seed):
    grid = (case["nx"], case["ny"], case["nz"])
    d = inputs.hydrogen(case["nat"], case["rho"], case["T"], grid, seed=seed,
                        functional=case["functional"], vel_seed=seed + 1)
    # an orthorhombic cell whose edges follow the grid's, at the same volume
    L0 = d["L"][0]
    edge = np.array(grid, dtype=np.float64)
    L = edge * (L0 ** 3 / edge.prod()) ** (1.0 / 3.0)
    d["ions"] = d["ions"] * (L / L0)
    d["L"] = tuple(L)
    d["cell"] = np.diag(L)
    if case["tri"]:
        shear = np.array([[0.0, 0.0, 0.0], [0.10, 0.0, 0.0], [-0.07, 0.12, 0.0]]) * L.min()
        d["cell"] = np.diag(L) + shear
        d["ions"] = (d["ions"] / L) @ d["cell"]
    return d


def _density(case, d, seed):
    """sqrt of a hydrogen-like density: a uniform part and a Gaussian cloud on
    every ion, with a smooth modulation and a little noise; [nx, ny, nz] on
    the GPU, normalised to the electron number."""
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    grid = (case["nx"], case["ny"], case["nz"])
    frac = torch.as_tensor(d["ions"] @ np.linalg.inv(d["cell"]), device="cuda")
    prof = []
    for a, n in enumerate(grid):
        L = float(np.linalg.norm(d["cell"][a]))
        x = torch.arange(n, dtype=torch.float64, device="cuda") / n
        dx = x[None, :] - frac[:, a:a + 1]
        p = sum(torch.exp(-((dx + s) * L / 0.9) ** 2) for s in (-2, -1, 0, 1, 2))
        prof.append(p)
    n = torch.einsum("ax,ayz->xyz", prof[0], prof[1][:, :, None] * prof[2][:, None, :]) \
        if case["nat"] * grid[1] * grid[2] < 2 ** 27 else _by_chunks(prof)
    n = n / n.mean() + 0.3
    n = n * (1.0 + 0.01 * torch.randn(grid, generator=g, device="cuda", dtype=torch.float64))
    omega = float(np.linalg.det(d["cell"]))
    return torch.sqrt(n * (case["nat"] / omega / n.mean()))


def _by_chunks(prof):
    return sum(torch.einsum("ax,ayz->xyz", prof[0][i:i + 128],
                            prof[1][i:i + 128, :, None] * prof[2][i:i + 128, None, :])
               for i in range(0, prof[0].shape[0], 128))


def _context(case, d):
    return ofdft.Context(None if case["tri"] else d["L"], d["grid"], d["ions"], d["Z"], d["T"], d["functional"],
                         precision=case["precision"], cell=d["cell"] if case["tri"] else None)


def _batch_systems(case, seed):
    r = np.random.default_rng(seed)
    out = []
    for i in range(case["count"]):
        # sizes spread evenly over the range, so that every seed's batch is as much work
        f = (i + 0.5) / case["count"]
        nat = int(round(math.exp(math.log(case["nat"]) + f * math.log(case["nat_hi"] / case["nat"]))))
        rho = math.exp(r.uniform(math.log(0.8), math.log(1.25))) * case["rho"]
        T = math.exp(r.uniform(math.log(0.5), math.log(2.0))) * case["T"]
        edge = inputs.grid_edge(inputs.cell_edge(nat, rho), 0.25, 32, 160)
        fn = ("fttf", "sga", "vt84f")[i % 3]
        d = inputs.hydrogen(nat, rho, T, edge, seed=int(seed) * 100 + i, functional=fn)
        d["cell"] = np.diag(d["L"])
        out.append(d)
    return out


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        ctxs = [_context(dict(case, tri=False), d) for d in _batch_systems(case, seed)]
        return dict(kind=kind, ctxs=ctxs)
    d = _system(case, seed)
    if kind == "static":
        phi = _density(case, d, seed).reshape(-1).contiguous()
        return dict(kind=kind, d=d, phi=phi, v=torch.empty_like(phi))
    s = dict(kind=kind, d=d, ctx=_context(case, d), steps=case.get("steps", 0))
    if kind in ("evaluate", "forces"):
        s["phi"] = _density(case, d, seed).cpu().numpy()
    if kind == "forces":
        s["ctx"].set_phi(s.pop("phi"))
    return s


# -------------------------------------------------------------------- calls
def _split(E):
    return np.array([E[k] for k in KEYS_E]), np.array([E[k] for k in KEYS_P])


def run(state):
    kind = state["kind"]
    if kind == "static":
        d = state["d"]
        E = ofdft.ofdft_energy_potential_static(d["cell"], d["grid"], d["ions"], d["Z"], d["T"], d["functional"],
                                                state["phi"].data_ptr(), state["v"].data_ptr())
        return [*_split(E), state["v"]]
    if kind == "batch":
        for c in state["ctxs"]:
            c.set_phi()
        E, _, st = ofdft.ofdft_batch_minimize([c.ctx for c in state["ctxs"]], gtol=1e-8)
        if st != 0:
            raise RuntimeError("batch status %d" % st)
        return [[*_split(e), c.density()] for e, c in zip(E, state["ctxs"])]
    ctx = state["ctx"]
    if kind == "evaluate":
        E, v = ctx.energy_potential(state["phi"])
        return [*_split(E), v]
    if kind == "forces":
        E, _ = ctx.energy_potential(None, want_v=False)
        F, P = ctx.forces()
        return [*_split(E), F]
    ctx.set_phi()
    if kind == "minimise":
        E, _ = ctx.minimize(gtol=1e-8)
        return [*_split(E), ctx.density()]
    d = state["d"]
    o = ctx.md_step(0.2, d["T"], nsteps=state["steps"], pos=d["ions"], vel=d["vel"], gtol=1e-8)
    return [*_split(o["E"]), o["F"], o["pos"], o["vel"], ctx.density()]


def _evals(case):
    """Typical energy + potential evaluations of a pass (the counts the solver takes at gtol 1e-8)."""
    per = {"fttf": 40, "sga": 150, "vt84f": 500, "kst2": 300}[case["functional"]]
    return {"static": 1, "evaluate": 1, "forces": 2, "minimise": per, "batch": 200,
            "md": per * (1 + case.get("steps", 0))}[case["kind"]]


def work(case):
    """One evaluation reads phi, writes v and makes 17 one-axis transforms of a
    real field (5 for ftTF: three forward, with the inverse's three, each
    2.5 n log2 n flops) and about 200 flops of pointwise functional per
    point; forces add one complex multiply-add per ion and half-spectrum
    point.  A solve repeats the evaluation, but needs only its inputs and
    results moved."""
    if case["kind"] == "batch":
        n = 0.0
        for i in range(case["count"]):
            f = (i + 0.5) / case["count"]
            nat = math.exp(math.log(case["nat"]) + f * math.log(case["nat_hi"] / case["nat"]))
            n += inputs.grid_edge(inputs.cell_edge(int(round(nat)), case["rho"]), 0.25, 32, 160) ** 3
        lg = 5.5
    else:
        n = float(case["nx"] * case["ny"] * case["nz"])
        lg = (math.log2(case["nx"]) + math.log2(case["ny"]) + math.log2(case["nz"])) / 3.0
    transforms = 6 if case["functional"] == "fttf" and case["kind"] != "batch" else 17
    flops = _evals(case) * n * (transforms * 2.5 * lg + 200.0)
    bytes_ = 16.0 * n
    if case["kind"] in ("md", "forces"):
        flops += (1 + case.get("steps", 0)) * case["nat"] * 0.5 * n * 16.0
    return {"bytes": bytes_, "flops": flops}


# ---------------------------------------- the same equations in binary64 torch
def _fermi(eta, want):
    """Integrals of the Fermi function at eta (1-D): I_{1/2}, I_{3/2} and
    I_{-1/2} with its first three derivatives, as want names them.  With
    x = u^2 the integrands are smooth; below u0 = sqrt(eta - 40) the Fermi
    function is 1 and the integral is taken in closed form."""
    key = "_gl"
    if key not in _fermi.__dict__:
        x, w = np.polynomial.legendre.leggauss(24)
        _fermi._gl = (x, w)
    x, w = _fermi._gl
    a = torch.sqrt(torch.clamp(eta - 40.0, min=0.0))
    b = torch.sqrt(torch.clamp(eta, min=0.0) + 40.0)
    out = {k: torch.zeros_like(eta) for k in want}
    if "I12" in want:
        out["I12"] += (2.0 / 3.0) * a ** 3
    if "I32" in want:
        out["I32"] += (2.0 / 5.0) * a ** 5
    if "M0" in want:
        out["M0"] += 2.0 * a
    panels = 12
    h = (b - a) / panels
    for p in range(panels):
        for xi, wi in zip(x, w):
            u = a + h * (p + 0.5 * (xi + 1.0))
            u2 = u * u
            f = torch.sigmoid(eta - u2)
            c = h * (0.5 * wi) * 2.0
            if "I12" in want:
                out["I12"] += c * u2 * f
            if "I32" in want:
                out["I32"] += c * u2 * u2 * f
            if "M0" in want:
                out["M0"] += c * f
            if "M1" in want:
                q = f * torch.sigmoid(u2 - eta)
                out["M1"] += c * q
                out["M2"] += c * q * (1.0 - 2.0 * f)
                out["M3"] += c * q * (1.0 - 6.0 * q)
    return out


def _temperature_functions(t):
    """xi, zeta, A, B and their t-derivatives at reduced temperatures t."""
    y = (2.0 / 3.0) * t ** -1.5
    eta = torch.where(t < 0.6, 1.0 / t - (math.pi ** 2 / 12.0) * t, torch.log(y * (2.0 / math.sqrt(math.pi))))
    for _ in range(12):
        m = _fermi(eta, ("I12", "M0"))
        step = torch.log(m["I12"] / y) * m["I12"] / (0.5 * m["M0"])
        eta = eta - step
        if float(torch.max(torch.abs(step) / (1.0 + torch.abs(eta)))) < 1e-14:
            break
    m = _fermi(eta, ("I12", "I32", "M0", "M1", "M2", "M3"))
    I32, M0, M1, M2, M3 = m["I32"], m["M0"], m["M1"], m["M2"], m["M3"]
    yt = -t ** -2.5
    et = 2.0 * yt / M0
    ett = 5.0 * t ** -3.5 / M0 - 2.0 * yt * M1 * et / M0 ** 2
    kap = (5.0 / 3.0) * t * (eta - (2.0 / 3.0) * I32 / y)
    k1 = (5.0 / 3.0) * (eta - (5.0 / 3.0) * I32 / y)
    k2 = -2.5 * (et + (5.0 / 3.0) * I32 / (y * t))
    h = 6.0 * y * M1 / M0 ** 2
    H1 = 6.0 * (0.5 * M1 / M0 + y * M2 / M0 ** 2 - 2.0 * y * M1 ** 2 / M0 ** 3)
    H2 = 6.0 * (M2 / M0 - 1.5 * M1 ** 2 / M0 ** 2 + y * M3 / M0 ** 2 - 6.0 * y * M1 * M2 / M0 ** 3
                + 6.0 * y * M1 ** 3 / M0 ** 4)
    h1, h2 = H1 * et, H2 * et * et + H1 * ett
    xi, ze, dxi, dze = kap - t * k1, -t * k1, -t * k2, -k1 - t * k2
    A, B = (h - t * h1) / xi, t * h1 / ze
    dA = -t * h2 / xi - (h - t * h1) * dxi / xi ** 2
    dB = (h1 + t * h2) / ze - t * h1 * dze / ze ** 2
    return xi, ze, A, B, dxi, dze, dA, dB


def _enhance(functional, x):
    if functional == "sga":
        return 1.0 + (5.0 / 27.0) * x, torch.full_like(x, 5.0 / 27.0)
    if functional == "kst2":
        den = 1.0 + 0.29424 * x
        return 1.0 + 2.03087 * x / den, 2.03087 / den ** 2
    mu, al = 2.778, 1.2965
    e1, em, den = torch.exp(-al * x), -torch.expm1(-al * x * x), 1.0 + mu * x
    xs = torch.where(x > 1e-150, x, torch.ones_like(x))
    em_x = torch.where(x > 1e-150, em / xs, al * x)
    F = 1.0 - mu * x * e1 / den + em_x - em + (5.0 / 3.0) * x
    em_xx = torch.where(x > 1e-150, em_x / xs, torch.full_like(x, al))
    dF = (-mu * e1 * (1.0 - al * x - al * mu * x * x) / den ** 2
          + 2.0 * al * (1.0 - em) * (1.0 - x) - em_xx + 5.0 / 3.0)
    return F, dF


def _pointwise(functional, T, n, g2):
    """f_s, T s_s, d f_s/dn and W/grad n at points (1-D)."""
    k23 = (3.0 * math.pi ** 2) ** (2.0 / 3.0)
    ctf = 0.3 * k23
    tau0, dtau0 = ctf * n ** (5.0 / 3.0), (5.0 / 3.0) * ctf * n ** (2.0 / 3.0)
    t = 2.0 * T / (k23 * n ** (2.0 / 3.0))
    dtdn = -2.0 * t / (3.0 * n)
    xi, ze, A, B, dxi, dze, dA, dB = _temperature_functions(t)
    if functional == "fttf":
        return (tau0 * (xi - ze), tau0 * ze, dtau0 * (xi - ze) + tau0 * (dxi - dze) * dtdn, torch.zeros_like(n))
    cs = 1.0 / (4.0 * k23 * n ** (8.0 / 3.0))
    s2 = g2 * cs
    xt, xs = s2 * A, s2 * B
    Ft, dFt = _enhance(functional, xt)
    Fg, dFg = _enhance(functional, xs)
    Fs, dFs = 2.0 - Fg, -dFg
    f = tau0 * xi * Ft - tau0 * ze * Fs
    d = (dtau0 * (xi * Ft - ze * Fs) + tau0 * dtdn * (dxi * Ft - dze * Fs)
         + tau0 * xi * dFt * (-8.0 / 3.0 * xt / n + s2 * dA * dtdn)
         - tau0 * ze * dFs * (-8.0 / 3.0 * xs / n + s2 * dB * dtdn))
    return f, tau0 * ze * Fs, d, (tau0 * xi * dFt * A - tau0 * ze * dFs * B) * 2.0 * cs


def _pz81(n):
    g, b1, b2, a, b = -0.1423, 1.0529, 0.3334, 0.0311, -0.048
    den1 = 1.0 + b1 + b2
    D = g / den1 - b
    C = -g * (0.5 * b1 + b2) / den1 ** 2 - a - D     # value and slope continuous at r_s = 1
    rs = (3.0 / (4.0 * math.pi * n)) ** (1.0 / 3.0)
    ex = -0.75 * (3.0 / math.pi) ** (1.0 / 3.0) * n ** (1.0 / 3.0)
    sq, lr = torch.sqrt(rs), torch.log(rs)
    den = 1.0 + b1 * sq + b2 * rs
    hi = rs >= 1.0
    ec = torch.where(hi, g / den, a * lr + b + C * rs * lr + D * rs)
    dec = torch.where(hi, -g * (b1 / (2.0 * sq) + b2) / den ** 2, a / rs + C * (lr + 1.0) + D)
    return ex + ec, (4.0 / 3.0) * ex + ec - rs / 3.0 * dec


def _ewald(cell, R, Z):
    """Ewald energy and forces of point charges in a neutralising background."""
    dev = "cuda"
    A = torch.as_tensor(cell, dtype=torch.float64, device=dev)
    R = torch.as_tensor(R, dtype=torch.float64, device=dev)
    Z = torch.as_tensor(Z, dtype=torch.float64, device=dev)
    om = float(torch.linalg.det(A))
    Bm = 2.0 * math.pi * torch.linalg.inv(A).T
    high = [2.0 * math.pi / float(torch.linalg.norm(Bm[j])) for j in range(3)]
    al = 6.5 / min(high)
    rcut, gcut = 6.5 / al, 13.0 * al
    E, F = 0.0, torch.zeros_like(R)
    ni = [int(math.ceil(rcut / h)) + 1 for h in high]
    fr = R @ torch.linalg.inv(A)
    dfr = fr[:, None, :] - fr[None, :, :]
    dfr = dfr - torch.round(dfr)
    d0 = dfr @ A
    for i in range(-ni[0], ni[0] + 1):
        for j in range(-ni[1], ni[1] + 1):
            for k in range(-ni[2], ni[2] + 1):
                d = d0 + torch.tensor([float(i), float(j), float(k)], dtype=torch.float64, device=dev) @ A
                r2 = (d * d).sum(-1)
                use = (r2 > 1e-20) & (r2 < rcut * rcut)
                if not bool(use.any()):
                    continue
                r = torch.sqrt(torch.where(use, r2, torch.ones_like(r2)))
                zz = torch.where(use, Z[:, None] * Z[None, :], torch.zeros_like(r))
                er = torch.erfc(al * r) / r
                E += 0.5 * float((zz * er).sum())
                mag = zz * (er + 2.0 * al / math.sqrt(math.pi) * torch.exp(-(al * r) ** 2)) / (r * r)
                F += (mag[:, :, None] * d).sum(1)
    km = [int(math.ceil(gcut * float(torch.linalg.norm(A[j])) / (2.0 * math.pi))) for j in range(3)]
    ks = torch.cartesian_prod(*[torch.arange(-m, m + 1, dtype=torch.float64, device=dev) for m in km])
    G = ks @ Bm
    g2 = (G * G).sum(-1)
    sel = (g2 > 0.0) & (g2 < gcut * gcut)
    for Gc, gc in zip(G[sel].split(4096), g2[sel].split(4096)):
        w = torch.exp(-gc / (4.0 * al * al)) / gc
        ph = Gc @ R.T
        c, s = torch.cos(ph), torch.sin(ph)
        Sc, Ss = c @ Z, s @ Z
        E += 2.0 * math.pi / om * float((w * (Sc * Sc + Ss * Ss)).sum())
        F += 4.0 * math.pi / om * Z[:, None] * ((w[:, None] * (Sc[:, None] * s - Ss[:, None] * c)).T @ Gc)
    E -= al / math.sqrt(math.pi) * float((Z * Z).sum())
    E -= math.pi * float(Z.sum()) ** 2 / (2.0 * om * al * al)
    return E, F


def _exact(d, functional, grid, phi, forces):
    """Energies, pressures and the potential (or the forces) at phi, in binary64."""
    dev = "cuda"
    cell = np.asarray(d["cell"], dtype=np.float64)
    om = float(np.linalg.det(cell))
    N = grid[0] * grid[1] * grid[2]
    dV = om / N
    T = d["T"] * inputs.KB_HA_PER_K
    Bm = 2.0 * math.pi * np.linalg.inv(cell).T
    kint, kder = [], []
    for m in grid:
        k = np.fft.fftfreq(m, 1.0 / m)
        k[m // 2] = m // 2
        kd = k.copy()
        kd[m // 2] = 0.0
        kint.append(torch.as_tensor(k, device=dev))
        kder.append(torch.as_tensor(kd, device=dev))
    sh = [(-1, 1, 1), (1, -1, 1), (1, 1, -1)]

    def cart(ks, a):
        return sum(ks[j].reshape(sh[j]) * float(Bm[j, a]) for j in range(3))

    G2 = sum(cart(kint, a) ** 2 for a in range(3)).expand(grid).contiguous()
    n = phi * phi
    nG = torch.fft.fftn(n) / N
    inv = torch.where(G2 > 0.0, 1.0 / torch.where(G2 > 0.0, G2, torch.ones_like(G2)), torch.zeros_like(G2))
    rc = 0.25
    w = -4.0 * math.pi / om * torch.exp(-G2 * (rc * rc / 4.0)) * inv
    frac = torch.as_tensor(d["ions"] @ np.linalg.inv(cell), device=dev)
    Z = torch.as_tensor(d["Z"], device=dev)
    ph = [torch.exp(-2j * math.pi * frac[:, j:j + 1] * kint[j][None, :]) for j in range(3)]
    vG = torch.zeros(grid, dtype=torch.complex128, device=dev)
    for i in range(0, len(d["Z"]), 64):
        zx = (Z[i:i + 64, None] * ph[0][i:i + 64]).T
        yz = (ph[1][i:i + 64, :, None] * ph[2][i:i + 64, None, :]).reshape(zx.shape[1], -1)
        vG += (zx @ yz).reshape(grid)
    vG *= w
    E_H = 0.5 * om * 4.0 * math.pi * float((inv * (nG.real ** 2 + nG.imag ** 2)).sum())
    dot = nG.real * vG.real + nG.imag * vG.imag
    E_loc = om * float(dot.sum())
    P_loc = float((dot * (1.0 - G2 * (rc * rc / 2.0))).sum()) / 3.0
    F = None
    if forces:
        base = (w * torch.conj(nG)).reshape(-1, grid[2])
        F = torch.zeros((len(d["Z"]), 3), dtype=torch.float64, device=dev)
        for i in range(0, len(d["Z"]), 128):
            px, py, pz = (p[i:i + 128] for p in ph)
            S0 = (base @ pz.T).reshape(grid[0], grid[1], -1)
            S1 = (base @ (pz * kint[2]).T).reshape(grid[0], grid[1], -1)
            t = [torch.einsum("xya,ax,ay->a", S0, px * kint[0], py), torch.einsum("xya,ax,ay->a", S0, px, py * kint[1]),
                 torch.einsum("xya,ax,ay->a", S1, px, py)]
            for a in range(3):
                F[i:i + 128, a] = om * Z[i:i + 128] * torch.real(1j * sum(t[j] * float(Bm[j, a]) for j in range(3)))
    vH = torch.fft.ifftn(4.0 * math.pi * inv * nG + vG).real * N
    del vG, dot, inv, w
    gr = None
    g2 = torch.zeros_like(n)
    if functional != "fttf":
        gr = [torch.fft.ifftn(1j * cart(kder, a) * nG).real * N for a in range(3)]
        g2 = gr[0] ** 2 + gr[1] ** 2 + gr[2] ** 2
    parts = [_pointwise(functional, T, a, b) for a, b in zip(n.reshape(-1).split(1 << 20), g2.reshape(-1).split(1 << 20))]
    f, ts, dfdn, wc = (torch.cat(x).reshape(grid) for x in zip(*parts))
    div, wg = 0.0, 0.0
    if gr is not None:
        acc = 0.0
        for a in range(3):
            acc = acc + 1j * cart(kder, a) * torch.fft.fftn(wc * gr[a])
        div = torch.fft.ifftn(acc).real
        wg = dV * float((wc * g2).sum())
    eps, vxc = _pz81(n)
    vs = dfdn - div
    v = vs + vH + vxc
    E_ion, F_ion = _ewald(cell, d["ions"], d["Z"])
    F_s, TS, F_xc = dV * float(f.sum()), dV * float(ts.sum()), dV * float((n * eps).sum())
    tot = F_s + E_H + E_loc + F_xc + E_ion
    Ne = float(Z.sum())
    E = np.array([tot, F_s, -TS, E_H, E_loc, F_xc, E_ion, tot + TS, float((n * v).sum() / n.sum()),
                  Ne * math.pi * rc * rc * Ne / om])
    P_s = (dV * float((n * vs - f).sum()) + wg / 3.0) / om
    P = [P_s, dV * float((n * (vxc - eps)).sum()) / om, E_H / (3.0 * om), P_loc, E_ion / (3.0 * om)]
    return E, np.array([sum(P)] + P), v, None if F is None else F + F_ion


def exact(case, seed):
    if case["kind"] in ("minimise", "md", "batch"):
        return None          # hundreds of evaluations: minutes in plain torch
    d = _system(case, seed)
    grid = (case["nx"], case["ny"], case["nz"])
    phi = _density(case, d, seed)
    if case["kind"] == "forces":
        # set_phi normalises to the electron number (the density is already, to rounding)
        E, P, _, F = _exact(d, case["functional"], grid, phi, True)
        return [E, P, F]
    E, P, v, _ = _exact(d, case["functional"], grid, phi, False)
    return [E, P, v.reshape(-1) if case["kind"] == "static" else v]
