"""The work that a user of the library has it do, as cases to measure.

Each case is one pass through the public entry points: one application of
G, solves of the Born series on the padded grid (the workloads' 256^2 disk
and 2048^2 tissue, ragged sizes), a gradient with stored and with
checkpointed terms, a batched broadband sweep and its time signal, a second
harmonic with its plans built inside, and the paper's periodic iteration
(plain, with the k-space potential, preconditioned).  Sizes are those of the
workloads, the benchmark and the tests, or generic.

Inputs follow from the seed alone: smooth random media, transducer rows with
focused or steered phases and random apodisation.  exact() evaluates the
same quantities with torch in 64 bits from the same inputs, with its own
cell-averaged Green's table.
"""
import math

import numpy as np
import torch

from paper_2507_13754_gb300 import solvers, tbs

DEV = "cuda"
ALPHA_NP_M = 0.5 * 100.0 / (20.0 * math.log10(math.e))  # 0.5 dB/cm in Np/m (at 1 MHz)


# ---- the cases ----------------------------------------------------------------
def listed():
    return [
        # the smallest call: one application of G to one field, as an outer
        # iterative solver of the caller's makes them
        dict(name="green_64", kind="green", n=64, n_rhs=1, conj=False),
        # G^H on a handful of ragged fields (an outer adjoint solver)
        dict(name="green_adj_700x4", kind="green", n=700, n_rhs=4, conj=True),
        # a new medium and new sources on a small grid, 24 terms: the 256^2 disk workload
        dict(name="solve_256", kind="solve", n=256, n_rhs=1, f=1e6, medium="disk", absorbing=False, max_terms=24,
             tol=0.0, n_src=32),
        # an odd size with several sources, to a residual
        dict(name="solve_999x3", kind="solve", n=999, n_rhs=3, f=1e6, medium="tissue", absorbing=True, max_terms=64,
             tol=1e-6, n_src=16),
        # the benchmark's workload: absorbing tissue at 5 MHz, 128-element focused array, to 1e-6
        dict(name="solve_2048", kind="solve", n=2048, n_rhs=1, f=5e6, medium="tissue", absorbing=True, max_terms=64,
             tol=1e-6, n_src=128),
        # one step of an inversion: 16 sources, misfit on a receiver row, gradients in c and alpha
        dict(name="gradient_1024x16", kind="gradient", n=1024, n_rhs=16, max_terms=64, tol=1e-6, checkpoint=False),
        # the same with checkpointed terms on a ragged grid
        dict(name="gradient_ckpt_300x4", kind="gradient", n=300, n_rhs=4, max_terms=48, tol=1e-6, checkpoint=True),
        # a broadband sweep: six frequencies (2 .. 8 MHz over 48 mm: N = 512 .. 2048) x four angles in one batch
        dict(name="sweep_6x4", kind="sweep", n_freq=6, n_ang=4, f_lo=2e6, f_hi=8e6, side=48e-3, terms=24),
        # the time signal of a sweep at a line of receivers
        dict(name="synthesis_32x4", kind="synthesis", n_freq=32, n_rhs=4, f_lo=2e6, f_hi=5e6, side=48e-3, nx=512,
             n_t=672),
        # fundamental and second harmonic in water with a fat ellipse; the call builds both plans
        dict(name="second_harmonic_1024", kind="harmonic2", n=1024, n_rhs=1, f=2e6, max_terms=64, max_terms2=128,
             tol=1e-6, n_src=32),
        # the paper's 4096^2 run with the 1350 m/s cylinder
        dict(name="paper_4096", kind="periodic", n=4096, n_rhs=1, physics="plain", v_s=1350.0, terms=140),
        # its absorbing-dispersive medium on a coarser grid of the same domain
        dict(name="paper_kspace_1024", kind="periodic", n=1024, n_rhs=1, physics="kspace", v_s=0.0, terms=140),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["green", "solve", "solve", "gradient", "sweep", "synthesis", "harmonic2", "periodic", "periodic"])
    if kind == "green":
        n = _log(rng, 17, 2048)
        return dict(kind=kind, n=n, n_rhs=rng.randint(1, 4), conj=rng.random() < 0.5)
    if kind == "solve":
        n = _log(rng, 33, 2048)
        fixed = rng.random() < 0.4
        return dict(kind=kind, n=n, n_rhs=rng.randint(1, 4 if n < 1100 else 2), f=rng.choice([1e6, 2e6, 3e6, 5e6]),
                    medium=rng.choice(["disk", "tissue", "tissue"]), absorbing=rng.random() < 0.6,
                    max_terms=24 if fixed else 64, tol=0.0 if fixed else 1e-6, n_src=_log(rng, 1, max(2, n // 8)))
    if kind == "gradient":
        n = _log(rng, 100, 1024)
        return dict(kind=kind, n=n, n_rhs=rng.randint(1, 8), max_terms=rng.choice([32, 48, 64]), tol=1e-6,
                    checkpoint=rng.random() < 0.4)
    if kind == "sweep":
        lo = rng.uniform(1e6, 4e6)
        return dict(kind=kind, n_freq=rng.randint(2, 6), n_ang=rng.randint(1, 4), f_lo=lo,
                    f_hi=lo * rng.uniform(1.2, 2.0), side=rng.uniform(20e-3, 45e-3), terms=rng.choice([12, 16, 24]))
    if kind == "synthesis":
        lo = rng.uniform(1e6, 2e6)
        return dict(kind=kind, n_freq=rng.randint(3, 80), n_rhs=rng.randint(1, 4), f_lo=lo, f_hi=2.0 * lo,
                    side=rng.uniform(20e-3, 48e-3), nx=_log(rng, 16, 600), n_t=_log(rng, 64, 1500))
    if kind == "harmonic2":
        return dict(kind=kind, n=_log(rng, 120, 1024), n_rhs=rng.randint(1, 2), f=rng.choice([1e6, 2e6]), max_terms=64,
                    max_terms2=128, tol=1e-6, n_src=rng.randint(4, 32))
    physics = rng.choice(["plain", "kspace", "cbs"])
    n = rng.choice([128, 256, 512, 1024, 2048])
    return dict(kind="periodic", n=n, n_rhs=rng.randint(1, 2), physics=physics,
                v_s=0.0 if physics == "kspace" else rng.uniform(1250.0, 1800.0), terms=rng.randint(60, 160))


# ---- inputs: from the case and the seed alone -----------------------------------
def _smooth(n, corr, g):
    """Smooth random field in [-1, 1] with a correlation length of corr cells."""
    k = torch.fft.fftfreq(n, device=DEV, dtype=torch.float64)
    h = torch.exp(-((math.pi * corr) ** 2) * (k[:, None] ** 2 + k[None, :] ** 2) / 2.0)
    w = torch.randn((n, n), generator=g, device=DEV, dtype=torch.float64)
    f = torch.fft.ifft2(torch.fft.fft2(w) * h).real
    return f / f.abs().max()


def _disk(n, cy, cx, ry, rx):
    y = torch.arange(n, device=DEV, dtype=torch.float64)
    return ((y[:, None] - cy) / ry) ** 2 + ((y[None, :] - cx) / rx) ** 2 <= 1.0


def _array(n, count, row):
    """Columns and rows of a transducer row centred on the grid."""
    count = max(1, min(count, n - 2))
    pitch = max(1, min(4, (n - 2) // count))
    first = (n - (count - 1) * pitch) // 2
    ix = (first + pitch * np.arange(count)).astype(np.int32)
    return ix, np.full(count, min(row, n - 1), np.int32)


def _inputs(case, seed):
    """Everything of a case but its plans: numbers, host sources, device fields."""
    g = torch.Generator(device=DEV)
    g.manual_seed(seed * 7919 + 17)
    r = np.random.default_rng([seed, 2507])
    kind = case["kind"]
    s = dict(case)
    if kind == "green":
        n = case["n"]
        s.update(f=1e6, c0=1500.0, dx=1500.0 / 1e6 / 8)
        s["field"] = torch.view_as_complex(torch.randn((case["n_rhs"], n, n, 2), generator=g, device=DEV))
    elif kind == "solve":
        n, f, c0 = case["n"], case["f"], 1540.0
        dx = c0 / f / 8
        if case["medium"] == "disk":
            shift = r.uniform(-0.05, 0.05, 2) * n
            inside = _disk(n, n / 2 + shift[0], n / 2 + shift[1], n * 40 / 256, n * 40 / 256)
            c = torch.where(inside, c0 * 1.02, c0)
        else:
            c = c0 * (1.0 + 0.02 * _smooth(n, max(2.0, 1e-3 / dx), g))
        alpha = None
        if case["absorbing"]:
            a = ALPHA_NP_M * (f / 1e6) ** 1.1
            alpha = (a * (1.0 + 0.3 * _smooth(n, max(2.0, n / 16), g))).float()
        ix, iy = _array(n, case["n_src"], min(16, n // 8))
        k0 = 2 * math.pi * f / c0
        foc = min(40e-3, 0.5 * n * dx)
        amp = []
        for _ in range(case["n_rhs"]):
            x = (ix - n / 2 - r.uniform(-0.1, 0.1) * n) * dx
            amp.append((1 + 0.2 * r.standard_normal(ix.size)) * np.exp(-1j * k0 * (np.sqrt(x * x + foc * foc) - foc)))
        s.update(c0=c0, dx=dx, ypow=1.1, fref=0.8 * f, c=c.float(), alpha=alpha, ix=ix, iy=iy,
                 amp=np.array(amp).astype(np.complex64))
    elif kind == "gradient":
        n, f, c0 = case["n"], 3e6, 1540.0
        dx = c0 / f / 8
        c = (c0 * (1.0 + 0.01 * _smooth(n, n / 10, g))).float()
        alpha = (ALPHA_NP_M * 3.0 ** 1.1 * (1.0 + 0.2 * _smooth(n, n / 10, g))).float()
        m = case["n_rhs"]
        ix = np.round((np.arange(m) + 0.5) * n / m + r.uniform(-0.2, 0.2, m) * n / m).astype(np.int32)
        iy = np.full(m, max(1, 24 * n // 1024), np.int32)
        amp = np.diag((1 + 0.1 * r.standard_normal(m)) * np.exp(2j * math.pi * r.random(m))).astype(np.complex64)
        data = 0.02 * torch.view_as_complex(torch.randn((m, n, 2), generator=g, device=DEV))
        s.update(f=f, c0=c0, dx=dx, ypow=1.1, fref=f, c=c, alpha=alpha, ix=ix, iy=iy, amp=amp, data=data,
                 row=1000 * n // 1024)
    elif kind == "sweep":
        parts, c0 = [], 1500.0
        th = np.deg2rad(np.linspace(-30.0, 30.0, case["n_ang"]) + r.uniform(-3, 3))
        off = r.uniform(-0.05, 0.05, 2)
        for k in range(case["n_freq"]):
            f = case["f_lo"] + (case["f_hi"] - case["f_lo"]) * k / (case["n_freq"] - 1)
            dx = c0 / f / 8
            n = int(round(case["side"] / dx))
            inside = _disk(n, n * (0.5 + off[0]), n * (0.5 + off[1]), n * 7.5 / 48, n * 7.5 / 48)
            ix = np.clip(np.round((112 + np.arange(32)) / 256 * n), 0, n - 1).astype(np.int32)
            iy = np.full(32, int(round(n / 16)), np.int32)
            w = math.exp(-(((f - 5e6) / 1.5e6) ** 2))
            x = (ix - n / 2) * dx
            amp = np.stack([w * np.exp(-2j * math.pi * f / c0 * x * math.sin(t)) for t in th]).astype(np.complex64)
            parts.append(dict(n=n, f=f, dx=dx, c0=c0, c=torch.where(inside, 1530.0, c0).float(), ix=ix, iy=iy, amp=amp))
        s["parts"] = parts
    elif kind == "synthesis":
        c0, nf = 1500.0, case["n_freq"]
        fs = [case["f_lo"] + (case["f_hi"] - case["f_lo"]) * k / max(1, nf - 1) for k in range(nf)]
        dxs = [c0 / f / 8 for f in fs]
        ns = [int(round(case["side"] / d)) for d in dxs]
        s["fields"] = [0.1 * torch.view_as_complex(torch.randn((case["n_rhs"], n, n, 2), generator=g, device=DEV))
                       for n in ns]
        df = (fs[-1] - fs[0]) / max(1, nf - 1)
        s.update(fs=fs, dxs=dxs, ws=[df * math.exp(-(((f - 3e6) / 1.5e6) ** 2)) for f in fs],
                 y0=(0.75 + r.uniform(-0.1, 0.1)) * case["side"], sx=case["side"] / max(1, case["nx"] - 1),
                 dt=1.0 / df / case["n_t"])
    elif kind == "harmonic2":
        n, f, c0 = case["n"], case["f"], 1500.0
        shift = r.uniform(-0.05, 0.05, 2) * n
        inside = _disk(n, n / 2 + shift[0], n / 2 + shift[1], n / 24, n / 48)
        ix, iy = _array(n, case["n_src"], min(16, n // 8))
        amp = 1e6 * (1 + 0.2 * r.standard_normal((case["n_rhs"], ix.size)))
        s.update(c0=c0, dx=c0 / f / 8, ypow=2.0, c=torch.where(inside, 1450.0, c0).float(),
                 beta=torch.where(inside, 5.0, 3.5).float(), rho=torch.full((n, n), 1000.0, device=DEV),
                 alpha=torch.full((n, n), 0.0022 * 2 * ALPHA_NP_M * (f / 1e6) ** 2, device=DEV), ix=ix, iy=iy,
                 amp=amp.astype(np.complex64))
    else:
        # the paper's 81.92 mm domain, 10 mm line source and absorbing layer on an n^2 grid
        n, c0, f = case["n"], 1500.0, 1007080.0
        q = 4096 // n
        dx = 2e-5 * q
        c = torch.full((n, n), c0, device=DEV)
        if case["v_s"]:
            rad, cx = 1e-3 / dx, (675 + 2010) / q + r.uniform(-0.02, 0.02) * n
            c = torch.where(_disk(n, n / 2, cx, rad, rad), case["v_s"], c).float()
        half = max(1, 250 // q)
        iy = np.arange(n // 2 - half, n // 2 + half + 1, dtype=np.int32)
        ix = np.full_like(iy, 675 // q)
        amp = -1e6j * dx * dx * (1 + 0.2 * r.standard_normal((case["n_rhs"], iy.size)))
        s.update(c0=c0, f=f, dx=dx, c=c.float().contiguous(), ix=ix, iy=iy, amp=amp.astype(np.complex64), layer=450 // q)
    return s


# ---- what a user's program holds, and one pass ------------------------------------
def _periodic_args(s):
    kw = dict(stop_mode=tbs.TBS_STOP_L1_ROW, periodic=True, abl_width=s["layer"], abl_zeta=2148.0,
              div_window=1 << 30, div_factor=math.inf)
    if s["physics"] == "kspace":
        kw.update(kspace_alpha0=5.5e-10, kspace_nu=1.5)
    if s["physics"] == "cbs":
        kw.update(cbs=True, eps_factor=0.0)
    return kw


def _records(n_rhs):
    return torch.zeros(n_rhs * 32, dtype=torch.uint8, device=DEV)


def _terms(info, n_rhs):
    """Terms and status of each right-hand side, from the device records."""
    return info.view(torch.int32).view(n_rhs, 8)[:, :2]


def prepare(case, seed):
    s = _inputs(case, seed)
    kind = case["kind"]
    if kind == "green":
        s["plan"] = tbs.Plan(s["n"], s["dx"], s["f"], s["c0"], n_rhs=s["n_rhs"], max_terms=1)
    elif kind == "solve":
        s["plan"] = tbs.Plan(s["n"], s["dx"], s["f"], s["c0"], n_rhs=s["n_rhs"], max_terms=s["max_terms"], tol=s["tol"])
        s["info"] = _records(s["n_rhs"])
    elif kind == "gradient":
        s["plan"] = tbs.Plan(s["n"], s["dx"], s["f"], s["c0"], n_rhs=s["n_rhs"], max_terms=s["max_terms"], tol=s["tol"],
                             keep_terms=True, checkpoint=s["checkpoint"])
        s["c"].requires_grad_(True)
        s["alpha"].requires_grad_(True)
    elif kind == "sweep":
        plans = [tbs.Plan(p["n"], p["dx"], p["f"], p["c0"], n_rhs=s["n_ang"], max_terms=s["terms"], tol=0.0,
                          div_window=1 << 30, div_factor=math.inf) for p in s["parts"]]
        s["batch"] = tbs.Batch(plans)
    elif kind == "periodic":
        s["plan"] = tbs.Plan(s["n"], s["dx"], s["f"], s["c0"], n_rhs=s["n_rhs"], max_terms=s["terms"], tol=0.0,
                             **_periodic_args(s))
        s["info"] = _records(s["n_rhs"])
    return s


def run(s):
    kind = s["kind"]
    if kind == "green":
        return s["plan"].apply_green(s["field"], conj_kernel=s["conj"])
    if kind == "solve":
        p = s["plan"]
        p.set_medium(s["c"], s["alpha"], s["ypow"], s["fref"])
        p.set_sources(s["ix"], s["iy"], s["amp"])
        psi, info = p.solve(sync=False, info=s["info"])
        return {"psi": psi, "terms": _terms(info, s["n_rhs"])}
    if kind == "gradient":
        psi = solvers.TBSField.apply(s["c"], s["alpha"], s["plan"], s["ix"], s["iy"], s["amp"], s["ypow"], s["fref"])
        d = psi[:, s["row"], :] - s["data"]
        loss = 0.5 * torch.view_as_real(d).square().sum()
        gc, ga = torch.autograd.grad(loss, (s["c"], s["alpha"]))
        return {"psi": psi.detach(), "grad_c": gc, "grad_alpha": ga}
    if kind == "sweep":
        b = s["batch"]
        for p, q in zip(b.plans, s["parts"]):
            p.set_medium(q["c"], None, 1.0, q["f"])
            p.set_sources(q["ix"], q["iy"], q["amp"])
        b.solve()
        return list(b.psi)
    if kind == "synthesis":
        return tbs.synthesize(s["fields"], s["dxs"], s["fs"], s["ws"], (0.0, s["y0"]), (s["sx"], 0.0), (s["nx"], 1),
                              0.0, s["dt"], s["n_t"])
    if kind == "harmonic2":
        psi1, i1, psi2, i2 = solvers.second_harmonic(
            s["n"], s["dx"], s["f"], s["c0"], s["c"], s["alpha"], s["ypow"], s["beta"], s["rho"], s["ix"], s["iy"],
            s["amp"], max_terms=s["max_terms"], tol=s["tol"], n_rhs=s["n_rhs"], max_terms_harmonic=s["max_terms2"])
        return {"psi1": psi1, "psi2": psi2, "terms": [i["terms"] for i in i1 + i2]}
    p = s["plan"]
    p.set_medium(s["c"], None, 1.0, s["f"])
    p.set_sources(s["ix"], s["iy"], s["amp"])
    psi, info = p.solve(sync=False, info=s["info"])
    return {"psi": psi, "terms": _terms(info, s["n_rhs"])}


# ---- what a pass cannot do without --------------------------------------------------
def _padded(n):
    m = 16
    while m < 2 * n - 1:
        m *= 2
    return m


def _green_flops(n, rhs):
    """One padded G: the transforms of the n nonzero rows and of every column, both ways, and the product."""
    m = _padded(n)
    return rhs * (2 * (n + m) * 5.0 * m * math.log2(m) + 6.0 * m * m)


def work(case):
    kind, r = case["kind"], case.get("n_rhs", 1)
    if kind == "green":
        n = case["n"]
        return {"bytes": 16 * r * n * n + 8 * (_padded(n) // 2 + 1) ** 2, "flops": _green_flops(n, r)}
    if kind == "solve":
        n = case["n"]
        t = case["max_terms"] if case["tol"] == 0 else 8  # to a residual: at least so many
        return {"bytes": (8 + 8 * r) * n * n + 8 * (_padded(n) // 2 + 1) ** 2, "flops": t * (_green_flops(n, r) + 16.0 * r * n * n)}
    if kind == "gradient":
        n = case["n"]
        return {"bytes": (16 + 8 * r) * n * n + 8 * (_padded(n) // 2 + 1) ** 2, "flops": 2 * 6 * _green_flops(n, r)}
    if kind == "sweep":
        b = f = 0.0
        for k in range(case["n_freq"]):
            n = int(round(case["side"] * 8 * (case["f_lo"] + (case["f_hi"] - case["f_lo"]) * k / (case["n_freq"] - 1)) / 1500.0))
            b += (4 + 8 * case["n_ang"]) * n * n + 8 * (_padded(n) // 2 + 1) ** 2
            f += case["terms"] * (_green_flops(n, case["n_ang"]) + 16.0 * case["n_ang"] * n * n)
        return {"bytes": b, "flops": f}
    if kind == "synthesis":
        k = case["n_freq"]
        return {"bytes": 8.0 * r * case["nx"] * (case["n_t"] + 4 * k), "flops": 8.0 * r * case["nx"] * case["n_t"] * k}
    if kind == "harmonic2":
        n = case["n"]
        return {"bytes": (16 + 16 * r) * n * n, "flops": 2 * 10 * _green_flops(n, r)}
    n, t = case["n"], case["terms"]
    return {"bytes": (4 + 8 * r) * n * n, "flops": t * r * (4 * 5.0 * n * n * math.log2(n) + 30.0 * n * n)}


# ---- the same in 64 bits --------------------------------------------------------------
def _bessel(r, k0):
    z = k0 * r
    return torch.complex(-0.25 * torch.special.bessel_y0(z), 0.25 * torch.special.bessel_j0(z))


def _green_table(n, k0, dx):
    """(1/dx^2) x the integral of (i/4) H0^(1)(k0 r) over each cell, offsets 0 .. n-1 in both axes."""
    i = torch.arange(n, device=DEV, dtype=torch.float64)
    out = torch.zeros((n, n), device=DEV, dtype=torch.complex128)

    def cells(size, order):
        x, w = np.polynomial.legendre.leggauss(order)
        t = torch.zeros((size, size), device=DEV, dtype=torch.complex128)
        for a in range(order):
            for b in range(order):
                px, py = (i[:size] + 0.5 * x[a]) * dx, (i[:size] + 0.5 * x[b]) * dx
                t += 0.25 * w[a] * w[b] * _bessel(torch.hypot(px[None, :], py[:, None]), k0)
        return t

    out += cells(n, 6)
    q = min(n, 4)
    out[:q, :q] = cells(q, 20)
    # the self cell: eight triangles in polar coordinates, the logarithm in closed form
    x, w = np.polynomial.legendre.leggauss(32)
    th, wt = (x + 1) * math.pi / 8, w * math.pi / 8
    big = 0.5 * dx / np.cos(th)
    r = torch.tensor(0.5 * big[:, None] * (x + 1)[None, :], device=DEV)
    wr = torch.tensor(0.5 * big[:, None] * w[None, :] * wt[:, None], device=DEV) * r
    v = 8.0 * (wr * (_bessel(r, k0) + torch.log(r) / (2 * math.pi))).sum() / dx ** 2
    out[0, 0] = v - (math.log(0.5 * dx) + 0.5 * (math.log(2.0) - 3.0 + 0.5 * math.pi)) / (2 * math.pi)
    return out


class _Padded:
    """G of the padded grid, one field at a time."""

    def __init__(self, n, dx, f, c0):
        self.n, self.m, self.dx = n, _padded(n), dx
        t = _green_table(n, 2 * math.pi * f / c0, dx)
        full = torch.zeros((self.m, self.m), device=DEV, dtype=torch.complex128)
        idx = torch.arange(n, device=DEV)
        neg = (self.m - idx) % self.m
        for iy in (idx, neg):
            for ix in (idx, neg):
                full[iy[:, None], ix[None, :]] = t
        self.gh = torch.fft.fft2(full) * dx * dx

    def __call__(self, u, conj=False):
        s = torch.fft.fft2(u, s=(self.m, self.m))
        s *= self.gh.conj() if conj else self.gh
        return torch.fft.ifft2(s)[: self.n, : self.n]


def _momentum(c, alpha, f, ypow, fref):
    p = (2 * math.pi * f / c.detach().double()).to(torch.complex128)
    tdel = 0.0
    if alpha is not None:
        tdel = math.tan(math.pi * ypow / 2) * (1.0 - (fref / f) ** (ypow - 1.0))
        p = p + alpha.detach().double() * complex(tdel, 1.0)
    return p, tdel


def _source(n, dx, ix, iy, amp):
    s = np.zeros((n, n), np.complex128)
    np.add.at(s, (iy, ix), amp.astype(np.complex128) / dx ** 2)
    return torch.from_numpy(s).to(DEV)


def _series(g, v, src, max_terms, tol, keep=None):
    u = g(src)
    psi = torch.zeros_like(u)
    for t in range(max_terms):
        if t:
            u = g(v * u)
        psi = psi + u
        if keep is not None:
            keep.append(u)
        if tol and float(torch.linalg.vector_norm(u)) < tol * float(torch.linalg.vector_norm(psi)):
            break
    return psi, t + 1


def _exact_periodic(s):
    n, dx, k2 = s["n"], s["dx"], (2 * math.pi * s["f"] / s["c0"]) ** 2
    u = (2 * math.pi * s["f"] / s["c"].double()) ** 2 - k2
    eps = 1.01 * float(u.abs().max()) if s["physics"] == "cbs" else 0.8 * k2
    p = torch.fft.fftfreq(n, device=DEV, dtype=torch.float64) * (2 * math.pi / dx)
    p2 = p[:, None] ** 2 + p[None, :] ** 2
    gt = 1.0 / torch.complex(p2 - k2, torch.full_like(p2, -eps))
    i = torch.arange(n, device=DEV, dtype=torch.float64)
    edge = torch.minimum(i, n - 1 - i)
    a1 = torch.where(edge < s["layer"], 1.0 / (1.0 + torch.exp(-2148.0 * (edge * dx - 0.5 * s["layer"] * dx))), 1.0)
    a2 = a1[:, None] * a1[None, :]
    v = torch.complex(u, torch.full_like(u, -eps))
    green = lambda x: torch.fft.ifft2(gt * torch.fft.fft2(x))  # noqa: E731
    if s["physics"] == "kspace":
        a0, nu, w = 5.5e-10, 1.5, 2 * math.pi * s["f"]
        tau, eta = -2 * a0 * s["c0"] ** (nu - 1), 2 * a0 * s["c0"] ** nu * math.tan(math.pi * nu / 2)
        pm = p2.sqrt()
        gv = gt * torch.complex(eta * pm ** (nu + 1), -(tau * w * pm ** nu + eps))
    out = []
    for r in range(s["n_rhs"]):
        src = _source(n, dx, s["ix"], s["iy"], s["amp"][r])
        psi0 = psi = green(src)
        for _ in range(s["terms"] - 1):
            if s["physics"] == "kspace":
                psi = a2 * (torch.fft.ifft2(gv * torch.fft.fft2(psi)) + psi0)
            elif s["physics"] == "cbs":
                psi = a2 * (psi + (1j / eps) * v * (green(v * psi + src) - psi))
            else:
                psi = a2 * green(v * psi + src)
        out.append(psi)
    return {"psi": torch.stack(out), "terms": None}


def exact(case, seed):
    s = _inputs(case, seed)
    kind = case["kind"]
    if kind == "green":
        g = _Padded(s["n"], s["dx"], s["f"], s["c0"])
        return torch.stack([g(x.to(torch.complex128), s["conj"]) for x in s["field"]])
    if kind == "solve":
        g = _Padded(s["n"], s["dx"], s["f"], s["c0"])
        p, _ = _momentum(s["c"], s["alpha"], s["f"], s["ypow"], s["fref"])
        v = p * p - (2 * math.pi * s["f"] / s["c0"]) ** 2
        psi = [_series(g, v, _source(s["n"], s["dx"], s["ix"], s["iy"], a), s["max_terms"], s["tol"])[0] for a in s["amp"]]
        return {"psi": torch.stack(psi), "terms": None}
    if kind == "gradient":
        n = s["n"]
        g = _Padded(n, s["dx"], s["f"], s["c0"])
        p, tdel = _momentum(s["c"], s["alpha"], s["f"], s["ypow"], s["fref"])
        v = p * p - (2 * math.pi * s["f"] / s["c0"]) ** 2
        psis, q = [], torch.zeros((n, n), device=DEV, dtype=torch.complex128)
        for r in range(s["n_rhs"]):
            us = []
            psi, t = _series(g, v, _source(n, s["dx"], s["ix"], s["iy"], s["amp"][r]), s["max_terms"], s["tol"], us)
            psis.append(psi)
            gr = torch.zeros_like(psi)
            gr[s["row"]] = psi[s["row"]] - s["data"][r]
            ub = gr
            for j in range(t - 2, -1, -1):
                lam = g(ub, conj=True)
                q += lam.conj() * us[j]
                ub = gr + v.conj() * lam
        c = s["c"].double()
        return {"psi": torch.stack(psis), "grad_c": (q * 2 * p * (-2 * math.pi * s["f"] / c ** 2)).real,
                "grad_alpha": (q * 2 * p * complex(tdel, 1.0)).real}
    if kind == "sweep":
        out = []
        for q in s["parts"]:
            g = _Padded(q["n"], q["dx"], q["f"], q["c0"])
            p, _ = _momentum(q["c"], None, q["f"], 1.0, q["f"])
            v = p * p - (2 * math.pi * q["f"] / q["c0"]) ** 2
            out.append(torch.stack([_series(g, v, _source(q["n"], q["dx"], q["ix"], q["iy"], a), s["terms"], 0.0)[0]
                                    for a in q["amp"]]))
        return out
    if kind == "synthesis":
        x = torch.arange(s["nx"], device=DEV, dtype=torch.float64) * s["sx"]
        t = torch.arange(s["n_t"], device=DEV, dtype=torch.float64) * s["dt"]
        out = torch.zeros((s["n_rhs"], s["nx"], s["n_t"]), device=DEV, dtype=torch.complex128)
        for f, dx, w, fld in zip(s["fs"], s["dxs"], s["ws"], s["fields"]):
            n = fld.shape[-1]
            u = (x / dx).clamp(0, n - 1)
            i0 = u.floor().long().clamp(max=n - 2)
            fx = u - i0
            vy = min(max(s["y0"] / dx, 0.0), n - 1)
            j0 = min(int(vy), n - 2)
            fy = vy - j0
            rows = (1 - fy) * fld[:, j0].to(torch.complex128) + fy * fld[:, j0 + 1].to(torch.complex128)
            a = (1 - fx) * rows[:, i0] + fx * rows[:, i0 + 1]
            cyc = f * t
            ph = torch.exp(torch.complex(torch.zeros_like(cyc), -2 * math.pi * (cyc - cyc.round())))
            out += w * a[:, :, None] * ph
        return out[:, None]
    if kind == "harmonic2":
        n, f, k0 = s["n"], s["f"], 2 * math.pi * s["f"] / s["c0"]
        xi = s["beta"].double() / (s["rho"].double() * s["c"].double() ** 4)
        psi1, psi2 = [], []
        g = _Padded(n, s["dx"], f, s["c0"])
        p, _ = _momentum(s["c"], s["alpha"], f, s["ypow"], f)
        for a in s["amp"]:
            psi1.append(_series(g, p * p - k0 ** 2, _source(n, s["dx"], s["ix"], s["iy"], a), s["max_terms"], s["tol"])[0])
        g = _Padded(n, s["dx"], 2 * f, s["c0"])
        p, _ = _momentum(s["c"], s["alpha"] * 2.0 ** s["ypow"], 2 * f, s["ypow"], 2 * f)
        for u in psi1:
            src = -0.5 * xi * (4 * math.pi * f) ** 2 * u * u
            psi2.append(_series(g, p * p - 4 * k0 ** 2, src, s["max_terms2"], s["tol"])[0])
        return {"psi1": torch.stack(psi1), "psi2": torch.stack(psi2), "terms": None}
    return _exact_periodic(s)
