"""The work a user of this framework has it do, as measurable cases.

Every case goes through the package's public classes.  Sizes and parameters
are those of the repository's tests and benchmark or generic; fields are what a
run is made of: the developed states of nearly every step of a coarsening run
(smooth domains and interfaces), the random fields of solver right-hand sides,
and rest (C = 0) for the Cahn-Hilliard-Cook runs.
"""
import math

import torch

import paper_2101_06550_gb300 as chx

PI2 = 2.0 * math.pi


def listed():
    return [
        # one small simulation advanced and watched step by step: launches and latency
        {"name": "step_f64_128", "kind": "step", "precision": "f64", "nx": 128, "ny": 128, "lx": PI2, "ly": PI2,
         "gamma": 0.01, "dt": 1e-3, "nsteps": 1},
        # a rectangular domain with unequal spacing and segment lengths that are no power of two
        {"name": "step_f64_600x450", "kind": "step", "precision": "f64", "nx": 600, "ny": 450, "lx": 7.0, "ly": 3.0,
         "gamma": 0.01, "dt": 1e-4, "nsteps": 2},
        # the single large run of the benchmark
        {"name": "step_f64_2048", "kind": "step", "precision": "f64", "nx": 2048, "ny": 2048, "lx": PI2, "ly": PI2,
         "gamma": 0.005, "dt": 5e-4, "nsteps": 2},
        # mixed precision: a medium grid, and the single large run
        {"name": "step_f32r_512", "kind": "step", "precision": "f32r", "nx": 512, "ny": 512, "lx": PI2, "ly": PI2,
         "gamma": 0.01, "dt": 1e-3, "nsteps": 4},
        {"name": "step_f32r_2048", "kind": "step", "precision": "f32r", "nx": 2048, "ny": 2048, "lx": PI2, "ly": PI2,
         "gamma": 0.005, "dt": 5e-4, "nsteps": 2},
        # simulations of uneven sizes and coefficients advanced together, then read back
        {"name": "ensemble_f32r_18", "kind": "ensemble", "n0": 128, "cap0": 8, "n1": 256, "cap1": 6, "n2": 512,
         "cap2": 4, "dt": 1e-3, "nsteps": 8},
        # thermal forcing from rest, deviates drawn on the device
        {"name": "cook_f64_1024", "kind": "cook", "precision": "f64", "nx": 1024, "ny": 1024, "lx": PI2, "ly": PI2,
         "gamma": 0.01, "dt": 1e-3, "sigma": 1e-14, "nsteps": 2},
        # the batched solvers: one matrix for all systems, and one per system factorised anew for every solve
        {"name": "penta_1024x65536", "kind": "penta", "mode": "uniform", "dtype": "f64", "n": 1024, "batch": 65536,
         "sigma": 7.0e3},
        {"name": "penta_rewrite_512x16384", "kind": "penta", "mode": "rewrite", "dtype": "f64", "n": 512,
         "batch": 16384, "sigma": 20.0},
        # the batched one-dimensional time steps
        {"name": "ch1d_256x262144", "kind": "ch1d", "n": 256, "batch": 262144, "gamma": 0.01, "nsteps": 1},
        {"name": "cn_diffusion_1024x65536", "kind": "cn1d", "order": 2, "rewrite": False, "n": 1024, "batch": 65536,
         "dt": 1e-5, "nsteps": 1},
        # what a coarsening study samples: mass, free energy, s and k1 of a field
        {"name": "observables_1024", "kind": "observables", "nx": 1024, "ny": 1024, "lx": PI2, "ly": PI2,
         "gamma": 0.01},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _size(rng, lo, hi):
    """A size on [lo, hi], spread over the logarithm: half of them multiples of 32, the rest any number."""
    n = _log_int(rng, lo, hi)
    return max(lo, n // 32 * 32) if n >= 64 and rng.random() < 0.5 else n


def draw(rng):
    kind = rng.choice(["step", "step", "step", "ensemble", "cook", "penta", "penta", "tri", "ch1d", "cn1d",
                       "observables"])
    if kind in ("step", "cook", "observables"):
        nx = _size(rng, 128, 2048)
        ny = nx if rng.random() < 0.5 else _size(rng, max(128, nx // 3), min(2048, 3 * nx))
        dx = PI2 / _log_int(rng, max(128, min(nx, ny) // 2), max(nx, ny))
        dy = dx if nx == ny or rng.random() < 0.5 else dx * rng.uniform(0.8, 1.25)
        case = {"kind": kind, "nx": nx, "ny": ny, "lx": nx * dx, "ly": ny * dy,
                "gamma": rng.choice([0.005, 0.01, 0.02])}
        if kind == "observables":
            return case
        # implicit coefficients (2/3) gamma dt / dx^4 up to 2e4, as the large run has
        case["dt"] = min(1e-3, 3e4 * min(dx, dy) ** 4 / case["gamma"])
        case["precision"] = rng.choice(["f64", "f32r"])
        case["nsteps"] = rng.randint(1, 4) if nx * ny < 1 << 18 else rng.randint(1, 2) if nx * ny < 1 << 20 else 1
        if kind == "cook":
            case["sigma"] = 1e-14
        return case
    if kind == "ensemble":
        n = sorted(_size(rng, 96, 512) for _ in range(3))
        return {"kind": kind, "n0": n[0], "cap0": rng.randint(2, 8), "n1": n[1], "cap1": rng.randint(1, 6), "n2": n[2],
                "cap2": rng.randint(1, 4), "dt": 1e-3, "nsteps": rng.randint(2, 8)}
    if kind in ("penta", "tri"):
        mode = rng.choice(["uniform", "rewrite"])
        n = _size(rng, 64, 1024)
        most = (3 << 21 if mode == "rewrite" else 1 << 26) // n
        dtype = rng.choice(["f64", "f64", "f32", "refine"]) if kind == "penta" and mode == "uniform" else "f64"
        return {"kind": kind, "mode": mode, "dtype": dtype, "n": n, "batch": _size(rng, 1024, max(1025, most)),
                "sigma": 10 ** rng.uniform(0, 1.7 if dtype == "f32" else 4)}
    n = _size(rng, 64, 1024)
    batch = _size(rng, 2048, (1 << 26) // n)
    if kind == "ch1d":
        return {"kind": kind, "n": n, "batch": batch, "gamma": 0.01, "nsteps": 1}
    order, rewrite = rng.choice([2, 4]), rng.random() < 0.3
    if rewrite:
        batch = min(batch, (3 << 20) // n)
    return {"kind": kind, "order": order, "rewrite": rewrite, "n": n, "batch": batch,
            "dt": 10 ** rng.uniform(-9, -7) if order == 4 else 10 ** rng.uniform(-6, -4), "nsteps": 1}


# -- inputs ---------------------------------------------------------------------------------------------------------

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _uniform(g, shape, lo, hi):
    return torch.rand(shape, generator=g, device="cuda", dtype=torch.float64).mul_(hi - lo).add_(lo)


def _smooth(g, ny, nx, lx, ly, length):
    """A zero-mean, unit-variance random field with the given correlation length."""
    f = torch.fft.rfft2(torch.randn((ny, nx), generator=g, device="cuda", dtype=torch.float64))
    ky = torch.fft.fftfreq(ny, ly / ny / PI2, device="cuda", dtype=torch.float64)[:, None]
    kx = torch.fft.rfftfreq(nx, lx / nx / PI2, device="cuda", dtype=torch.float64)[None, :]
    f *= torch.exp(-0.5 * length ** 2 * (kx ** 2 + ky ** 2))
    f[0, 0] = 0
    u = torch.fft.irfft2(f, s=(ny, nx))
    return u / u.std()


def _fields(g, ny, nx, lx, ly, gamma, dt):
    """C^n and C^{n-1} of a coarsening state: domains of +-1 with interfaces a few sqrt(gamma) wide."""
    length = 4.0 * math.sqrt(gamma)
    now = torch.tanh(1.5 * _smooth(g, ny, nx, lx, ly, length)).mul_(0.95)
    return now, now - dt * _smooth(g, ny, nx, lx, ly, length)


def _step_inputs(case, seed):
    if case["kind"] == "cook":
        z = torch.zeros((case["ny"], case["nx"]), dtype=torch.float64, device="cuda")
        return z, z.clone()
    return _fields(_gen(seed), case["ny"], case["nx"], case["lx"], case["ly"], case["gamma"], case["dt"])


def _groups(case):
    return [(case["n%d" % k], case["cap%d" % k], [0.005, 0.01, 0.02]) for k in range(3)]


def _ensemble_inputs(case, seed):
    """(n, side, [(gamma, C^n, C^{n-1}) per slot]) of every group."""
    g = _gen(seed)
    out = []
    for n, cap, gammas in _groups(case):
        side = n * PI2 / 256
        out.append((n, side, [(gammas[s % 3], *_fields(g, n, n, side, side, gammas[s % 3], case["dt"]))
                              for s in range(cap)]))
    return out


def _band_rows(case, seed):
    """PER_SYSTEM rows of I + D^T K D, K > 0 varying by row and system: D the second (penta) or first (tri)
    periodic difference.  Interleaved [n, batch] diagonals from the leftmost to the rightmost."""
    k = _uniform(_gen(seed + 7919), (case["n"], case["batch"]), 0.5 * case["sigma"], 1.5 * case["sigma"])
    up, dn = torch.roll(k, -1, 0), torch.roll(k, 1, 0)  # k_{i+1}, k_{i-1}
    if case["kind"] == "tri":  # fluxes k_i between points i - 1 and i
        return [-k, 1.0 + k + up, -up]
    return [dn, -2.0 * (dn + k), 1.0 + dn + 4.0 * k + up, -2.0 * (k + up), up]


def _uniform_row(case):
    s = case["sigma"]
    return [s, -4 * s, 1 + 6 * s, -4 * s, s] if case["kind"] == "penta" else [-s, 1 + 2 * s, -s]


def _rhs(case, seed):
    dtype = torch.float32 if case["dtype"] == "f32" else torch.float64
    return _uniform(_gen(seed), (case["n"], case["batch"]), -1.0, 1.0).to(dtype)


def _batched(case, seed):
    """Interleaved 1D states: the small random fields of a quench (ch1d), smooth waves (Crank-Nicolson)."""
    g = _gen(seed)
    if case["kind"] == "ch1d":
        return _uniform(g, (case["n"], case["batch"]), -0.1, 0.1)
    x = torch.arange(case["n"], device="cuda", dtype=torch.float64)[:, None] / case["n"]
    phase = _uniform(g, (1, case["batch"]), 0.0, PI2)
    return torch.cos(2 * PI2 * x + phase) + 0.25 * torch.cos(5 * PI2 * x - phase)


def _ch1d_dt(case):
    return 0.1 * PI2 / case["n"]


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case}
    if kind in ("step", "cook"):
        prec = chx.PREC_F64 if case["precision"] == "f64" else chx.PREC_F32_REFINE
        s["plan"] = chx.ChPlan(case["nx"], case["ny"], case["lx"], case["ly"], case["gamma"], case["dt"], prec)
        s["work"] = s["plan"].alloc_work()
        s["now"], s["prev"] = _step_inputs(case, seed)
        if kind == "cook":
            s["rho"] = torch.empty(2 * case["nx"] * case["ny"], dtype=torch.float64, device="cuda")
            s["seed"], s["step"] = int(seed), 0
    elif kind == "observables":
        s["plan"] = chx.ChPlan(case["nx"], case["ny"], case["lx"], case["ly"], case["gamma"], 1e-3)
        s["c"] = _fields(_gen(seed), case["ny"], case["nx"], case["lx"], case["ly"], case["gamma"], 0.0)[0]
        s["out"] = torch.empty(4, dtype=torch.float64, device="cuda")
    elif kind == "ensemble":
        s["ens"] = chx.Ensemble(case["dt"], chx.PREC_F32_REFINE)
        s["groups"] = []
        for n, side, slots in _ensemble_inputs(case, seed):
            gid = s["ens"].group_create(n, side, slots[0][0], len(slots))
            for k, (gamma, now, prev) in enumerate(slots):
                s["ens"].load(gid, k, now, prev, gamma)
            s["ens"].set_active(gid, len(slots))
            s["groups"].append((gid, torch.empty((2, len(slots), n, n), dtype=torch.float64, device="cuda")))
    elif kind in ("penta", "tri"):
        make = chx.PentaPlan if kind == "penta" else chx.TriPlan
        s["x"] = _rhs(case, seed)
        dtype = chx.F32 if case["dtype"] == "f32" else chx.F64
        if case["mode"] == "uniform":
            s["plan"] = make(case["n"], _uniform_row(case), case["batch"], mode=chx.COEF_UNIFORM, dtype=dtype)
        else:
            s["rows"] = [r.contiguous() for r in _band_rows(case, seed)]
            s["plan"] = make(case["n"], s["rows"], case["batch"], mode=chx.COEF_PER_SYSTEM, dtype=dtype)
    elif kind == "ch1d":
        s["plan"] = chx.Ch1DPlan(case["n"], case["batch"], PI2, case["gamma"], _ch1d_dt(case))
        s["c"] = _batched(case, seed)
    else:
        s["plan"] = chx.CN1DPlan(case["order"], case["n"], case["batch"], 1.0, 1.0, case["dt"], case["rewrite"])
        s["c"] = _batched(case, seed)
    torch.cuda.synchronize()
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "step":
        s["plan"].step(s["now"], s["prev"], s["work"], case["nsteps"])
        return s["now"], s["prev"]
    if kind == "cook":
        s["plan"].cook_run(s["now"], s["prev"], s["work"], s["rho"], case["nsteps"], case["sigma"], s["seed"],
                           step0=s["step"])
        s["step"] += case["nsteps"]
        return s["now"], s["prev"], s["rho"]
    if kind == "observables":
        return s["plan"].observables(s["c"], s["out"])
    if kind == "ensemble":
        s["ens"].step(case["nsteps"])
        for gid, out in s["groups"]:
            for k in range(out.shape[1]):
                s["ens"].read(gid, k, out[0, k], out[1, k])
        return [out for _, out in s["groups"]]
    if kind in ("penta", "tri"):
        if case["mode"] == "rewrite":
            s["plan"].refactor(s["rows"])
        if kind == "penta":
            return s["plan"].solve(s["x"], refine=case["dtype"] == "refine")
        return s["plan"].solve(s["x"])
    return s["plan"].step(s["c"], case["nsteps"])


def work(case):
    """Bytes: each input read once, each result written once.  Floating-point operations of the scheme per point
    (a multiply-add counts two): 26 + 2 x 17 + 1 for the 2D step, 9 / 5 multiply-adds for a prefactorised
    pentadiagonal / tridiagonal row, and what forming the factors or the right-hand side adds."""
    kind = case["kind"]
    if kind in ("step", "cook"):
        p = case["nx"] * case["ny"]
        return {"bytes": p * (32 if kind == "step" else 48), "flops": 61.0 * p * case["nsteps"]}
    if kind == "observables":
        p = case["nx"] * case["ny"]
        return {"bytes": 8 * p + 32, "flops": p * (16 + 2.5 * math.log2(p))}
    if kind == "ensemble":
        p = sum(cap * n * n for n, cap, _ in _groups(case))
        return {"bytes": 64 * p, "flops": 61.0 * p * case["nsteps"]}
    p = case["n"] * case["batch"]
    if kind in ("penta", "tri"):
        penta, rewrite = kind == "penta", case["mode"] == "rewrite"
        coef = 8 * (5 if penta else 3) if rewrite else 0
        return {"bytes": p * ((8 if case["dtype"] == "f32" else 16) + coef),
                "flops": p * ((18.0 if penta else 10.0) + ((40.0 if penta else 14.0) if rewrite else 0.0))}
    if kind == "ch1d":
        return {"bytes": 16 * p, "flops": 26.0 * p * case["nsteps"]}
    penta = case["order"] == 4
    return {"bytes": 16 * p, "flops": p * case["nsteps"] * ((20.0 if penta else 12.0) +
                                                             ((40.0 if penta else 14.0) if case["rewrite"] else 0.0))}


# -- the same in 64 bits, from the equations ------------------------------------------------------------------------

def _symbol(n, power):
    """Eigenvalues of the negative second difference (-delta^2), to a power, in Fourier order."""
    k = torch.arange(n, device="cuda", dtype=torch.float64)
    return (4.0 * torch.sin(math.pi * k / n) ** 2) ** power


def _circulant_solve(f, symbol, dim):
    h = symbol[: f.shape[dim] // 2 + 1]
    return torch.fft.irfft(torch.fft.rfft(f, dim=dim) / (h[:, None] if dim == 0 else h[None, :]), n=f.shape[dim],
                           dim=dim)


def _step_exact(now, prev, lx, ly, gamma, dt, nsteps):
    ny, nx = now.shape
    dx, dy = lx / nx, ly / ny

    def lap(u):
        return (torch.roll(u, 1, 1) + torch.roll(u, -1, 1) - 2 * u) / dx ** 2 + \
               (torch.roll(u, 1, 0) + torch.roll(u, -1, 0) - 2 * u) / dy ** 2

    ax, ay = 2 / 3 * gamma * dt / dx ** 4, 2 / 3 * gamma * dt / dy ** 4
    for _ in range(nsteps):
        bar = 2 * now - prev
        r = -2 / 3 * (now - prev) + 2 / 3 * dt * lap(now ** 3 - now - gamma * lap(bar))
        v = _circulant_solve(_circulant_solve(r, 1 + ax * _symbol(nx, 2), 1), 1 + ay * _symbol(ny, 2), 0)
        now, prev = bar + v, now
    return now, prev


def _observables_exact(c, lx, ly, gamma):
    ny, nx = c.shape
    dx, dy = lx / nx, ly / ny
    gx, gy = (torch.roll(c, -1, 1) - c) / dx, (torch.roll(c, -1, 0) - c) / dy
    energy = (0.25 * (c * c - 1) ** 2 + 0.5 * gamma * (gx * gx + gy * gy)).sum() * dx * dy

    def weights(n):  # Simpson's rule on the closed period for an even count, the trapezoid rule for an odd one
        w = torch.ones(n, device="cuda", dtype=torch.float64)
        if n % 2 == 0:
            w[0::2], w[1::2] = 2 / 3, 4 / 3
        return w

    mean = (weights(ny)[:, None] * weights(nx)[None, :] * c * c).sum() / (nx * ny)
    p = torch.fft.fft2(c).abs() ** 2
    k = torch.sqrt(torch.fft.fftfreq(ny, dy / PI2, device="cuda", dtype=torch.float64)[:, None] ** 2 +
                   torch.fft.fftfreq(nx, dx / PI2, device="cuda", dtype=torch.float64)[None, :] ** 2)
    p[0, 0], k[0, 0] = 0.0, 1.0
    return torch.stack([c.sum() * dx * dy, energy, 1 / (1 - mean), p.sum() / (p / k).sum()])


def _cyclic_band_solve(rows, f):
    """Cyclic band systems by elimination with the last w unknowns bordered (w = 2 or 1 neighbours to a side).
    rows: diagonals [n, batch] from the leftmost to the rightmost."""
    w = len(rows) // 2
    n, m = f.shape[0], f.shape[0] - w
    zero = torch.zeros_like(f[0])
    up, rhs = [], []  # row r solved for x_r: x_r = rhs[0] - sum up[j] x_{r+1+j} - sum_t rhs[1+t] x_{m+t}
    for r in range(m):
        band = [rows[w + o][r] if 0 <= r + o < m else zero for o in range(-w, w + 1)]
        cols = [f[r]] + [sum((rows[w + o][r] for o in range(-w, w + 1) if (r + o) % n == m + t), zero)
                         for t in range(w)]
        for o in range(-w, 0):
            if r + o < 0:
                continue
            q = band[w + o].clone()
            for j in range(w):
                band[w + o + 1 + j] = band[w + o + 1 + j] - q * up[r + o][j]
            cols = [c - q * p for c, p in zip(cols, rhs[r + o])]
        up.append([band[w + 1 + j] / band[w] for j in range(w)])
        rhs.append([c / band[w] for c in cols])
    z = [None] * m  # x_r = z[r][0] - sum_t z[r][1 + t] x_{m + t}
    for r in reversed(range(m)):
        z[r] = list(rhs[r])
        for j in range(w):
            if r + 1 + j < m:
                z[r] = [a - up[r][j] * b for a, b in zip(z[r], z[r + 1 + j])]
    mat = [[zero] * w for _ in range(w)]
    vec = [f[m + q] for q in range(w)]
    for q in range(w):
        for o in range(-w, w + 1):
            c, v = (m + q + o) % n, rows[w + o][m + q]
            if c >= m:
                mat[q][c - m] = mat[q][c - m] + v
            else:
                vec[q] = vec[q] - v * z[c][0]
                for t in range(w):
                    mat[q][t] = mat[q][t] - v * z[c][1 + t]
    if w == 1:
        tail = [vec[0] / mat[0][0]]
    else:
        det = mat[0][0] * mat[1][1] - mat[0][1] * mat[1][0]
        tail = [(vec[0] * mat[1][1] - mat[0][1] * vec[1]) / det, (mat[0][0] * vec[1] - vec[0] * mat[1][0]) / det]
    return torch.stack([z[r][0] - sum(z[r][1 + t] * tail[t] for t in range(w)) for r in range(m)] + tail)


def exact(case, seed):
    kind = case["kind"]
    if kind == "step":
        now, prev = _step_inputs(case, seed)
        return _step_exact(now, prev, case["lx"], case["ly"], case["gamma"], case["dt"], case["nsteps"])
    if kind == "cook":
        return None  # its deviates come from 32-bit functions
    if kind == "observables":
        c = _fields(_gen(seed), case["ny"], case["nx"], case["lx"], case["ly"], case["gamma"], 0.0)[0]
        return _observables_exact(c, case["lx"], case["ly"], case["gamma"])
    if kind == "ensemble":
        out = []
        for _, side, slots in _ensemble_inputs(case, seed):
            got = [_step_exact(now, prev, side, side, gamma, case["dt"], case["nsteps"]) for gamma, now, prev in slots]
            out.append(torch.stack([torch.stack([a for a, _ in got]), torch.stack([b for _, b in got])]))
        return out
    if kind in ("penta", "tri"):
        f = _rhs(case, seed).double()
        if case["mode"] == "uniform":
            return _circulant_solve(f, 1 + case["sigma"] * _symbol(case["n"], 2 if kind == "penta" else 1), 0)
        return _cyclic_band_solve(_band_rows(case, seed), f)
    c = _batched(case, seed)
    if kind == "ch1d":
        dx, dt = PI2 / case["n"], _ch1d_dt(case)
        for _ in range(case["nsteps"]):
            u = c ** 3 - c
            f = c + dt / dx ** 2 * (torch.roll(u, 1, 0) + torch.roll(u, -1, 0) - 2 * u)
            c = _circulant_solve(f, 1 + case["gamma"] * dt / dx ** 4 * _symbol(case["n"], 2), 0)
        return c
    sigma = 0.5 * case["dt"] * float(case["n"]) ** case["order"]
    symbol = 1 + sigma * _symbol(case["n"], case["order"] // 2)
    for _ in range(case["nsteps"]):
        c = _circulant_solve(c, symbol / (2 - symbol), 0)
    return c
