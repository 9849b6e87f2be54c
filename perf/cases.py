"""The calls of this framework whose time counts, with their inputs and what they have to return.

A case is one call a user's program makes in its time loop (or between two output times), on a
solver that the program keeps: time steps of the Coulomb and of the quadratic problem in both
precisions and with both integrators, the substeps on their own, and the diagnostics.  The grids
are those of the repository's workloads, its serving stream and its studies, down to the smallest
grid anybody steps and up to the largest whose solver leaves room on the card.

    listed()            the cases
    draw(rng)           one more of the same ranges
    prepare(case, seed) solver and Wigner function on the GPU
    run(state)          the call; returns what it computed
    work(case)          bytes and operations the call cannot do without
    exact(case, seed)   the same result by dense matrices and FFTs in 64 bits (no code of the
                        package), or None where that takes too long
"""
import math

import numpy as np
import torch

HBAR = M = 1.0

# Cells up to which exact() stays within some seconds, by potential.
EXACT_CELLS_COULOMB = 1.1e9
EXACT_CELLS = 1.3e9


def case(name, call, nx, nk, precision="fp32", half=8.0, lk=4.0, dt=0.02, centres=1, kappa=0.0,
         steps=1, patches=1, form="auto"):
    """call: "step" (Strang), "lpc1", "advect", "pflow", "theta", "tkm" or "diagnostics"; the box
    is [-half, half]^3 x [-lk, lk)^3; centres: nuclei of charge 1 (0: V = kappa/2 |x|^2);
    patches: along x1."""
    c = {"call": call, "nx1": nx[0], "nx2": nx[1], "nx3": nx[2], "nk": nk, "precision": precision,
         "half": half, "lk": lk, "dt": dt, "centres": centres, "kappa": kappa, "steps": steps,
         "patches": patches, "form": form}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # The electron-proton workload of the benchmark: the largest solver that fits thrice.
        case("electron_proton_48x32", "step", (48, 48, 48), 32, half=12.0),
        # The stationarity workload's grid, one step: an ordinary production step.
        case("hydrogen_32x32", "step", (32, 32, 32), 32, half=12.0, dt=0.025),
        # A chunk of five steps of a small request of the serving stream.
        case("serving_16x16", "step", (16, 16, 16), 16, dt=0.025, steps=5),
        # The smallest grid: a step while a program is being set up; latency only.
        case("smallest_8x8", "step", (8, 8, 8), 8, half=4.0),
        # The paper's own integrator on the two-centre problem, a serving-size grid.
        case("lpc1_two_centre_24x32", "lpc1", (24, 24, 24), 32, dt=0.01, centres=2),
        # Reference runs in double precision: the same step on the sizes of the parity studies.
        case("fp64_16x32", "step", (16, 16, 16), 32, "fp64"),
        case("fp64_24x16", "step", (24, 24, 24), 16, "fp64", dt=0.025),
        # The advection alone on a box with three different, odd line lengths.
        case("advect_ragged_41x27x33", "advect", (41, 27, 33), 32, half=10.0),
        # The Coulomb flow alone on a few x points, not a multiple of anything.
        case("pflow_7x5x6", "pflow", (7, 5, 6), 32, half=3.0, centres=2),
        # The oscillator study of Sec. 5.1: one long dimension in four patches, double precision.
        case("oscillator_patches_121x5x5", "step", (121, 5, 5), 32, "fp64", half=12.0, lk=3.2,
             dt=0.005, centres=0, kappa=0.3948, patches=4),
        # The modulated form of the Coulomb operator, for grids whose table would not fit.
        case("theta_modulated_16x32", "theta", (16, 16, 16), 32, form="modulated"),
        # What a run computes at every output time.
        case("diagnostics_32x32", "diagnostics", (32, 32, 32), 32, half=12.0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A case of the same ranges: any of the calls, grids from the smallest up to what costs less
    than the largest listed case, mostly with three different line lengths."""
    kind = rng.choice(["step", "step", "step", "lpc1", "advect", "pflow", "theta", "tkm",
                       "diagnostics", "quadratic", "fp64", "fp64"])
    call, precision, form = kind, "fp32", "auto"
    centres, kappa, patches, steps = rng.choice([1, 1, 2]), 0.0, 1, 1
    if kind == "quadratic":
        call, centres = rng.choice(["step", "step", "lpc1"]), 0
        kappa = 0.2 if call == "lpc1" else rng.choice([0.3948, 1.0])
        precision = rng.choice(["fp32", "fp64"])
    elif kind == "fp64":
        call, precision = rng.choice(["step", "step", "advect", "pflow", "theta", "diagnostics"]), "fp64"
    elif kind == "theta":
        form = rng.choice(["table", "modulated"])
    nk = rng.choice([8, 16, 32, 32])
    cells = 1.2e9 if precision == "fp32" else 1.0e8
    if form == "modulated":
        cells = 2.0e8
    top = max(5, int(round((cells / nk ** 3) ** (1.0 / 3.0))))
    top = min(top, 48)
    nx = [_log_int(rng, 4, top) for _ in range(3)]
    if rng.random() < 0.25:
        nx = [nx[0]] * 3
    if call == "advect" and rng.random() < 0.5:
        nx[0] = _log_int(rng, 4, 2 * top)
    if rng.random() < 0.2:
        patches = 2
        nx[0] = max(5, nx[0] | 1)
    if call == "step" and nx[0] * nx[1] * nx[2] * nk ** 3 < 3e7:
        steps = rng.choice([1, 1, 2, 5])
    half = rng.choice([4.0, 6.0] if call == "lpc1" else [4.0, 6.0, 8.0, 10.0])
    return case(None, call, nx, nk, precision, half=half,
                lk=rng.choice([3.2, 4.0]), dt=rng.choice([0.005, 0.01]), centres=centres,
                kappa=kappa, steps=steps, patches=patches, form=form)


# ---- inputs ----

def _grid(c):
    nx = (c["nx1"], c["nx2"], c["nx3"])
    xs = [np.linspace(-c["half"], c["half"], n) for n in nx]
    ks = (np.arange(c["nk"]) - c["nk"] // 2) * (2.0 * c["lk"] / c["nk"])
    return nx, xs, ks


def _centres(c):
    """The nuclei, away from every grid point of the boxes above."""
    if c["centres"] == 1:
        return [((0.13, -0.07, 0.11), 1.0)]
    return [((0.7, 0.013, -0.021), 1.0), ((-0.7, 0.013, -0.021), 1.0)][:c["centres"]]


def _inputs(c, seed):
    """A mixture of two unit-mass wavepackets with seeded centres, momenta and widths, as the
    workloads start from, on the GPU in the storage type."""
    rng = np.random.default_rng(seed)
    nx, xs, ks = _grid(c)
    dtype = torch.float32 if c["precision"] == "fp32" else torch.float64
    f = torch.empty(nx + (c["nk"],) * 3, dtype=dtype, device="cuda")
    parts = []
    for _ in range(2):
        x0, k0 = rng.uniform(-0.3, 0.3, 3) * c["half"], rng.uniform(-1.0, 1.0, 3)
        ax, ak = 0.5 * rng.uniform(0.8, 1.2), 2.0 * rng.uniform(0.8, 1.2)
        gx = [torch.as_tensor(np.exp(-ax * (xs[d] - x0[d]) ** 2), device="cuda") for d in range(3)]
        gk = [torch.as_tensor(np.exp(-ak * (ks - k0[d]) ** 2), device="cuda") for d in range(3)]
        kk = torch.einsum("i,j,k->ijk", *gk) * (0.5 * (ax * ak) ** 1.5 / math.pi ** 3)
        parts.append((gx, kk))
    for i in range(nx[0]):
        f[i] = sum((gx[0][i] * gx[1][:, None] * gx[2][None, :])[:, :, None, None, None] * kk
                   for gx, kk in parts).to(dtype)
    return f


def prepare(c, seed):
    import paper_2205_02380_gb300 as ch
    f = _inputs(c, seed)
    form = {"auto": ch.THETA_AUTO, "table": ch.THETA_TABLE, "modulated": ch.THETA_MODULATED}[c["form"]]
    solver = ch.Solver((c["nx1"], c["nx2"], c["nx3"]), c["nk"], -c["half"], c["half"], c["lk"],
                       nuclei=_centres(c), kappa=c["kappa"],
                       precision=ch.FP32_MIXED if c["precision"] == "fp32" else ch.FP64,
                       theta_form=form, integrator=ch.LPC1 if c["call"] == "lpc1" else ch.STRANG,
                       patches=(c["patches"], 1, 1))
    out = torch.empty_like(f) if c["call"] in ("theta", "tkm") else None
    return {"case": c, "f": f, "solver": solver, "out": out}


def run(state):
    c, s, f = state["case"], state["solver"], state["f"]
    call = c["call"]
    if call in ("step", "lpc1"):
        s.step(f, c["dt"], c["steps"])
        return f
    if call == "advect":
        s.advect(f, 0.5 * c["dt"])
        return f
    if call == "pflow":
        s.pflow(f, c["dt"])
        return f
    if call == "theta":
        s.theta(f, state["out"])
        return state["out"]
    if call == "tkm":
        s.tkm_convolve(f, state["out"])
        return state["out"]
    mass, energy = s.moments(f)
    return {"mass": mass, "energy": energy, "w1": s.reduced_wigner(f, 0), "w2": s.reduced_wigner(f, 1),
            "w3": s.reduced_wigner(f, 2), "p12": s.marginal_x12(f), "mean": np.array(s.expectations(f))}


# ---- what a pass cannot do without ----

def work(c):
    """Bytes: f read once and written once (the diagnostics only read it).  Operations: the
    padded convolutions by real-input FFTs (per application 7 N_k^2 complex transforms of length
    2 N_k, half of the padded ones' inputs being zero), a tridiagonal solve, its closure and a
    4-tap evaluation per line point and dimension, a length-N_k transform and its inverse per
    k-dimension for the quadratic potential."""
    cells = c["nx1"] * c["nx2"] * c["nx3"] * c["nk"] ** 3
    lg = math.log2(c["nk"])
    theta = 14 * 5 * lg + 57
    shift = 3 * 5 * lg + 9
    size = 4 if c["precision"] == "fp32" else 8
    advect = 3 * 20
    flops = {"step": 2 * advect + (4 * theta if c["centres"] else shift),
             "lpc1": 2 * advect + 2 * (theta if c["centres"] else shift) + 4,
             "advect": advect, "pflow": 4 * theta if c["centres"] else shift, "theta": theta,
             "tkm": theta, "diagnostics": 12}[c["call"]]
    return {"bytes": cells * size * (1 if c["call"] == "diagnostics" else 2),
            "flops": cells * flops * c["steps"]}


# ---- the same in 64 bits ----

def _weights(a):
    """Cubic B-spline values at the four nodes around a foot a (0 <= a < 1) left of a node."""
    b = 1.0 - a
    return [a ** 3 / 6, (-3 * a ** 3 + 3 * a ** 2 + 3 * a + 1) / 6,
            (-3 * b ** 3 + 3 * b ** 2 + 3 * b + 1) / 6, b ** 3 / 6]


def _closed_spline(m, h):
    """Inverse of the spline system of m + 1 nodes with given end slopes: rows eta_-1..eta_m+1,
    columns slope left, node values, slope right."""
    a = np.zeros((m + 3, m + 3))
    a[0, 0], a[0, 2], a[-1, -3], a[-1, -1] = -0.5 / h, 0.5 / h, -0.5 / h, 0.5 / h
    for i in range(m + 1):
        a[i + 1, i:i + 3] = [1 / 6, 2 / 3, 1 / 6]
    return np.linalg.inv(a)


def _advect_matrices(n, h, alphas, patches, n_nb=20):
    """For each shift alpha (in units of h) the n x n matrix that takes the node values of a line
    to the values of its spline at x_j - alpha h."""
    top = n - 1
    a = np.zeros((n + 2, n + 2))
    a[0, :3] = a[-1, -3:] = np.array([1.0, -2.0, 1.0]) / h ** 2
    for i in range(n):
        a[i + 1, i:i + 3] = [1 / 6, 2 / 3, 1 / 6]
    inv = np.linalg.inv(a)
    m = top // patches
    slope = np.zeros((patches + 1, n))      # end slopes of the patches from the node values
    for b in range(patches + 1):
        for j in range(n):
            if abs(j - b * m) <= n_nb:
                slope[b, j] = (inv[b * m + 2, j + 1] - inv[b * m, j + 1]) / (2 * h)
    solve = _closed_spline(m, h)
    etas = []
    for q in range(patches):
        rhs = np.zeros((m + 3, n))
        rhs[0], rhs[-1] = slope[q], slope[q + 1]
        rhs[1:-1, q * m:(q + 1) * m + 1] = np.eye(m + 1)
        etas.append(solve @ rhs)
    out = np.zeros((len(alphas), n, n))
    for i, al in enumerate(alphas):
        shift = math.floor(al)
        w = _weights(al - shift)
        for j in range(n):
            # the patch whose interval holds the foot (the left one at a node shared by two)
            q = min(max((j - shift - 1) // m, 0), patches - 1)
            first = j - shift - 2 - q * m
            for t in range(4):
                if -1 <= first + t <= m + 1:
                    out[i, j] += w[t] * etas[q][first + t + 1]
    return out


def _advect64(f, c, tau):
    nx, xs, ks = _grid(c)
    for d in range(3):
        h = 2.0 * c["half"] / (nx[d] - 1)
        mats = _advect_matrices(nx[d], h, HBAR * ks * tau / (M * h), c["patches"] if d == 0 else 1)
        mats = torch.as_tensor(mats, device=f.device)
        for q in range(c["nk"]):
            part = f.select(3 + d, q)
            moved = part.movedim(d, 0)
            got = (mats[q] @ moved.reshape(nx[d], -1)).reshape(moved.shape)
            part.copy_(got.movedim(0, d))
    return f


def _sine_integral(x):
    """Si of sorted values, by 16-point Gauss-Legendre between neighbours."""
    nodes, wts = np.polynomial.legendre.leggauss(16)
    lo = np.concatenate([[0.0], x[:-1]])
    total, parts = np.zeros_like(x), 1 + int(np.max(x - lo) / 1.5)
    step = (x - lo) / parts
    for p in range(parts):
        mid, r = lo + (p + 0.5) * step, 0.5 * step
        t = mid[:, None] + r[:, None] * nodes
        total += r * (np.sinc(t / math.pi) @ wts)
    return np.cumsum(total)


def _kernel_taps(nk, lk):
    """T of the truncated kernel method on (-N, N)^3, laid out circularly on (2N)^3."""
    m = 3 * nk
    n = np.arange(m)
    n = np.where(n < m // 2, n, n - m)
    sq = n[:, None, None] ** 2 + n[None, :, None] ** 2 + n[None, None, :] ** 2
    vals, at = np.unique(sq, return_inverse=True)
    xi, diam = 2.0 * math.pi * np.sqrt(vals) / (6.0 * lk), 2.0 * math.sqrt(3.0) * lk
    u = np.full(len(vals), 4.0 * math.pi * diam)
    u[1:] = 4.0 * math.pi * _sine_integral(xi[1:] * diam) / xi[1:]
    full = np.fft.ifftn(u[at.reshape(sq.shape)]).real
    p = np.concatenate([np.arange(nk), [0], np.arange(-nk + 1, 0)])
    t = full[np.ix_(p % m, p % m, p % m)]
    t[nk], t[:, nk], t[:, :, nk] = 0.0, 0.0, 0.0
    return torch.as_tensor(t, device="cuda"), torch.as_tensor(p, device="cuda", dtype=torch.float64)


def _coulomb64(f, c, outer, plain=False):
    """outer(f, theta) for every chunk of x points, theta(u) the truncated-kernel operator there
    (plain: the convolution with T itself)."""
    nx, xs, ks = _grid(c)
    nk, dk = c["nk"], 2.0 * c["lk"] / c["nk"]
    taps, p = _kernel_taps(nk, c["lk"])
    x = torch.cartesian_prod(*[torch.as_tensor(v, device="cuda") for v in xs])
    flat = f.reshape(-1, nk, nk, nk)
    step = max(1, 2 ** 26 // (2 * nk) ** 3)
    size = (2 * nk,) * 3
    for a in range(0, flat.shape[0], step):
        part = flat[a:a + step]
        if plain:
            spec = torch.fft.rfftn(taps)
        else:
            kern = 0.0
            for pos, charge in _centres(c):
                ph = [2.0 * dk * (x[a:a + step, d] - pos[d])[:, None] * p for d in range(3)]
                ang = ph[0][:, :, None, None] + ph[1][:, None, :, None] + ph[2][:, None, None, :]
                kern = kern - 2.0 * charge / (math.pi ** 2 * HBAR) * taps * torch.sin(ang)
            spec = torch.fft.rfftn(kern, dim=(1, 2, 3))

        def theta(u):
            v = torch.fft.irfftn(torch.fft.rfftn(u, s=size, dim=(1, 2, 3)) * spec, s=size, dim=(1, 2, 3))
            return v[:, :nk, :nk, :nk]
        part.copy_(outer(part, theta))
    return f


def _taylor(dt):
    def flow(f, theta):
        u = f
        for s in (4, 3, 2, 1):
            u = f + (dt / s) * theta(u)
        return u
    return flow


def _quadratic64(f, c, factor, add):
    """Along every k-dimension the multiplication of the spectrum by factor(xi, rate) with
    rate = kappa x_d / hbar; in turn, or (add) summed."""
    nx, xs, ks = _grid(c)
    nk = c["nk"]
    xi = math.pi * np.fft.fftfreq(nk, 1.0 / nk) / c["lk"]
    total = torch.zeros_like(f) if add else f
    for d in range(3):
        fac = torch.as_tensor(factor(xi[None, :], c["kappa"] * xs[d][:, None] / HBAR), device=f.device)
        shape = [1] * 6
        shape[d], shape[3 + d] = nx[d], nk
        fac = fac.reshape(shape)
        for i in range(nx[0]):
            part = fac[i:i + 1] if d == 0 else fac
            got = torch.fft.ifft(torch.fft.fft(f[i:i + 1], dim=3 + d) * part, dim=3 + d).real
            if add:
                total[i:i + 1] += got
            else:
                f[i:i + 1] = got
    return total


def _pflow64(f, c, dt):
    if c["centres"]:
        return _coulomb64(f, c, _taylor(dt))

    def shift(xi, rate):
        fac = np.exp(1j * xi * rate * dt)
        nyq = xi.shape[1] // 2
        fac[:, nyq] = np.cos(xi[:, nyq] * rate[:, 0] * dt)
        return fac
    return _quadratic64(f, c, shift, False)


def _theta64(f, c):
    if c["centres"]:
        return _coulomb64(f, c, lambda u, theta: theta(u))

    def deriv(xi, rate):
        fac = 1j * xi * rate
        fac[:, xi.shape[1] // 2] = 0.0
        return fac
    return _quadratic64(f, c, deriv, True)


def _diagnostics64(f, c):
    nx, xs, ks = _grid(c)
    h = [2.0 * c["half"] / (n - 1) for n in nx]
    dk = 2.0 * c["lk"] / c["nk"]
    marg = {}
    vol = h[0] * h[1] * h[2] * dk ** 3
    byx, sums = f.sum((3, 4, 5)), []
    for d in range(3):
        others = [e for e in range(3) if e != d]
        s = f.sum(others + [3 + e for e in others])
        sums.append(s)
        marg["w%d" % (d + 1)] = (s * h[others[0]] * h[others[1]] * dk ** 2).cpu().numpy()
    total = byx.sum()
    x = [torch.as_tensor(v, device=f.device) for v in xs]
    k = torch.as_tensor(ks, device=f.device)
    pot = 0.0
    for pos, charge in _centres(c):
        pot = pot - charge / torch.sqrt(sum(((x[d] - pos[d]) ** 2).reshape([-1 if e == d else 1 for e in range(3)])
                                            for d in range(3)))
    if not c["centres"]:
        pot = 0.5 * c["kappa"] * sum((x[d] ** 2).reshape([-1 if e == d else 1 for e in range(3)]) for d in range(3))
    kin = sum((sums[d].sum(0) * k ** 2).sum() for d in range(3)) * HBAR ** 2 / (2 * M)
    mean = [(byx.sum([e for e in range(3) if e != d]) * x[d]).sum() / total for d in range(3)]
    mean += [(sums[d].sum(0) * k).sum() / total for d in range(3)]
    return {"mass": float(total * vol), "energy": float((kin + (byx * pot).sum()) * vol), **marg,
            "p12": (byx.sum(2) * h[2] * dk ** 3).cpu().numpy(), "mean": np.array([float(v) for v in mean])}


def exact(c, seed):
    cells = c["nx1"] * c["nx2"] * c["nx3"] * c["nk"] ** 3
    coulomb = c["centres"] > 0 and c["call"] not in ("advect", "diagnostics")
    if cells * c["steps"] > (EXACT_CELLS_COULOMB if coulomb else EXACT_CELLS):
        return None
    f, dt, call = _inputs(c, seed).double(), c["dt"], c["call"]
    if call == "diagnostics":
        return _diagnostics64(f, c)
    if call == "advect":
        return _advect64(f, c, 0.5 * dt)
    if call == "pflow":
        return _pflow64(f, c, dt)
    if call == "theta":
        return _theta64(f, c)
    if call == "tkm":
        return _coulomb64(f, c, lambda u, conv: conv(u), plain=True)
    for _ in range(c["steps"]):
        if call == "step":
            f = _advect64(_pflow64(_advect64(f, c, 0.5 * dt), c, dt), c, 0.5 * dt)
        else:
            h = _advect64(_theta64(f.clone(), c), c, dt)
            f = _advect64(f, c, dt)
            pred = _theta64(f + dt * h, c)
            f = f + 0.5 * dt * pred + 0.5 * dt * h
    return f
