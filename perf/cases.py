"""Performance cases: the calls a user of this framework makes, over the range of sizes it is used at.

A pass of a `step` case is one radiative-transfer step as a hydrodynamical code drives it: new fields and
sources in device memory, one `Solver.step`, the rate and heating grids back in device memory. A `batch`
case is one run of a captured `Batch` over solves that already hold their fields and sources. A `serve`
case is a burst of requests to a `Server`, all polled, with host arrays in and out.

Inputs are made on the device from the seed: lognormal gas with P(k) ~ k^-2, power-law sources in the
densest 1% of cells, the cell size of a 20 Mpc/h box of 128^3 cells. `exact` traces the same inputs with
plain torch in 64 bits: every ray as one element of a vector, cell by cell.
"""
import math

import numpy as np
import torch

import paper_2512_12466_gb300 as nyx

MPC_CM = 3.0857e24
HUBBLE_H = 0.67742
MYR_S = 3.15576e13
DX_CM = 20.0 / HUBBLE_H * MPC_CM / 128          # cell size of the cosmological boxes
SIGMA = 6.3e-18
EV_ERG = 1.602176634e-12
TAU_MAX = 30.0
N_MIN = 4.0
T_BB = 1e5
COUNTS = ("rays", "splits", "escaped", "dropped_tau", "dropped_level", "segments", "secondary")
PHOTONS = ("emitted_ph", "absorbed_ph", "escaped_ph", "deposited_ph")


def step(name, n, sources, x, precision, **options):
    case = dict(name=name, kind="step", n=n, sources=sources, x=x, precision=precision, sigma_ln=1.0, overlap=3,
                periodic=False, blackbody=False, merge=False, chem=False)
    case.update(options)
    return case


def listed():
    return [
        # a test-sized box: what a unit test or an interactive session steps; launches and round trips count
        step("small_16_fp64", 16, 1, "thin", "fp64"),
        # a small coupled run with periodic boundaries: rays wrap and travel sqrt(3) box lengths
        step("periodic_40_fp32", 40, 6, "thin", "fp32", periodic=True),
        # the Stromgren test: one source, uniform neutral gas, the rate iterated with the ionization update
        step("stromgren_64_fp64", 64, 1, "uniform", "fp64", chem=True),
        # the 128^3 / 1024-source cosmological box before reionization: every ray dies near its source
        step("neutral_128_fp32", 128, 1024, "neutral", "fp32"),
        # the same box after reionization (optically thin), the main throughput workload, FP32 physics
        step("thin_128_fp32", 128, 1024, "thin", "fp32"),
        # its FP64 form, with a quarter of the sources
        step("thin_128_fp64", 128, 256, "thin", "fp64"),
        # the rate integrated over a blackbody spectrum, an odd grid size
        step("blackbody_81_fp32", 81, 64, "thin", "fp32", blackbody=True),
        # half-ionized gas on a ragged grid, FP64, the unthresholded overlap correction
        step("patchy_165_fp64", 165, 2048, "patchy", "fp64", overlap=2),
        # the largest catalog: 256^3, 32768 sources, bubble merging on
        step("merge_256_fp32", 256, 32768, "patchy", "fp32", sigma_ln=1.5, merge=True),
        # a box whose fields exceed the L2 cache
        step("thin_256_fp32", 256, 48, "thin", "fp32", sigma_ln=1.5),
        # many independent uneven solves traced together (parameter studies, subvolumes)
        dict(name="batch_48_fp32", kind="batch", solves=48, n_lo=32, n_hi=128, max_sources=2048, x="neutral",
             precision="fp32"),
        # a burst of requests to the server, host buffers in and out
        dict(name="serve_12_fp32", kind="serve", solves=12, n_lo=48, n_hi=112, max_sources=4096, x="patchy",
             precision="fp32"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("step", "step", "step", "step", "chem", "merge", "batch", "serve"))
    precision = rng.choice(("fp32", "fp32", "fp64"))
    if kind == "chem":
        return _unnamed(step("", _log_int(rng, 24, 96), 1, "uniform", precision, chem=True))
    if kind == "merge":
        return _unnamed(step("", _log_int(rng, 96, 240), _log_int(rng, 1024, 32768), "patchy", precision, sigma_ln=1.5,
                             merge=rng.random() < 0.7))
    if kind in ("batch", "serve"):
        return dict(kind=kind, solves=rng.randint(4, 12) if kind == "serve" else rng.randint(8, 48), n_lo=32,
                    n_hi=rng.randint(48, 112), max_sources=_log_int(rng, 64, 2048),
                    x="patchy" if kind == "serve" else "neutral", precision=precision)
    periodic = rng.random() < 0.25
    n = _log_int(rng, 12, 56) if periodic else _log_int(rng, 12, 176)
    x = rng.choice(("thin", "thin", "patchy", "neutral"))
    case = step("", n, 1, x, precision, overlap=rng.choice((3, 3, 3, 2, 0)), periodic=periodic,
                blackbody=rng.random() < 0.2)
    most = 2048
    while most > 1 and _segments(dict(case, sources=most)) > 4e9:
        most //= 2
    return _unnamed(dict(case, sources=_log_int(rng, 1, most)))


def _unnamed(case):
    return {k: v for k, v in case.items() if k != "name"}


# ---------------------------------------------------------------- inputs

def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _generator(seed):
    return torch.Generator(device=_device()).manual_seed(seed)


def _lognormal(n, mean, sigma_ln, gen):
    """mean * exp(s g) / <exp(s g)>, g a unit-variance Gaussian field with P(k) ~ k^-2; index order [iz, iy, ix]."""
    dev = _device()
    f = torch.fft.rfftn(torch.randn((n, n, n), dtype=torch.float64, device=dev, generator=gen))
    k = torch.fft.fftfreq(n, dtype=torch.float64, device=dev)
    kx = torch.fft.rfftfreq(n, dtype=torch.float64, device=dev)
    kk = torch.sqrt(k[:, None, None] ** 2 + k[None, :, None] ** 2 + kx[None, None, :] ** 2)
    kk[0, 0, 0] = math.inf
    g = torch.fft.irfftn(f / kk, s=(n, n, n))
    g = (g - g.mean()) / g.std()
    v = torch.exp(sigma_ln * g)
    return (mean * v / v.mean()).reshape(-1)


def _inputs(case, seed):
    """(n_H, x, cells, ndot, box_cm) of one solve, device tensors."""
    n, m, dev, gen = case["n"], case["sources"], _device(), _generator(seed)
    if case["x"] == "uniform":                      # the Stromgren test A, density and rate varied with the seed
        u = torch.rand(2, dtype=torch.float64, device=dev, generator=gen).tolist()
        n_h = torch.full((n ** 3,), 1e-3 * (0.9 + 0.2 * u[0]), dtype=torch.float64, device=dev)
        cells = torch.full((1, 3), n // 2, dtype=torch.int32, device=dev)
        ndot = torch.full((1,), 5e48 * (0.9 + 0.2 * u[1]), dtype=torch.float64, device=dev)
        return n_h, torch.zeros_like(n_h), cells, ndot, 0.0066 * MPC_CM
    n_h = _lognormal(n, 2e-4, case.get("sigma_ln", 1.0), gen)
    if case["x"] == "patchy":
        x = _lognormal(n, 1.0, 1.5, gen).clamp(0.0, 1.0)
    else:
        x = torch.full_like(n_h, 0.0 if case["x"] == "neutral" else 1.0 - 1e-4)
    top = torch.topk(n_h, max(1, round(0.01 * n ** 3)), sorted=False).indices.sort().values
    pick = top[torch.randint(0, len(top), (m,), device=dev, generator=gen)]
    cells = torch.stack([pick % n, pick // n % n, pick // (n * n)], dim=1).to(torch.int32).contiguous()
    u = torch.rand(m, dtype=torch.float64, device=dev, generator=gen)
    ndot = 1.0 / (1e-50 - u * (1e-50 - 1e-53))
    return n_h, x, cells, ndot, DX_CM * n


def _members(case, seed):
    """The solves of a batch or burst: uneven sizes and log-uniform source counts (the case's own), fields and
    sources by the seed."""
    rng = np.random.default_rng([case["solves"], case["n_hi"], case["max_sources"]])
    out = []
    for j in range(case["solves"]):
        n = int(rng.integers(case["n_lo"], case["n_hi"] + 1))
        m = int(np.clip(np.exp(rng.random() * np.log(case["max_sources"] + 1)), 1, case["max_sources"]))
        out.append((dict(n=n, sources=m, x=case["x"]), seed * 1000 + j))
    return out


def _dt(case):
    return 0.1 * MYR_S if case["chem"] else 0.0


def _options(case):
    o = dict(precision=nyx.RT_FP32 if case["precision"] == "fp32" else nyx.RT_FP64, n_min_ray=N_MIN, tau_max=TAU_MAX)
    if case["kind"] != "step":
        return o
    o.update(overlap_mode=case["overlap"], periodic=int(case["periodic"]))
    if case["blackbody"]:
        o.update(spectrum=nyx.RT_SPECTRUM_BLACKBODY, t_bb_K=T_BB)
    if case["merge"]:
        o.update(merge_mode=nyx.RT_MERGE_FORCED, merge_f_req=0.5)
    if case["chem"]:
        o.update(chem_iterate=1, alpha_B=2.59e-13, clumping=1.0, C_H=0.0)
    return o


# ---------------------------------------------------------------- prepare / run

def prepare(case, seed):
    if case["kind"] == "step":
        n_h, x, cells, ndot, box = _inputs(case, seed)
        solver = nyx.Solver(case["n"], box, **_options(case))
        return dict(case=case, solver=solver, n_h=n_h, x=x, cells=cells, ndot=ndot,
                    gamma=torch.empty_like(n_h), heat=torch.empty_like(n_h), x_out=torch.empty_like(n_h))
    if case["kind"] == "batch":
        solvers = []
        for c, s in _members(case, seed):
            n_h, x, cells, ndot, box = _inputs(c, s)
            solver = nyx.Solver(c["n"], box, **_options(case))
            solver.set_fields(n_h, x)
            solver.add_sources(cells, ndot)
            solvers.append(solver)
        gammas = [torch.empty(s.n ** 3, dtype=torch.float64, device="cuda") for s in solvers]
        batch = nyx.Batch(solvers)
        batch.run(gammas, None)                     # the first run measures the solves' work, the capture uses it
        batch.capture()
        return dict(case=case, solvers=solvers, batch=batch, gammas=gammas)
    requests = []
    for c, s in _members(case, seed):
        n_h, x, cells, ndot, box = _inputs(c, s)
        pinned = [t.cpu().pin_memory().numpy() for t in (n_h, x, cells.reshape(-1), ndot)]
        gamma = torch.empty(c["n"] ** 3, dtype=torch.float64, pin_memory=True).numpy()
        requests.append((c["n"], box, pinned, gamma))
    return dict(case=case, requests=requests, server=nyx.Server(precision=_options(case)["precision"]))


def run(state):
    case = state["case"]
    if case["kind"] == "step":
        s = state["solver"]
        s.set_fields(state["n_h"], state["x"])
        s.clear_sources()
        s.add_sources(state["cells"], state["ndot"])
        gamma, heat, stats = s.step(_dt(case), state["gamma"], state["heat"])
        out = dict(gamma=gamma, heat=heat)
        if case["chem"]:
            out["x"] = s.get_x(state["x_out"])
        else:
            out["counts"] = np.array([stats[k] for k in COUNTS])
            out["photons"] = np.array([stats[k] for k in PHOTONS])
        return out
    if case["kind"] == "batch":
        stats = state["batch"].run(state["gammas"], None)
        return dict(gamma=state["gammas"], segments=np.array([st["segments"] for st in stats]))
    server = state["server"]
    ids = [server.submit(n, box, n_h, x, cells, ndot, gamma=gamma, n_min_ray=N_MIN, tau_max=TAU_MAX)
           for n, box, (n_h, x, cells, ndot), gamma in state["requests"]]
    done = [server.poll(i, wait_s=60.0) for i in ids]
    return dict(gamma=[g for g, _, _, _ in done], segments=np.array([st["segments"] for _, _, st, _ in done]))


# ---------------------------------------------------------------- work

def _segments(case):
    """Ray-cell segments of a step, from counts of such boxes: 12.6 per cell and source where rays cross the whole
    box, over the sphere of sqrt(3) box lengths with periodic boundaries, about 270 per source in half-ionized gas,
    12 in neutral gas."""
    per_source = {"thin": 12.6 * case["n"] ** 3, "uniform": 2.2e5, "patchy": 270.0, "neutral": 12.0}[case["x"]]
    if case.get("periodic") and case["x"] == "thin":
        per_source *= 4 / 3 * math.pi * 3 ** 1.5
    return per_source * case["sources"]


def work(case):
    """Bytes: both fields and the sources read, the grids asked for written. Operations: about 30 a segment (optical
    depth, 1 - e^-tau, rate, overlap share, two budgets); the chemistry's iterations are not known beforehand and
    count once."""
    if case["kind"] == "step":
        cells = case["n"] ** 3
        return dict(bytes=(16 + 16 + 8 * case["chem"]) * cells + 20 * case["sources"], flops=30 * _segments(case) + 5 * cells)
    solves = [c for c, _ in _members(case, 0)]
    return dict(bytes=sum(24 * c["n"] ** 3 + 20 * c["sources"] for c in solves),
                flops=sum(30 * _segments(c) + 5 * c["n"] ** 3 for c in solves))


# ---------------------------------------------------------------- the same in 64 bits, with plain torch

def exact(case, seed):
    if case["kind"] != "step":
        gammas = [_exact_step(dict(step("", c["n"], c["sources"], c["x"], case["precision"]), **c), s)["gamma"]
                  for c, s in _members(case, seed)]
        return dict(gamma=gammas, segments=None)
    if _segments(case) * (6 if case["blackbody"] else 1) > 8e9:
        return None
    return _exact_step(case, seed)


def _exact_step(case, seed):
    n_h, x, cells, ndot, box = _inputs(case, seed)
    n = case["n"]
    dx = box / n
    cells, ndot = _dedup(cells.long(), ndot, n)
    if case["merge"]:
        cells, ndot = _merge_bubbles(cells, ndot, x, n, case["periodic"])
    xa, photons = x, None
    for _ in range(100):
        gamma, photons = _trace(case, n_h, xa, cells, ndot, dx)
        traced = xa
        if not case["chem"]:
            break
        ion = gamma
        tot = ion + traced * n_h * 2.59e-13
        u = _dt(case) * tot
        xeq = torch.where(tot > 0, ion / tot, x)
        x_end = xeq + (x - xeq) * torch.exp(-u)
        xa = torch.where(tot > 0, xeq + (x - xeq) * (-torch.expm1(-u) / u), x)
        if float((xa - traced).abs().max()) < 1e-6:
            break
    n_hi = (1.0 - traced) * n_h
    out = dict(gamma=gamma, heat=EV_ERG * gamma * n_hi)
    if case["chem"]:
        out["x"] = x_end
    else:
        out["counts"] = None
        out["photons"] = torch.tensor([float(ndot.sum()), photons[0], photons[1],
                                       float((gamma * n_hi).sum()) * dx ** 3], dtype=torch.float64)
    return out


def _dedup(cells, ndot, n):
    key = (cells[:, 0] * n + cells[:, 1]) * n + cells[:, 2]
    uniq, inv = torch.unique(key, sorted=True, return_inverse=True)
    rate = torch.zeros(len(uniq), dtype=torch.float64, device=key.device).index_add_(0, inv, ndot)
    return torch.stack([uniq // (n * n), uniq // n % n, uniq % n], dim=1), rate


def _directions(level, pix):
    """Quantised HEALPix nested pixel centres: |d_a| and sign of each component, in units of 2^-21."""
    ns = 1 << level
    face, m = pix // (ns * ns), pix % (ns * ns)
    fx, fy = torch.zeros_like(m), torch.zeros_like(m)
    for b in range(level):
        fx |= (m >> (2 * b) & 1) << b
        fy |= (m >> (2 * b + 1) & 1) << b
    row = face // 4
    ring = (row + 2) * ns - fx - fy - 1
    in_row = 2 * (face % 4) + (row != 1)
    north, south = ring < ns, ring > 3 * ns
    nr = torch.where(north, ring, torch.where(south, 4 * ns - ring, torch.full_like(ring, ns)))
    cap = (nr * nr).double() / float(3 * ns * ns)
    belt = (2 * ns - ring).double() * 2.0 / float(3 * ns)
    z = torch.where(north, 1.0 - cap, torch.where(south, cap - 1.0, belt))
    st = torch.sqrt(torch.where(north | south, cap * (2.0 - cap), (1.0 - belt) * (1.0 + belt)))
    shift = torch.where(north | south, torch.zeros_like(ring), (ring - ns) & 1)
    j = torch.div(in_row * nr + fx - fy + 1 + shift, 2, rounding_mode="trunc")
    j = torch.where(j > 4 * ns, j - 4 * ns, torch.where(j < 1, j + 4 * ns, j))
    phi = (j.double() - 0.5 * (shift + 1).double()) * (math.pi / 2) / nr.double()
    v = torch.stack([st * torch.cos(phi), st * torch.sin(phi), z])
    return torch.floor(v.abs() * 2.0 ** 21 + 0.5).long(), torch.where(v < 0, -1, 1)


def _merge_bubbles(cells, ndot, x, n, periodic):
    """Bubble radii by shell sampling, groups of overlapping bubbles, one source per group at the member nearest the
    flux-weighted centroid (x_th 0.9, f_req 0.5, shells every 2 cells to 16, at least 8 samples or all ionized)."""
    dev, m = cells.device, len(cells)
    at = lambda c: (c[..., 2] * n + c[..., 1]) * n + c[..., 0]
    mag, sgn = _directions(3, torch.arange(768, device=dev))
    d = (mag * sgn).double().T * 2.0 ** -21
    radius = torch.where(x[at(cells)] >= 0.9, 16.0, 0.0).double()
    todo = torch.nonzero(radius > 0).reshape(-1)
    for r in (2.0, 4.0, 6.0, 8.0, 10.0, 12.0, 14.0, 16.0):
        if not len(todo):
            break
        q = torch.floor(cells[todo][:, None, :].double() + 0.5 + r * d[None]).long()
        q = q % n if periodic else q
        ok = ((q >= 0) & (q < n)).all(-1)
        key = torch.where(ok, at(q), n ** 3).sort(dim=1).values
        first = torch.ones_like(key, dtype=torch.bool)
        first[:, 1:] = key[:, 1:] != key[:, :-1]
        first &= key < n ** 3
        ion = first & (x[key.clamp(max=n ** 3 - 1)] >= 0.9)
        tot, good = first.sum(1), ion.sum(1)
        fail = torch.where(tot < 8, good < tot, good.double() / tot.clamp(min=1).double() < 0.5)
        radius[todo[fail]] = r - 2.0
        todo = todo[~fail]
    image = (lambda v: (v + n // 2) % n - n // 2) if periodic else (lambda v: v)
    pos = torch.nonzero(radius > 0).reshape(-1)
    label = torch.arange(m, device=dev)
    if len(pos):
        c, rr = cells[pos], radius[pos]
        d2 = (image(c[:, None, :] - c[None]) ** 2).sum(-1)
        near = d2.double() <= (rr[:, None] + rr[None]) ** 2 + 1e-6
        low = torch.arange(len(pos), device=dev)
        while True:                                 # each member takes the smallest label in reach, until nothing changes
            new = torch.where(near, low[None], len(pos)).amin(1)
            new = new[new]
            if torch.equal(new, low):
                break
            low = new
        label[pos] = pos[low]
    root, inv = torch.unique(label, sorted=True, return_inverse=True)
    total = lambda v: torch.zeros(len(root), dtype=torch.float64, device=dev).index_add_(0, inv, v)
    flux = total(ndot)
    unwrapped = cells[root][inv] + image(cells - cells[root][inv])
    centre = torch.stack([total(ndot * unwrapped[:, a].double()) for a in range(3)], 1) / flux[:, None]
    centre = torch.floor(centre + 0.5).long()
    centre = centre % n if periodic else centre.clamp(0, n - 1)
    d2 = (image(cells - centre[inv]) ** 2).sum(1)
    best = torch.full((len(root),), 1 << 62, dtype=torch.int64, device=dev)
    best.scatter_reduce_(0, inv, d2 * m + torch.arange(m, device=dev), "amin")
    return cells[best % m], flux


def _spectrum():
    """Nodes s = sigma_nu / sigma_0 and weights of the blackbody's photon numbers above the threshold."""
    theta = 13.598 * EV_ERG / (1.380649e-16 * T_BB)
    u, w = np.polynomial.legendre.leggauss(48)
    u, w = 0.5 * (u + 1.0), 0.5 * w
    w = w * np.exp(-theta / u) / -np.expm1(-theta / u) / u ** 4
    return list(zip((u ** 3).tolist(), (w / w.sum()).tolist()))


CHUNK = 1 << 23                                     # rays traced together


def _trace(case, n_h, x, cells, ndot, dx):
    """Gamma, and the photons absorbed and escaped: rays of a level walk from its start sphere to its split sphere."""
    n, dev = case["n"], n_h.device
    mode, periodic = case["overlap"], case["periodic"]
    nodes = _spectrum() if case["blackbody"] else None
    n_hi = (1.0 - x) * n_h
    kappa = SIGMA * dx * n_hi
    takes = (n_hi > 0) & ((n_h >= 0.01 * float(n_h.mean())) if mode == 3 else torch.ones_like(n_h, dtype=torch.bool))
    rate = ndot / 12.0 * SIGMA / dx ** 2
    gamma = torch.zeros_like(n_h)
    rq = math.floor(math.sqrt(3.0 / (math.pi * N_MIN)) * 2.0 ** 24 + 0.5)
    rs = math.floor(math.sqrt(3.0) * n * 2.0 ** 24 + 0.5)
    absorbed, escaped = 0.0, 0.0
    m = len(ndot)
    src = torch.arange(m, device=dev).repeat_interleave(12)
    one = torch.ones(12 * m, dtype=torch.float64, device=dev)
    stack = [(0, src, torch.arange(12, device=dev).repeat(m), one, torch.zeros_like(one))]
    while stack:
        level, src, pix, P, tau = stack.pop()
        if len(src) > CHUNK:
            stack.append((level, src[CHUNK:], pix[CHUNK:], P[CHUNK:], tau[CHUNK:]))
            src, pix, P, tau = src[:CHUNK], pix[:CHUNK], P[:CHUNK], tau[:CHUNK]
        mag, sgn = _directions(level, pix)
        norm = torch.sqrt((mag * mag).sum(0).double()) * 2.0 ** -21
        split = not periodic or (rq << level) < rs
        q0, q1 = rq << (level - 1) if level else 0, rq << level if split else rs
        k = (q0 * mag + (1 << 44)) >> 45            # crossings done at the start sphere
        t0, t_end = q0 * 2.0 ** -24, q1 * 2.0 ** -24
        i = cells[src].T + sgn * k
        inside = ((i >= 0) & (i < n)).all(0) if not periodic else torch.ones_like(src, dtype=torch.bool)
        i = i % n if periodic else i
        left = lambda P, tau: sum(w * torch.exp(-s * tau) for s, w in nodes) * P if nodes else P
        out = ~inside
        if bool(out.any()):
            escaped += float((left(P[out], tau[out]) * ndot[src[out]]).sum()) / 12.0
        t = torch.full_like(P, t0)
        ray = [v[..., inside] for v in (src, pix, P, tau, t, norm, mag, sgn, k, i)]
        kids = []
        while ray[0].numel():
            src, pix, P, tau, t, norm, mag, sgn, k, i = ray
            ta = torch.where(mag > 0, (2 * k + 1).double() * 2.0 ** 20 / mag.clamp(min=1).double(), math.inf)
            tn = ta.amin(0)
            end = tn >= t_end
            tn = torch.where(end, t_end, tn)
            ds = (tn - t) * norm
            cell = (i[2] * n + i[1]) * n + i[0]
            kap = kappa[cell]
            dtau = kap * ds
            if nodes:
                frac, psi = torch.zeros_like(P), torch.zeros_like(P)
                for s, w in nodes:
                    e = w * torch.exp(-s * tau)
                    frac -= e * torch.expm1(-s * dtau)
                    psi += s * e
                a = P * frac
                thin = P * psi * ds
            else:
                a = P * -torch.expm1(-dtau)
                thin = P * ds
            g = rate[src] * torch.where(kap > 0, a / kap, thin)
            absorbed += float((a * ndot[src]).sum()) / 12.0
            if mode:
                mid = 0.5 * (t + tn)
                p = mid * mag.double() * 2.0 ** -21 - k.double()      # offset from the cell centre, along the ray
                p = p * sgn.double()
                face = torch.stack([0.5 + p[0], 0.5 - p[0], 0.5 + p[1], 0.5 - p[1], 0.5 + p[2], 0.5 - p[2]])
                de, f = face.min(0).values, face.argmin(0)
                l_pix = mid * norm * math.sqrt(math.pi / 3.0) / 2.0 ** level
                axis, up = f // 2, f % 2 * 2 - 1
                j = [i[b] + up * (axis == b) for b in range(3)]
                if periodic:
                    j = [v % n for v in j]
                there = (j[0] >= 0) & (j[0] < n) & (j[1] >= 0) & (j[1] < n) & (j[2] >= 0) & (j[2] < n)
                c2 = torch.where(there, (j[2] * n + j[1]) * n + j[0], 0)
                use = (2.0 * de < l_pix) & there & takes[c2]
                share = torch.where(use, 0.5 + de / l_pix, 1.0)
                gamma.index_add_(0, cell, g * share)
                gamma.index_add_(0, c2[use], (g * (1.0 - share) * kap)[use] / kappa[c2[use]])
            else:
                gamma.index_add_(0, cell, g)
            tau = tau + dtau
            P = P if nodes else P - a
            spent = tau >= TAU_MAX
            hit = (ta == tn) & ~end
            k, i = k + hit, i + sgn * hit
            i = i % n if periodic else i
            gone = ~end & ~spent & ~((i >= 0) & (i < n)).all(0)
            done = end & ~spent
            if split:
                kids.append([v[done] for v in (src, pix, P, tau)])
            else:
                gone = gone | done
            escaped += float((left(P[gone], tau[gone]) * ndot[src[gone]]).sum()) / 12.0
            keep = ~(end | spent | gone)
            ray = [v[..., keep] for v in (src, pix, P, tau, tn, norm, mag, sgn, k, i)]
        if kids:
            src, pix, P, tau = (torch.cat(v) for v in zip(*kids))
            if len(src):
                pix = 4 * pix.repeat_interleave(4) + torch.arange(4, device=dev).repeat(len(src))
                stack.append((level + 1, src.repeat_interleave(4), pix, 0.25 * P.repeat_interleave(4),
                              tau.repeat_interleave(4)))
    return gamma, (absorbed, escaped)
