"""What the framework's users have it do, as cases for a timing program.

A case is one call sequence through the public entry points (``native``) on a
medium and a set of sources: coupled steps of one grid (state in, trace,
update, rates out), single traces, batches of grids, finite-light steps.  The
media are those of ``synth`` (Test 1 of arXiv:1012.2865, the log-normal clumpy
medium, Application 5), drawn here on the GPU from a seed.  ``exact`` is the
method written out in plain FP64 torch operations.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1012_2865_gb300 import native, synth

DEV = "cuda"
MYR_S = 3.15576e13
KPC_CM = 3.0856775814913673e21
ALPHA_B = 2.59e-13
DT_S = 0.5 * MYR_S
EV_ERG = 1.602176634e-12
E_ION = (13.6, 24.6, 54.4)                  # H I, He I, He II
SIGMA = (6.3e-18, 7.43e-18, 1.58e-18)
PHI_C, F_TERM, LEVEL0, MAX_LEVEL = 5.1, 1e-10, 1, 14
SIDES = (32, 48, 64, 96, 128, 192)          # grid sides of a batch


# --------------------------------------------------------------------------
# The cases
# --------------------------------------------------------------------------
def _case(name, kind, n, medium, nsrc, precision="fp32_mixed", **more):
    nx, ny, nz = (n, n, n) if isinstance(n, int) else n
    c = dict(name=name, kind=kind, nx=nx, ny=ny, nz=nz, medium=medium, nsrc=nsrc, precision=precision,
             off_lattice=False, fc=False, adaptive=False)
    c.update(more)
    return c


def listed():
    return [
        # the smallest real call: the paper's Test 1 at 32^3 in plain FP64, one coupled step from the neutral medium
        _case("test1_32_fp64", "step", 32, "neutral", 1, "fp64"),
        # the convergence run late in its evolution: a step of the 128^3 Stroemgren sphere
        _case("stromgren_128", "step", 128, "front", 1),
        # the same step on the FP64 path, which users run to check the mixed one
        _case("stromgren_128_fp64", "step", 128, "front", 1, "fp64"),
        # that step for a code that keeps its state on the host: pinned buffers, uploads and read-backs not waited for
        _case("stromgren_128_host", "host", 128, "front", 1),
        # a reionisation box at its start: 1000 galaxies in a neutral clumpy medium, heating on
        _case("clumpy_256", "trace", 256, "clumpy", 1000),
        # and at its end: an ionised box that every ray crosses, the longest trace of a run
        _case("ionised_128", "trace", 128, "ionised", 24),
        # a zoom region: odd sides, galaxies at any position, part ionised, the step length from the I-front
        _case("zoom_150x101x77", "step", (150, 101, 77), "partial", 12, off_lattice=True, adaptive=True),
        # galaxies at any position with the covering-factor correction on
        _case("covering_96", "trace", 96, "clumpy", 60, off_lattice=True, fc=True),
        # hydrogen and helium ionising photons, each with its own absorber and rates
        _case("helium_128", "trace", 128, "typed", 30),
        # Application 5: a step with a finite speed of light, packages of every age in flight
        _case("pulse_128", "flight", 128, "pulse", 1, cells_per_step=1.96),
        # many independent boxes in one launch
        _case("batch_24", "batch", 192, "clumpy", 256, grids=24, steps=0),
        # the served form: requests of several sizes advanced together by captured steps
        _case("serve_8", "batch", 128, "clumpy", 64, grids=8, steps=3),
    ]


def draw(rng):
    def side(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def many(lo, hi):
        return max(1, side(lo, hi))

    prec = "fp64" if rng.random() < 0.2 else "fp32_mixed"
    kind = rng.choice(["front", "step", "host", "clumpy", "ionised", "typed", "flight", "batch", "serve"])
    if kind in ("front", "host"):
        n = side(32, 128 if prec == "fp64" or kind == "host" else 256)
        c = _case("", "host" if kind == "host" else "step", n, "front", 1, "fp32_mixed" if kind == "host" else prec)
    elif kind == "step":
        n = tuple(side(32, 96 if prec == "fp64" else 160) for _ in range(3))
        c = _case("", "step", n, rng.choice(["partial", "neutral"]), many(1, 12), prec,
                  off_lattice=rng.random() < 0.7, adaptive=rng.random() < 0.5)
    elif kind == "clumpy":
        n = tuple(side(48, 128 if prec == "fp64" else 224) for _ in range(3))
        c = _case("", "trace", n, "clumpy", many(10, 100 if prec == "fp64" else 800), prec,
                  off_lattice=rng.random() < 0.5, fc=rng.random() < 0.3)
    elif kind == "ionised":
        n = tuple(side(32, 64 if prec == "fp64" else 128) for _ in range(3))
        c = _case("", "trace", n, "ionised", many(1, 3 if prec == "fp64" else 24), prec, off_lattice=rng.random() < 0.5)
    elif kind == "typed":
        n, m = (side(32, 64), many(3, 9)) if prec == "fp64" else (side(48, 128), many(3, 30))
        c = _case("", "trace", n, "typed", m, prec, off_lattice=rng.random() < 0.5)
    elif kind == "flight":
        c = _case("", "flight", side(48, 128), "pulse", 1, cells_per_step=rng.uniform(1.5, 6.0))
    else:
        c = _case("", "batch", rng.choice((64, 96, 128, 192)), "clumpy", many(8, 256 if kind == "batch" else 64),
                  grids=rng.randint(2, 24 if kind == "batch" else 8), steps=0 if kind == "batch" else rng.randint(1, 3))
    del c["name"]
    return c


# --------------------------------------------------------------------------
# Inputs, on the GPU, from the seed
# --------------------------------------------------------------------------
def _generator(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _f32(a):
    return a.float().double()


def _lognormal(dims, gen, mean=1e-2, sigma=1.0):
    """Log-normal density from a Gaussian field with P(k) ~ k^-3, flattened x-fastest."""
    nx, ny, nz = dims
    w = torch.fft.rfftn(torch.randn((nz, ny, nx), generator=gen, device=DEV, dtype=torch.float64))
    k = torch.sqrt(torch.fft.fftfreq(nz, device=DEV, dtype=torch.float64)[:, None, None] ** 2 +
                   torch.fft.fftfreq(ny, device=DEV, dtype=torch.float64)[None, :, None] ** 2 +
                   torch.fft.rfftfreq(nx, device=DEV, dtype=torch.float64)[None, None, :] ** 2)
    amp = torch.where(k > 0, k, torch.ones_like(k)) ** -1.5
    amp[0, 0, 0] = 0.0
    g = torch.fft.irfftn(w * amp, s=(nz, ny, nx))
    g = (g - g.mean()) / g.std()
    e = torch.exp(sigma * g)
    return _f32((mean * e / e.mean()).reshape(-1))


def _radius(dims, at):
    """Distance of every cell centre from `at` (cell units), x fastest."""
    x, y, z = (torch.arange(n, device=DEV, dtype=torch.float64) + 0.5 - p for n, p in zip(dims, at))
    return torch.sqrt(x[None, None, :] ** 2 + y[None, :, None] ** 2 + z[:, None, None] ** 2).reshape(-1)


def _inputs(case, seed, dims=None, nsrc=None):
    dims = dims or (case["nx"], case["ny"], case["nz"])
    nsrc = nsrc or case["nsrc"]
    gen, rng = _generator(seed), np.random.default_rng(seed)
    medium = case["medium"]
    ncell = dims[0] * dims[1] * dims[2]
    box_kpc = 1000.0 if medium == "pulse" else 6.6
    box = synth.box_cm(dims[0], box_kpc)
    dx = box / dims[0]
    g = dict(dims=dims, box_len_cm=box, dx=dx)
    ones = torch.ones(ncell, device=DEV, dtype=torch.float64)
    if medium in ("front", "neutral") and nsrc == 1 and not case["off_lattice"]:
        # Test 1: uniform gas, one source in the corner; late snapshots hold an ionised octant behind the I-front
        g["pos_cm"], g["ndot"], g["e_ph_eV"] = np.zeros((1, 3)), np.array([5e48 * rng.uniform(0.95, 1.05)]), np.array([13.6])
        g["n_H"] = _f32(1e-3 * ones)
        x = ones.clone()
        if medium == "front":
            rs = (3 * 5e48 / (4 * math.pi * ALPHA_B * 1e-6)) ** (1 / 3)
            t = rng.uniform(450.0, 550.0) * MYR_S
            r_if = rs * (1 - math.exp(-t * ALPHA_B * 1e-3)) ** (1 / 3) / dx
            w = 3.0 * max(dims) / 128.0
            x = 1e-3 + (1 - 1e-3) / (1 + torch.exp(-(_radius(dims, (0, 0, 0)) - r_if) / w))
    elif medium == "pulse":
        g["pos_cm"], g["ndot"] = np.zeros((1, 3)), np.array([float(synth.pulse_rate(0.0)) * rng.uniform(1.0, 50.0)])
        g["e_ph_eV"] = np.array([29.6])
        g["n_H"], x = _f32(1e-4 * ones), 1e-5 * ones
        g["light_cm"] = case["cells_per_step"] * dx
    else:
        g["n_H"] = _lognormal(dims, gen)
        if case["off_lattice"]:
            g["pos_cm"] = rng.uniform(0, 1, (nsrc, 3)) * np.array(dims) * dx
        else:
            g["pos_cm"] = synth.cell_centre_cm(np.stack([rng.integers(0, d, nsrc) for d in dims], axis=1), dx)
        g["ndot"] = np.exp(rng.uniform(math.log(1e48), math.log(1e50), nsrc))
        g["e_ph_eV"] = rng.uniform(13.6, 29.6, nsrc)
        x = ones.clone()
        if medium == "ionised":
            x = 1e-4 * ones
        elif medium == "partial":
            # bubbles around the sources, a few cells wide fronts between them and the neutral gas
            r = torch.full_like(ones, float("inf"))
            for p in g["pos_cm"] / dx:
                r = torch.minimum(r, _radius(dims, p) / rng.uniform(0.1, 0.25) / min(dims))
            x = 1e-3 + (1 - 1e-3) / (1 + torch.exp(-(r - 1.0) * 12.0))
    g["x_HI"], g["x_HII"] = x, 1.0 - x
    g["types"] = np.zeros(nsrc, dtype=np.int32)
    if medium == "typed":
        g["types"] = (np.arange(nsrc) % 3).astype(np.int32)
        g["e_ph_eV"] = np.array(E_ION)[g["types"]] + rng.uniform(0.0, 16.0, nsrc)
        g["n_he"] = torch.stack([_f32(0.079 * 0.9 * g["n_H"]), _f32(0.079 * 0.1 * g["n_H"])])
    g["sigma_cm2"] = np.array(SIGMA)[g["types"]]
    return g


def _members(case, seed):
    """The grids of a batch: sides up to the case's, 1 to nsrc sources each; the seed draws what they hold."""
    rng = np.random.default_rng(case["nsrc"])
    sides = [s for s in SIDES if s <= case["nx"]]
    out = []
    for i in range(case["grids"]):
        n = int(rng.choice(sides))
        out.append(_inputs(case, seed * 1000 + i, (n, n, n), int(rng.integers(1, case["nsrc"] + 1))))
    return out


def _params(case, g):
    p = dict(level0=LEVEL0, phi_c=PHI_C, f_term=F_TERM, max_level=MAX_LEVEL, fc=case["fc"])
    if "light_cm" in g:
        p["light_cm"] = g["light_cm"]
    return p


_ctx = None


def _context():
    global _ctx
    if _ctx is None:
        _ctx = native.rt_ctx_create(torch.cuda.current_device())
    return _ctx


def _dtype(case):
    return native.RT_DTYPE_F64 if case["precision"] == "fp64" else native.RT_DTYPE_F32


def prepare(case, seed):
    torch.cuda.synchronize()
    st = dict(case=case)
    if case["kind"] == "batch":
        st["inputs"] = _members(case, seed)
        st["grids"] = [native.Grid(_context(), g, case["precision"]) for g in st["inputs"]]
        st["batch"] = native.Batch(_context())
        for gr in st["grids"]:
            st["batch"].add(gr)
        st["params"] = _params(case, st["inputs"][0])
        if case["steps"]:
            st["batch"].step(1, DT_S, 10, ALPHA_B, **st["params"])  # sizes the queue, captures the step
        else:
            st["batch"].trace(**st["params"])                      # sizes the queue
        return st
    g = st["input"] = _inputs(case, seed)
    gr = st["grid"] = native.Grid(_context(), g, case["precision"])
    if case["medium"] == "typed":
        gr.set_absorbers(g["n_he"][0].contiguous(), g["n_he"][1].contiguous())
        gr.set_source_types(g["types"])
    st["params"] = _params(case, g)
    if case["kind"] == "flight":
        # until light has crossed the box and packages of every age are in flight
        diag = math.sqrt(sum(n * n for n in g["dims"]))
        for _ in range(int(diag / case["cells_per_step"]) + 3):
            gr.set_source_rates(g["ndot"])
            gr.trace(**st["params"])
    else:
        gr.trace(**st["params"])  # a run's first trace sizes the queue
    if case["kind"] == "host":
        st["hx"], st["hz"] = g["x_HI"].cpu().pin_memory(), g["x_HII"].cpu().pin_memory()
        st["out"] = [[torch.empty(gr.ncell, dtype=torch.float32).pin_memory() for _ in range(2)] for _ in range(2)]
        st["turn"] = 0
    return st


def run(state):
    case, kind = state["case"], state["case"]["kind"]
    dt = _dtype(case)
    if kind == "batch":
        b = state["batch"]
        if not case["steps"]:
            b.trace(sync=False, **state["params"])
            return [native.rt_get_rates(gr.h, gr.ncell, dt, "device", want=("kph", "gamma")) for gr in state["grids"]]
        for gr, g in zip(state["grids"], state["inputs"]):
            native.rt_set_state(gr.h, g["x_HI"], g["x_HII"])
        b.step(case["steps"], DT_S, 10, ALPHA_B, **state["params"])
        return [gr.rates(dt, "device") for gr in state["grids"]]
    gr, g = state["grid"], state["input"]
    if kind == "host":
        k, x = state["out"][state["turn"]]
        state["turn"] ^= 1
        native.rt_set_state_async(gr.h, state["hx"], state["hz"])
        gr.trace(sync=False, **state["params"])
        gr.chem(DT_S, 10, ALPHA_B)
        native.rt_wait_rates(gr.h)  # the previous step's results are on the host
        native.rt_get_rates_async(gr.h, kph=k, x_HI=x, dtype=dt)
        return dict(kph=k, x_HI=x)
    if kind == "flight":
        gr.set_source_rates(g["ndot"])
        gr.trace(sync=False, **state["params"])
        return native.rt_get_rates(gr.h, gr.ncell, dt, "device", want=("kph", "gamma"))
    if kind == "step":
        native.rt_set_state(gr.h, g["x_HI"], g["x_HII"])
        gr.trace(sync=False, **state["params"])
        step = DT_S
        if case["adaptive"]:
            step = native.rt_timestep(gr.h, eps_ion=0.05, alpha_B=ALPHA_B, sigma_front=SIGMA[0], tau_front=0.5, dt_max=DT_S)
        gr.chem(step, 10, ALPHA_B)
        out = gr.rates(dt, "device")
        if case["adaptive"]:
            out["dt_s"] = np.float32(step)  # the step length is an FP32 quantity on either path
        return out
    b = gr.trace(**state["params"])
    out = dict(budget=np.array([b["emitted"], b["absorbed"], b["escaped"]]), counts=b["counts"].astype(np.int64))
    for t in range(3 if case["medium"] == "typed" else 1):
        if t == 0:
            r = native.rt_get_rates(gr.h, gr.ncell, dt, "device", want=("kph", "gamma"))
        else:
            r = gr.rates_typed(t, dt, "device")
        out["rates%d" % t] = dict(kph=r["kph"], gamma=r["gamma"])
    return out


def work(case):
    """Bytes: every field of the call once.  Flops: about 40 operations for each
    cell a package crosses (three plane distances, optical depth, e^-tau,
    deposits), and rays sample a cell that a source reaches some 9 (corner) to
    17 (interior) times at Phi_c = 5.1."""
    e = 8 if case["precision"] == "fp64" else 4
    if case["kind"] == "batch":
        sides = [s for s in SIDES if s <= case["nx"]]
        cells = case["grids"] * sum(s ** 3 for s in sides) / len(sides)
        nsrc, passes = case["grids"] * (case["nsrc"] + 1) / 2, max(1, case["steps"])
        side = max(sides) / 2
    else:
        cells, nsrc, passes, side = case["nx"] * case["ny"] * case["nz"], case["nsrc"], 1, case["nx"]
    # cells that one source reaches: the whole box when ionised, else until the
    # optical depth ends its rays (n_H = 1e-2 per cm^3 clumpy gas; voids carry rays about four times the mean path)
    if case["medium"] in ("ionised", "front", "pulse"):
        reach = cells
    elif case["medium"] == "neutral" and case["nsrc"] == 1:
        reach = min(cells, 0.52 * (23.0 / (6.3e-18 * 1e-3 * 6.6 * KPC_CM / side)) ** 3)
    else:
        reach = min(cells, 4.2 * (4 * 23.0 / (6.3e-18 * 1e-2 * 6.6 * KPC_CM / side)) ** 3)
    if case["medium"] == "partial":
        reach = max(reach, cells / 4)
    if case["medium"] == "typed":
        reach = max(reach, cells / 3)            # the He II third of the sources lights the whole box
    segments = passes * nsrc * reach * (9 if case["medium"] in ("front", "pulse") else 17)
    steps = case["kind"] in ("step", "host") or (case["kind"] == "batch" and case["steps"])
    fields = 8 + 8 + 2 * e                       # n_H, x_HI read; k_ph, Gamma written
    if steps:
        fields += 8 + 8 + 8 + e                  # x_HII read, both fractions written, x_HI handed out
    update = cells * 600 * passes if steps else 0  # 10 substeps
    return dict(bytes=cells * fields * (3 if case["medium"] == "typed" else 1), flops=segments * 40 + update)


# --------------------------------------------------------------------------
# The method in plain FP64 torch operations
# --------------------------------------------------------------------------
def _direction(level, pix):
    """Unit vectors of nested HEALPix pixel centres."""
    ns = 1 << level
    face, ipf = pix // (ns * ns), pix % (ns * ns)
    ix, iy = torch.zeros_like(pix), torch.zeros_like(pix)
    for b in range(level):
        ix |= ((ipf >> (2 * b)) & 1) << b
        iy |= ((ipf >> (2 * b + 1)) & 1) << b
    s, k = ix + iy + 1, face % 4
    north, south = face < 4, face >= 8
    cap_n, cap_s = north & (s > ns), south & (s < ns)
    nr = torch.where(cap_n, 2 * ns - s, torch.where(cap_s, s, torch.full_like(s, ns)))
    zq = 2 * torch.where(north, s, torch.where(south, s - 2 * ns, s - ns))
    tnum = torch.where(north | south, 2 * k + 1, 2 * k) * nr + ix - iy
    omz = (nr * nr).double() / float(3 * ns * ns)
    zb = zq.double() / float(3 * ns)
    cap = cap_n | cap_s
    z = torch.where(cap, torch.where(cap_s, -(1.0 - omz), 1.0 - omz), zb)
    st = torch.where(cap, torch.sqrt(omz * (2.0 - omz)), torch.sqrt((1.0 - zb) * (1.0 + zb)))
    b = 2 * nr
    a = tnum % (4 * b)
    q, m = a // b, a % b
    low, diag = 2 * m < b, 2 * m == b
    ang = (math.pi * 0.5) * (torch.where(low, m, b - m).double() / b.double())
    u, v = torch.cos(ang), torch.sin(ang)
    c0, s0 = torch.where(low, u, v), torch.where(low, v, u)
    half = math.sqrt(0.5)
    c0, s0 = torch.where(diag, half, c0), torch.where(diag, half, s0)
    c0, s0 = torch.where(m == 0, 1.0, c0), torch.where(m == 0, 0.0, s0)
    c = torch.where(q == 0, c0, torch.where(q == 1, -s0, torch.where(q == 2, -c0, s0)))
    s = torch.where(q == 0, s0, torch.where(q == 1, c0, torch.where(q == 2, -s0, -c0)))
    return torch.stack([st * c, st * s, z])


def _plane(c, s, n):
    """Distance from the source to the next cell plane on each axis."""
    t = ((c + (n > 0)).double() - s) / n
    return torch.where(n == 0, torch.full_like(t, float("inf")), t)


def _trace64(g, absorber, fc):
    """k_ph, Gamma ([type][cell]), (emitted, absorbed, escaped) and packages per level."""
    dims = torch.tensor(g["dims"], device=DEV)[:, None]
    nx, ny, _ = g["dims"]
    ncell, dx, nsrc = g["n_H"].numel(), g["dx"], len(g["ndot"])
    put = lambda a: torch.as_tensor(np.asarray(a, dtype=np.float64), device=DEV)  # noqa: E731
    S, sig = put(g["pos_cm"]).T.contiguous() / dx, put(g["sigma_cm2"])
    unit = put(g["ndot"]) / (12.0 * 4 ** LEVEL0)
    types = torch.as_tensor(g["types"].astype(np.int64), device=DEV)
    heat = (put(g["e_ph_eV"]) - put(E_ION)[types]) * EV_ERG
    n_abs = absorber.reshape(-1)
    K, G = torch.zeros_like(n_abs), torch.zeros_like(n_abs)
    zero = torch.zeros((), device=DEV, dtype=torch.float64)
    absorbed, escaped = zero.clone(), zero.clone()
    tau_term, counts = -math.log(F_TERM), [0] * (MAX_LEVEL + 1)
    src = torch.arange(nsrc, device=DEV).repeat_interleave(12 * 4 ** LEVEL0)
    pix = torch.arange(12 * 4 ** LEVEL0, device=DEV).repeat(nsrc)
    start = torch.zeros(src.numel(), device=DEV, dtype=torch.float64)
    level_in = (src, pix, start, torch.ones_like(start), start.clone())
    for level in range(LEVEL0, MAX_LEVEL + 1):
        rsplit = math.sqrt(12.0 * 4.0 ** level / (4.0 * math.pi * PHI_C)) if level < MAX_LEVEL else float("inf")
        theta = math.sqrt(4.0 * math.pi / (12.0 * 4.0 ** level))
        counts[level] = level_in[0].numel()
        nxt = []
        for lo in range(0, counts[level], 4_000_000):
            src, pix, r, P, tau = (v[lo:lo + 4_000_000] for v in level_in)
            n, s = _direction(level, pix), S[:, src]
            u = s + r * n
            c = torch.where(n < 0, torch.ceil(u) - 1, torch.floor(u)).long()
            inside = ((c >= 0) & (c < dims)).all(0)
            escaped += (P * unit[src])[~inside].sum()
            w = torch.nonzero(inside)[:, 0]
            src, pix, r, P, tau, n, s, c = src[w], pix[w], r[w], P[w], tau[w], n[:, w], s[:, w], c[:, w]
            while src.numel():
                t = _plane(c, s, n)
                rn = t.min(0).values
                split = rn > rsplit
                if bool(split.any()):
                    w = torch.nonzero(split)[:, 0]
                    four = torch.arange(4, device=DEV)
                    nxt.append((src[w].repeat_interleave(4), (4 * pix[w][:, None] + four).reshape(-1),
                                r[w].repeat_interleave(4), (P[w] / 4).repeat_interleave(4), tau[w].repeat_interleave(4)))
                    w = torch.nonzero(~split)[:, 0]
                    src, pix, r, P, tau, rn = src[w], pix[w], r[w], P[w], tau[w], rn[w]
                    n, s, c, t = n[:, w], s[:, w], c[:, w], t[:, w]
                dr = torch.clamp(rn - r, min=0.0)
                idx = c[0] + nx * (c[1] + ny * c[2]) + ncell * types[src]
                nh, un = n_abs[idx], unit[src]
                dtau = sig[src] * dx * nh * dr
                am = -torch.expm1(-dtau)
                phi = torch.where(dtau > 0, am / dtau, torch.ones_like(am))
                cover = torch.ones_like(phi)
                if fc:
                    L = r * theta
                    far = (s + n * (r + 0.5 * dr) - (c.double() + 0.5)).abs().max(0).values
                    cover = torch.where(L > 0, torch.clamp((0.5 + (0.5 - far) / L) ** 2, max=1.0), cover)
                add = P * un * sig[src] * dr / (dx * dx) * phi * cover
                dP = P * am
                absorbed += (dP * un).sum()
                P, tau = P - dP, tau + dtau
                end = tau > tau_term
                add = add + torch.where(end, P * un / (nh * dx ** 3) * cover, zero)
                absorbed += torch.where(end, P * un, zero).sum()
                K.index_add_(0, idx, add)
                G.index_add_(0, idx, add * heat[src])
                c = c + torch.where((t == rn) & (n != 0), torch.where(n > 0, 1, -1), 0)
                r = rn
                out = ~((c >= 0) & (c < dims)).all(0) & ~end
                escaped += torch.where(out, P * un, zero).sum()
                if bool((end | out).any()):
                    w = torch.nonzero(~(end | out))[:, 0]
                    src, pix, r, P, tau, n, s, c = src[w], pix[w], r[w], P[w], tau[w], n[:, w], s[:, w], c[:, w]
        if not nxt:
            break
        level_in = tuple(torch.cat(v) for v in zip(*nxt))
    budget = torch.stack([put(g["ndot"]).sum(), absorbed, escaped])
    return K.reshape(absorber.shape), G.reshape(absorber.shape), budget, counts


def _update64(n, x, z, k, dt_s, nsub):
    """Backward Euler of dx/dt = alpha_B n (1 - x)^2 - k x, the smaller fraction kept and the other its complement."""
    h = dt_s / nsub
    a, hk = h * ALPHA_B * n, h * k
    b = 1.0 + hk
    for _ in range(nsub):
        root = torch.sqrt(b * b + 4.0 * a * (z + hk))
        xn, zn = 2.0 * (a + x) / (2.0 * a + b + root), 2.0 * (z + hk) / (b + root)
        x, z = torch.where(xn <= zn, xn, 1.0 - zn), torch.where(xn <= zn, 1.0 - xn, zn)
    return x, z


def _timestep64(g, x, k):
    """Eq. dtelec with a 3^3 Gaussian over the cells of the grid, its minimum."""
    nx, ny, nz = g["dims"]
    n = g["n_H"]
    rate = (k + n * (1.0 - x) * ALPHA_B).abs()
    front = (SIGMA[0] * g["dx"] * n * x > 0.5) & (rate > 0)
    dt = torch.where(front, torch.clamp(0.05 / rate, max=DT_S), DT_S).reshape(1, 1, nz, ny, nx) / DT_S
    d = torch.arange(-1.0, 2.0, device=DEV, dtype=torch.float64)
    w = torch.exp(-0.5 * (d[:, None, None] ** 2 + d[None, :, None] ** 2 + d[None, None, :] ** 2)).reshape(1, 1, 3, 3, 3)
    conv = torch.nn.functional.conv3d
    return float((conv(dt, w, padding=1) / conv(torch.ones_like(dt), w, padding=1)).min()) * DT_S


def _step64(g, x, z, fc, dt_s, adaptive=False):
    k, gamma, _, _ = _trace64(g, g["n_H"] * x, fc)
    if adaptive:
        dt_s = _timestep64(g, x, k)
    x, z = _update64(g["n_H"], x, z, k, dt_s, 10)
    return k, gamma, x, z, dt_s


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        out = []
        for g in _members(case, seed):
            if not case["steps"]:
                k, gamma, _, _ = _trace64(g, g["n_H"] * g["x_HI"], case["fc"])
                out.append(dict(kph=k, gamma=gamma, x_HI=None))
                continue
            x, z = g["x_HI"], g["x_HII"]
            for _ in range(case["steps"]):
                k, gamma, x, z, _ = _step64(g, x, z, case["fc"], DT_S)
            out.append(dict(kph=k, gamma=gamma, x_HI=x))
        return out
    g = _inputs(case, seed)
    if kind == "flight":
        # once packages of every age are in flight a step deposits, shell by shell, what one whole trace does
        k, gamma, _, _ = _trace64(g, g["n_H"] * g["x_HI"], False)
        return dict(kph=k, gamma=gamma, x_HI=None)
    if kind in ("step", "host"):
        k, gamma, x, _, dt = _step64(g, g["x_HI"], g["x_HII"], case["fc"], DT_S, case["adaptive"])
        if kind == "host":
            return dict(kph=k, x_HI=x)
        return dict(kph=k, gamma=gamma, x_HI=x, **({"dt_s": dt} if case["adaptive"] else {}))
    absorber = (g["n_H"] * g["x_HI"])[None]
    if case["medium"] == "typed":
        absorber = torch.cat([absorber, g["n_he"]])
    k, gamma, budget, _ = _trace64(g, absorber, case["fc"])
    out = dict(budget=budget, counts=None)
    for t in range(absorber.shape[0]):
        out["rates%d" % t] = dict(kph=k[t], gamma=gamma[t])
    return out
