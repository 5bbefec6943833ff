"""The workloads this package is timed on, through its public entry points.

A case is a dict of plain values: `kind` names the entry point (a solve, a
field solve, a batch, a plan rebuilt for a new box and used once), n_x, n_y,
n_z the cells, L_x, L_y, L_z the box, `algo` and `dtype` the plan's options.
Sources are charge densities as a particle code deposits them: a few Gaussian
bunches, each cell with its own shot noise.
"""
import math
import random

import torch

import paper_2405_02603_gb300 as fsp

BATCH_SIZES = (32, 48, 64, 96, 128, 160)


def _cube(name, kind, n, algo, dtype, L=1.0):
    return {"name": name, "kind": kind, "nx": n, "ny": n, "nz": n, "Lx": L, "Ly": L, "Lz": L, "algo": algo,
            "dtype": dtype}


def listed():
    return [
        # the smallest call: the paper's accuracy test grid in the package's
        # default precision; a time step of a small particle run
        _cube("solve_f64_n32_vg", "solve", 32, "vg", "f64"),
        # a served small request (the server issues the same launches)
        _cube("solve_f32_n64_he", "solve", 64, "he", "f32", 2.0),
        # a mesh chosen for the physics, not for the transform: odd, 3 * 5^2,
        # default method and precision
        _cube("solve_f64_n75_vg_dct", "solve", 75, "vg_dct", "f64"),
        # the ordinary mesh of the precision study
        _cube("solve_f32_n128_vg", "solve", 128, "vg", "f32"),
        # the headline workload: one Vico-Greengard solve at N = 256 in the
        # mixed-precision form, in plain FP64 and in the double-float form
        _cube("solve_f32_n256_vg", "solve", 256, "vg", "f32"),
        _cube("solve_f64_n256_vg", "solve", 256, "vg", "f64"),
        _cube("solve_f64df_n256_vg", "solve", 256, "vg", "f64df"),
        # the largest cube
        _cube("solve_f32_n512_vg_dct", "solve", 512, "vg_dct", "f32"),
        # the particle push wants E = -grad phi: three components per step
        _cube("field_f32_n256_vg", "field", 256, "vg", "f32"),
        # the 1 x 1 x 2 box of the weak-scaling runs
        {"name": "box_f32_256x256x512_vg_dct", "kind": "solve", "nx": 256, "ny": 256, "nz": 512, "Lx": 1.0, "Ly": 1.0,
         "Lz": 2.0, "algo": "vg_dct", "dtype": "f32"},
        # many uneven sources at once: 64 solves of mixed radices in one
        # persistent launch, the batch replayed as a time loop would
        {"name": "batch_f32_64_vg_dct", "kind": "batch", "count": 64, "mix": 2406, "Lx": 1.0, "Ly": 1.0, "Lz": 1.0,
         "algo": "vg_dct", "dtype": "f32"},
        # bunch-fitted boxes: the box changes each step, so the spectrum is
        # built for it, used for one solve and dropped
        _cube("refit_f64_n96_vg_dct", "refit", 96, "vg_dct", "f64"),
    ]


def _smooth(lo, hi):
    """The 2/3/5-smooth sizes in [lo, hi]."""
    out = []
    for n in range(lo, hi + 1):
        m = n
        for p in (2, 3, 5):
            while m % p == 0:
                m //= p
        if m == 1:
            out.append(n)
    return out


def _log_pick(rng, sizes):
    """One of `sizes`, spread evenly over the logarithm of the range."""
    x = math.exp(rng.uniform(math.log(sizes[0]), math.log(sizes[-1])))
    return min(sizes, key=lambda n: abs(math.log(n) - math.log(x)))


def draw(rng):
    kind = rng.choice(("solve", "solve", "solve", "solve", "solve", "field", "box", "batch", "refit"))
    L = round(rng.uniform(0.5, 2.0), 3)
    if kind == "batch":
        return {"kind": "batch", "count": rng.randint(8, 48), "mix": rng.randrange(1 << 20), "Lx": L, "Ly": L, "Lz": L,
                "algo": rng.choice(("he", "vg_dct")), "dtype": rng.choice(("f32", "f32", "f64"))}
    if kind == "refit":
        c = _cube("", "refit", _log_pick(rng, _smooth(24, 128)), rng.choice(("he", "vg_dct")),
                  rng.choice(("f64", "f32")), L)
    elif kind == "field":
        dtype = rng.choice(("f32", "f64"))
        c = _cube("", "field", _log_pick(rng, _smooth(24, 256 if dtype == "f32" else 128)),
                  rng.choice(("he", "vg", "vg_dct")), dtype, L)
    elif kind == "box":
        dtype = rng.choice(("f32", "f64"))
        sizes = _smooth(24, 256 if dtype == "f32" else 128)
        n = [_log_pick(rng, sizes) for _ in range(2)]
        n.append(rng.choice([m for m in sizes if min(n) <= m <= 2 * min(n)]))
        h = L / max(n)
        c = {"kind": "solve", "nx": n[0], "ny": n[1], "nz": n[2], "Lx": h * n[0], "Ly": h * n[1], "Lz": h * n[2],
             "algo": "he" if 3 * min(n) < 1.2 * math.sqrt(sum(m * m for m in n)) else rng.choice(("he", "vg_dct")),
             "dtype": dtype}
    else:
        dtype = rng.choice(("f32", "f32", "f64", "f64", "f64df"))
        if dtype == "f64df":
            n = rng.choice((32, 64, 128, 256))
        else:
            n = _log_pick(rng, _smooth(16, 384 if dtype == "f32" else 200))
        c = _cube("", "solve", n, rng.choice(("he", "vg", "vg_dct") if n <= 200 else ("he", "vg_dct")), dtype, L)
    c.pop("name", None)
    return c


def _batch_sizes(case):
    rng = random.Random(case["mix"])
    return [rng.choice(BATCH_SIZES) for _ in range(case["count"])]


def _shape(case):
    return case["nx"], case["ny"], case["nz"]


def _box(case):
    return case["Lx"], case["Ly"], case["Lz"]


def _source(n, L, dtype, seed):
    """(n_z, n_y, n_x): eight Gaussian bunches of about unit charge with 2 %
    shot noise per cell, rounded to the plan's array type."""
    rng = random.Random(seed)
    rho = torch.zeros((n[2], n[1], n[0]), dtype=torch.float64, device="cuda")
    x = [(torch.arange(n[a], dtype=torch.float64, device="cuda") + 0.5) / n[a] - 0.5 for a in range(3)]
    for _ in range(8):
        sigma, weight = rng.uniform(0.03, 0.08), rng.uniform(0.5, 1.5)
        g = [torch.exp(-((x[a] - rng.uniform(-0.3, 0.3)) ** 2) / (2 * sigma ** 2)) for a in range(3)]
        amp = weight / ((2 * math.pi) ** 1.5 * sigma ** 3 * L[0] * L[1] * L[2])
        rho += amp * g[2][:, None, None] * g[1][None, :, None] * g[0][None, None, :]
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    rho *= 1 + 0.02 * torch.randn(rho.shape, generator=gen, dtype=torch.float64, device="cuda")
    return rho.to(fsp.torch_dtype(dtype))


def _sources(case, seed):
    """The sources of one pass, as a list."""
    L, dtype = _box(case), case["dtype"]
    if case["kind"] == "batch":
        return [_source((n, n, n), L, dtype, 1000003 * seed + i) for i, n in enumerate(_batch_sizes(case))]
    return [_source(_shape(case), L, dtype, seed)]


def _plan(case, n, L):
    if n[0] == n[1] == n[2] and L[0] == L[1] == L[2]:
        return fsp.Plan(n[0], L[0], case["algo"], case["dtype"])
    return fsp.Plan(n, L, case["algo"], case["dtype"])


def prepare(case, seed):
    rhos = _sources(case, seed)
    L = _box(case)
    state = {"case": case, "rho": rhos[0]}
    if case["kind"] == "batch":
        # plans of one size share the stored spectrum, each with its own workspace
        spectra, plans = {}, []
        for n in _batch_sizes(case):
            if n not in spectra:
                plans.append(fsp.Plan(n, L[0], case["algo"], case["dtype"]))
                spectra[n] = plans[-1].spectrum()
            else:
                plans.append(fsp.Plan.from_spectrum(n, L[0], case["algo"], case["dtype"], spectra[n]))
        state["phis"] = [torch.empty_like(r) for r in rhos]
        state["batch"] = fsp.Batch(plans, rhos, state["phis"])
    elif case["kind"] == "refit":
        state["phi"] = torch.empty_like(rhos[0])
    else:
        plan = state["plan"] = _plan(case, _shape(case), L)
        if case["kind"] == "field":
            plan.field_init()
            state["E"] = [torch.empty_like(rhos[0]) for _ in range(3)]
        else:
            state["phi"] = torch.empty_like(rhos[0])
    return state


def run(state):
    case = state["case"]
    if case["kind"] == "solve":
        return state["plan"].solve_into(state["rho"], state["phi"])
    if case["kind"] == "field":
        return state["plan"].solve_field_into(state["rho"], *state["E"])
    if case["kind"] == "batch":
        state["batch"].launch()
        return state["phis"]
    plan = _plan(case, _shape(case), _box(case))
    plan.solve_into(state["rho"], state["phi"])
    plan.close()
    return state["phi"]


# ------------------------------------------------------------------ work --
def _fft(n):
    return 5.0 * n * math.log2(n)


def _solve_work(n, dtype):
    """The source in, the potential out, the spectrum read once; the pruned
    transforms of the doubled grid and the multiply."""
    nx, ny, nz = n
    r = 4 if dtype == "f32" else 8
    rows = ny * nz * _fft(nx)
    cols = nz * (nx + 1) * _fft(2 * ny)
    lines = 2 * ny * (nx + 1)
    return {"bytes": r * (2 * nx * ny * nz + (nx + 1) * (ny + 1) * (nz + 1)),
            "flops": 2 * rows + 2 * cols + lines * (2 * _fft(2 * nz) + 2 * 2 * nz)}


def work(case):
    if case["kind"] == "batch":
        each = [_solve_work((n, n, n), case["dtype"]) for n in _batch_sizes(case)]
        return {k: sum(w[k] for w in each) for k in ("bytes", "flops")}
    n, dtype = _shape(case), case["dtype"]
    nx, ny, nz = n
    w = _solve_work(n, dtype)
    r = 4 if dtype == "f32" else 8
    if case["kind"] == "field":
        # one forward transform, three multiplies and three inverses
        fwd = (w["flops"] - 2 * 2 * nz * 2 * ny * (nx + 1)) / 2
        w["flops"] = 4 * fwd + 3 * 2 * 2 * nz * 2 * ny * (nx + 1)
        w["bytes"] = r * (4 * nx * ny * nz + 3 * (nx + 1) * (ny + 1) * (nz + 1))
    elif case["kind"] == "refit":
        # the solve, its source and potential, and real even transforms of
        # the (2n+1)^3 octant of samples (pruned as each axis is done) and
        # of the (n+1)^3 kernel
        dct = lambda m: 2.5 * m * math.log2(m)  # noqa: E731
        if case["algo"] != "he":
            w["flops"] += (2 * nz + 1) * ((2 * ny + 1) * dct(2 * nx) + (nx + 1) * dct(2 * ny)) + \
                (nx + 1) * (ny + 1) * dct(2 * nz)
        w["flops"] += (ny + 1) * (nz + 1) * dct(nx) + (nx + 1) * (nz + 1) * dct(ny) + (nx + 1) * (ny + 1) * dct(nz)
        w["bytes"] = r * 2 * nx * ny * nz
    return w


# ----------------------------------------------------------------- exact --
def _along(v, a):
    """A vector along axis a (x, y, z) of an array [z][y][x]."""
    return v.reshape([-1 if 2 - a == d else 1 for d in range(3)])


def _even_dft(t, dim):
    """sum over the even extension (period 2 (len - 1)) of t cos, first half."""
    m = t.shape[dim]
    ext = torch.cat((t, t.narrow(dim, 1, m - 2).flip(dim)), dim)
    del t
    return torch.fft.rfft(ext, dim=dim).real.contiguous()


def _odd_dft(t, dim):
    """sum over the odd extension of t sin, first half."""
    m = t.shape[dim]
    ext = torch.cat((t, -t.narrow(dim, 1, m - 2).flip(dim)), dim)
    del t
    return -torch.fft.rfft(ext, dim=dim).imag.contiguous()


def _kernel(algo, n, h, comp=None):
    """T[m], m in [0, n] per axis: the Green's function's samples, or (comp)
    those of its negative derivative along axis comp."""
    ar = lambda c: torch.arange(c, dtype=torch.float64, device="cuda")  # noqa: E731
    if algo == "he":
        c = [_along(ar(n[a] + 1) * h[a], a) for a in range(3)]
        r = torch.sqrt(c[0] ** 2 + c[1] ** 2 + c[2] ** 2)
        r[0, 0, 0] = 1.0
        if comp is None:
            return 1.0 / (4 * math.pi * r)
        return c[comp] / (4 * math.pi * r ** 3)
    Lt = 1.1 * math.sqrt(sum((n[a] * h[a]) ** 2 for a in range(3)))
    k = [_along(ar(2 * n[a] + 1) * (2 * math.pi / (4 * n[a] * h[a])), a) for a in range(3)]
    kk = torch.sqrt(k[0] ** 2 + k[1] ** 2 + k[2] ** 2)
    kk[0, 0, 0] = 1.0
    g = 2.0 * (torch.sin(0.5 * Lt * kk) / kk) ** 2
    g[0, 0, 0] = 0.5 * Lt * Lt
    del kk
    if comp is not None:
        g *= k[comp]
    for a in range(3):
        g = (_odd_dft if a == comp else _even_dft)(g, 2 - a).narrow(2 - a, 0, n[a] + 1).contiguous()
    return g / math.prod(4 * n[a] * h[a] for a in range(3))


def _convolve(T, rho, h, comp=None):
    """h^3 sum_j T[|i - j|] rho_j, by the transform of the doubled grid; with
    comp, T is odd in that axis."""
    n = rho.shape[::-1]
    for a in range(3):
        dim, m = 2 - a, n[a]
        if a == comp:  # an odd sequence vanishes at the fold
            pos = T.narrow(dim, 0, m)
            T = torch.cat((pos, torch.zeros_like(T.narrow(dim, m, 1)), -pos.narrow(dim, 1, m - 1).flip(dim)), dim)
        else:
            T = torch.cat((T, T.narrow(dim, 1, m - 1).flip(dim)), dim)
    spec = torch.fft.rfftn(T)
    del T
    spec *= torch.fft.rfftn(rho, s=[2 * m for m in rho.shape])
    out = torch.fft.irfftn(spec, s=[2 * m for m in rho.shape])
    return (out[:rho.shape[0], :rho.shape[1], :rho.shape[2]] * (h[0] * h[1] * h[2])).contiguous()


def exact(case, seed):
    rhos, L = _sources(case, seed), _box(case)
    if case["kind"] == "batch":
        kernels, out = {}, []
        for n, rho in zip(_batch_sizes(case), rhos):
            h = [L[a] / n for a in range(3)]
            if n not in kernels:
                kernels[n] = _kernel(case["algo"], (n, n, n), h)
            out.append(_convolve(kernels[n], rho.double(), h))
        return out
    n = _shape(case)
    h = [L[a] / n[a] for a in range(3)]
    rho = rhos[0].double()
    if case["kind"] == "field":
        return tuple(_convolve(_kernel(case["algo"], n, h, a), rho, h, a) for a in range(3))
    return _convolve(_kernel(case["algo"], n, h), rho, h)
