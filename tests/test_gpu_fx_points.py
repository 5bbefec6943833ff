"""FP64 solves of point-like sources: lines that one cell, or a few, dominate,
where the fixed-point scale is set by the 1-norm and the values of the first
butterfly reach its bound.  One cell at every leg of the first radices, one
particle deposited on eight cells, one y-row per plane, over the mantissas of
the amplitude, through every entry point that runs the FP64 passes; against the
same convolution by torch's FP64 transforms with the plan's own spectrum."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# as in test_gpu_fx.py: both sides round about 3 log2(2N) times in each
# direction, each time by at most 2^-53 of a line's norm
TOL = 64 * 2.0 ** -53
AMPS = [1.0, 1.1, 1.25, 1.4, 1.6, 1.8]
SPECIALISED = [32, 48, 64, 96, 128, 192, 256]
GENERIC = [16, 50, 75, 100, 125]


def transform(S, rho):
    """The convolution with the octant S."""
    import torch
    for d in range(2):  # z and y are folded, x is the half spectrum
        S = torch.cat((S, S.narrow(d, 1, S.shape[d] - 2).flip(d)), d)
    n = [2 * m for m in rho.shape]
    f = torch.fft.rfftn(rho, s=n) * S
    return torch.fft.irfftn(f, s=n, norm="forward")[:rho.shape[0], :rho.shape[1], :rho.shape[2]]


def spectrum(plan):
    import torch
    return torch.from_numpy(plan.spectrum()).cuda()


def legs(n):
    """Positions in every eighth and every fifth of the box, odd ones too."""
    return sorted({(2 * k + 1) * n // 16 for k in range(8)} | {(2 * k + 1) * n // 10 for k in range(5)} | {0, n - 1})


def cells(shape, seed):
    """Sources of one cell: every leg in y, the amplitudes in turn, x and z
    (the phases) drawn; as many more with a leg in z."""
    import torch
    rng = np.random.default_rng(seed)
    nz, ny, nx = shape
    for axis, n in ((1, ny), (0, nz)):
        for i, p in enumerate(legs(n)):
            at = [int(rng.integers(m)) for m in shape]
            at[axis] = p
            rho = torch.zeros(shape, dtype=torch.float64, device="cuda")
            rho[tuple(at)] = AMPS[(i + seed) % len(AMPS)]
            yield rho


def planes(shape, seed):
    """One cell per z-plane (every plane its own y, x and amplitude), and one
    whole y-row per plane: a line of the second pass each."""
    import torch
    rng = np.random.default_rng(seed)
    nz, ny, nx = shape
    z = torch.arange(nz, device="cuda")
    y = torch.from_numpy(rng.permutation(max(ny, nz))[:nz] % ny).cuda()
    a = torch.tensor([AMPS[(i + seed) % len(AMPS)] for i in range(nz)], dtype=torch.float64, device="cuda")
    rho = torch.zeros(shape, dtype=torch.float64, device="cuda")
    rho[z, y, torch.from_numpy(rng.integers(nx, size=nz)).cuda()] = a
    yield rho
    rho = torch.zeros(shape, dtype=torch.float64, device="cuda")
    rho[z, y, :] = a[:, None]
    yield rho


def particles(shape, seed, count):
    """Single particles, each deposited on eight cells."""
    import torch
    rng = np.random.default_rng(seed)
    for i in range(count):
        at = [int(rng.integers(m - 1)) for m in shape]
        w = [rng.uniform(0.0, 1.0) ** 3 for _ in range(3)]
        rho = torch.zeros(shape, dtype=torch.float64, device="cuda")
        for c in range(8):
            b = [(c >> d) & 1 for d in range(3)]
            rho[tuple(at[d] + b[d] for d in range(3))] = AMPS[i % 6] * np.prod([w[d] if b[d] else 1 - w[d] for d in range(3)])
        yield rho


def sources(shape, seed):
    big = max(shape) > 128
    for i, rho in enumerate(cells(shape, seed)):
        if not big or i % 3 == seed % 3:
            yield rho
    for s in range(1 if big else 3):
        yield from planes(shape, seed + s)
    yield from particles(shape, seed, 2 if big else 6)


def check(got, want, scale):
    err, ref = float((got - want).abs().max()), float(scale.abs().max())
    assert err <= TOL * ref, err / ref


@pytest.mark.parametrize("N", SPECIALISED + GENERIC)
def test_solve(fsp, N):
    plan = fsp.Plan(N, 1.0, "he", "f64")
    S = spectrum(plan)
    for rho in sources((N, N, N), N):
        want = transform(S, rho)
        check(plan.solve(rho), want, want)


def test_largest_length(fsp):
    plan = fsp.Plan(512, 1.0, "he", "f64")
    S = spectrum(plan)
    for rho in list(cells((512, 512, 512), 1))[3::7]:
        want = transform(S, rho)
        check(plan.solve(rho), want, want)


@pytest.mark.parametrize("N", [64, 128])
def test_f64df(fsp, N):
    plan = fsp.Plan(N, 1.0, "vg_dct", "f64df")
    S = spectrum(plan)
    for rho in sources((N, N, N), 7):
        want = transform(S, rho)
        check(plan.solve(rho), want, want)


@pytest.mark.parametrize("n3", [(32, 64, 128), (128, 32, 64), (64, 256, 512), (30, 45, 64), (40, 75, 50)])
def test_boxes(fsp, n3):
    plan = fsp.Plan(n3, tuple(n / 64 for n in n3), "he", "f64")
    S = spectrum(plan)
    for rho in sources(n3[::-1], 3):
        want = transform(S, rho)
        check(plan.solve(rho), want, want)


@pytest.mark.parametrize("N", [64, 75])
def test_field(fsp, N):
    """E = -grad phi against the convolution with x_a / (4 pi r^3)."""
    import torch
    plan = fsp.Plan(N, 1.0, "he", "f64")
    plan.field_init()
    h = 1.0 / N
    ax = torch.arange(N + 1, dtype=torch.float64, device="cuda") * h
    r2 = ax[:, None, None] ** 2 + ax[None, :, None] ** 2 + ax[None, None, :] ** 2
    r2[0, 0, 0] = 1.0
    for a in range(3):
        shape = [1, 1, 1]
        shape[2 - a] = -1
        T = ax.reshape(shape) / (4 * np.pi * r2 ** 1.5)
        full = T
        for d in range(3):
            if d == 2 - a:
                pos = full.narrow(d, 0, N)
                full = torch.cat((pos, torch.zeros_like(full.narrow(d, N, 1)), -pos.narrow(d, 1, N - 1).flip(d)), d)
            else:
                full = torch.cat((full, full.narrow(d, 1, N - 1).flip(d)), d)
        K = torch.fft.rfftn(full)
        for rho in list(sources((N, N, N), a))[::2]:
            want = torch.fft.irfftn(K * torch.fft.rfftn(rho, s=[2 * N] * 3), s=[2 * N] * 3)[:N, :N, :N] * h ** 3
            check(plan.solve_field(rho)[a], want, want)


def test_batch(fsp):
    import torch
    Ns = [64, 50, 32, 75, 128]
    plans = [fsp.Plan(N, 1.0, "he", "f64") for N in Ns]
    spectra = [spectrum(p) for p in plans]
    for k in range(6):
        rhos = [list(cells((N, N, N), k))[(5 * k) % 13] for N in Ns]
        phis = [torch.empty_like(r) for r in rhos]
        b = fsp.Batch(plans, rhos, phis)
        b.launch()
        assert b.wait() == fsp.FSP_OK
        for S, r, f in zip(spectra, rhos, phis):
            want = transform(S, r)
            check(f, want, want)
        b.close()


@pytest.mark.parametrize("N", [8, 15, 16, 25, 32])
def test_noalloc(fsp, N):
    import torch
    plan = fsp.Plan(N, 1.0, "he", "f64")
    S = spectrum(plan)
    for rho in sources((N, N, N), 2):
        phi = torch.full_like(rho, float("nan"))
        want = transform(S, rho)
        check(fsp.solve_noalloc(S, rho, phi), want, want)


@pytest.mark.parametrize("n", [16, 25, 50, 60, 64, 90, 128, 150, 200, 250, 256, 450, 512, 1024])
@pytest.mark.parametrize("sign", [-1, 1])
def test_c2c_single_entries(fsp, n, sign):
    """Every position of a line, every amplitude, several phases."""
    import torch
    rng = np.random.default_rng(n)
    pos = np.repeat(np.arange(n), len(AMPS))
    x = np.zeros((len(pos), n), np.complex128)
    x[np.arange(len(pos)), pos] = np.tile(AMPS, n) * np.exp(2j * np.pi * rng.uniform(size=len(pos)))
    t = torch.from_numpy(x).cuda()
    got = fsp.fft_c2c(t, sign)
    want = torch.fft.fft(t) if sign < 0 else torch.fft.ifft(t, norm="forward")
    err = float(((got - want).abs().amax(1) / t.abs().sum(1)).max())
    assert err <= TOL, err
