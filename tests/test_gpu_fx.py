"""The FP64 passes in 64-bit fixed point against the same convolution by
torch's FP64 transforms (with the plan's own spectrum): every specialised
length and odd ones on the generic engine, sources over the whole range of
exponents, boxes, and lines that hold an infinity or a NaN.
"""
import numpy as np
import pytest

import fsp_inputs as I

pytestmark = pytest.mark.gpu

# both sides round about 3 log2(2N) times in each direction, each time by at
# most 2^-53 of a line's norm: 54 roundings at N = 512
TOL = 64 * 2.0 ** -53


@pytest.fixture(scope="module")
def fsp():
    import paper_2405_02603_gb300 as m
    return m


def reference(plan, rho):
    import torch
    S = torch.from_numpy(plan.spectrum()).cuda()
    for d in range(2):  # z and y are folded, x is the half spectrum
        S = torch.cat((S, S.narrow(d, 1, S.shape[d] - 2).flip(d)), d)
    n = [2 * m for m in rho.shape]
    f = torch.fft.rfftn(rho, s=n) * S
    phi = torch.fft.irfftn(f, s=n, norm="forward")
    return phi[:rho.shape[0], :rho.shape[1], :rho.shape[2]]


def check(plan, rho):
    """Against the convolution of the absolute values, which is what the
    rounding of a transform is relative to (the kernel is positive)."""
    import torch
    t = torch.from_numpy(rho).cuda()
    a, b = plan.solve(t), reference(plan, t)
    assert float((a - b).abs().max()) <= TOL * float(reference(plan, t.abs()).max())


@pytest.mark.parametrize("N", [32, 48, 64, 96, 128, 192, 256, 2, 3, 5, 15, 18, 45, 50, 75, 120, 125, 135])
@pytest.mark.parametrize("kind", ["mixture", "random", "impulse", "checkerboard"])
def test_lengths(fsp, N, kind):
    if kind == "mixture":
        rho = I.gaussian_mixture(N)
    elif kind == "random":
        rho = I.random_field(N, 3)
    elif kind == "impulse":
        rho = I.impulse(N, at=(N - 1, 0, N // 2))
    else:  # nothing but the highest frequency: the products with S are small against both factors
        i = np.arange(N)
        rho = (-1.0) ** (i[:, None, None] + i[None, :, None] + i[None, None, :])
    check(fsp.Plan(N, 1.0, "he", "f64"), rho)


def test_largest_length(fsp):
    check(fsp.Plan(512, 1.0, "he", "f64"), I.random_field(512, 3))


@pytest.mark.parametrize("n3", [(32, 64, 128), (128, 32, 64), (64, 256, 512), (30, 45, 64)])
def test_boxes(fsp, n3):
    check(fsp.Plan(n3, tuple(n / 64 for n in n3), "he", "f64"), I.random_field3(n3, 5))


@pytest.mark.parametrize("scale", [1e-307, 1e-290, 1e-40, 1e40, 1e290])
@pytest.mark.parametrize("L", [1.0, 1e-12, 1e15])
@pytest.mark.parametrize("N", [32, 30])
def test_exponents(fsp, N, scale, L):
    """The whole range of exponents, in sources and in spectra.  Powers of two
    scale the arrays exactly, so the reference is the solve at unit scale."""
    import torch
    unit = 2.0 ** np.round(np.log2(scale))
    p = fsp.Plan(N, L, "he", "f64")
    t = torch.from_numpy(I.gaussian_mixture(N)).cuda()
    b = p.solve(t)
    a = p.solve(t * unit)
    if not np.isfinite(float(b.abs().max()) * unit * 64 * N ** 3):  # the transforms overflow
        return
    # results and coefficients below 2^-1022 are subnormal, 2^-1074 apart: one
    # rounding per pass, summed over the box by the transforms and S
    fuzz = 64 * 2.0 ** -1074 * N ** 3 * max(1.0, float(p.spectrum().max()) * 8 * N ** 3)
    assert float((a - b * unit).abs().max()) <= TOL * float((b * unit).abs().max()) + fuzz


@pytest.mark.parametrize("bad", [float("inf"), float("-inf"), float("nan")])
@pytest.mark.parametrize("N", [32, 30])
def test_non_finite(fsp, N, bad):
    import torch
    p = fsp.Plan(N, 1.0, "he", "f64")
    t = torch.from_numpy(I.random_field(N, 1)).cuda()
    t[3, 4, 5] = bad
    assert not bool(torch.isfinite(p.solve(t)).any())
    t[3, 4, 5] = 0.0
    assert bool(torch.isfinite(p.solve(t)).all())
    assert bool((p.solve(torch.zeros_like(t)) == 0).all())
